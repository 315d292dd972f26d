"""GPU parity at the sizes where a kernel's tiles, remainders and dispatch borders lie, against the same oracles as the
other GPU tests."""
import pytest

from test_gpu_block import bk, test_avgpool as check_avgpool, test_dwconv3x3_module as check_dwconv   # noqa: F401 (bk: a fixture)

pytestmark = pytest.mark.gpu


# B, H, W, C_in, R, S: tiles of 8 x 16 and 8 x 8 output pixels, 64 and 32 channels; one pixel past a tile, a channel block half
# outside the tensor, replication that splits a channel block (one pixel per thread), more tiles than resident blocks, stride 3
@pytest.mark.parametrize("shape", [(2, 17, 17, 64, 1, 1), (1, 9, 25, 40, 1, 1), (2, 16, 16, 96, 1, 1), (3, 18, 34, 64, 1, 2), (1, 33, 17, 24, 1, 2),
                                   (1, 12, 12, 48, 2, 1), (1, 8, 24, 32, 2, 2), (2, 1, 40, 128, 1, 1), (90, 1, 1, 1024, 1, 1), (1, 13, 10, 32, 1, 3)])
def test_dwconv_tiles(bk, oracle, shape):
    check_dwconv(bk, oracle, shape)


@pytest.mark.parametrize("shape", [(1, 1, 1, 8, 1, 1), (3, 14, 10, 24, 3, 2), (2, 12, 12, 8, 2, 4), (70, 28, 28, 64, 1, 2)])
def test_avgpool_items(bk, oracle, shape):
    check_avgpool(bk, oracle, shape)
