"""The C-ABI library loads and exports every symbol include/bcnn.h declares (no GPU needed)."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "bcnn.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(bcnn_[a-z0-9_]+)\s*\(", text)))


def test_header_symbols_are_exported():
    from paper_2010_00704_b200 import build, binding
    lib = ctypes.CDLL(build.build())
    names = _declared()
    assert "bcnn_pack" in names and "bcnn_conv2d_b1_fused" in names and "bcnn_gemm_b1" in names
    for n in names:
        assert hasattr(lib, n), n
    assert set(binding.EXPORTS) <= set(names)


def test_status_strings_and_version():
    from paper_2010_00704_b200 import build, binding
    build.build()
    assert binding.version() >= 100
    assert binding.status_string(0) == "ok"
    assert "align" in binding.status_string(-3)
    assert "workspace" in binding.status_string(binding.ERR_WORKSPACE)
    assert "wait" in binding.status_string(binding.ERR_TIMEOUT)
    # the device error codes name the engine and the role whose wait gave up
    for code in (101, 102, 103, 111, 112, 113, 121, 122, 123, 124, 125, 126, 131, 132, 133, 134, 141, 142, 143, 144, 145, 146, 151, 152, 153, 154, 155, 156,
                 binding.SELFTEST_TIMEOUT_CODE):
        assert "timed out" in binding.status_string(code)
    assert binding.status_string(77) == "device-side error code"


def test_workspace_bytes_is_zero_for_every_shape():
    # no kernel uses scratch memory: the query exists so that callers can size one buffer per model anyway
    from paper_2010_00704_b200 import build, binding, workloads as wl
    build.build()
    for l in wl.BACKBONE18 + wl.BLOCK_STACK + wl.STEM_DOWN:
        for fused in (False, True):
            assert binding.bcnn_workspace_bytes(256, l.H, l.W, l.C_in, l.C_out, l.k, l.k, l.stride, l.pad, fused) == 0
    assert binding.bcnn_workspace_bytes(1, 16384, 1, 9216, 16384, 1, 1, 1, 0) == 0      # a GEMM of the sweep
    assert binding.bcnn_workspace_bytes(1, 4, 4, 48, 32, 1, 1, 1, 0) == 0                # invalid shape: still 0


def test_argument_validation_needs_no_device():
    # validation runs before any CUDA call, so bad arguments are reported on a CPU-only box too
    from paper_2010_00704_b200 import build, binding
    build.build()
    lib = binding.load()
    a = ctypes.c_void_p(4096)
    assert lib.bcnn_gemm_b1(None, a, a, 8, 8, 32, None) == -1
    assert lib.bcnn_gemm_b1(a, a, a, 8, 8, 48, None) == -2          # K not a multiple of 32
    assert lib.bcnn_gemm_b1(a, a, a, 0, 8, 32, None) == -1
    assert lib.bcnn_gemm_b1(ctypes.c_void_p(4100), a, a, 8, 8, 32, None) == -3
    assert lib.bcnn_gemm_b1_fused(a, a, None, a, 8, 32, 32, None) == -1
    assert lib.bcnn_gemm_b1_fused(a, a, a, a, 8, 40, 32, None) == -2  # N not a multiple of 32
    assert lib.bcnn_conv2d_b1(a, a, a, 1, 4, 4, 48, 8, 3, 3, 1, 1, None) == -2
    assert lib.bcnn_conv2d_b1(a, a, a, 1, 2, 2, 32, 8, 5, 5, 1, 0, None) == -1   # kernel larger than image
    assert lib.bcnn_conv2d_b1(a, a, a, 1, 4, 4, 32, 8, 3, 3, 0, 1, None) == -1
    assert lib.bcnn_pack(a, None, a, 1, 2, 2, 12, 2, None) == -2
    assert lib.bcnn_pack(None, None, a, 1, 2, 2, 32, 1, None) == -1
    assert lib.bcnn_conv2d_b1_engine(99, a, a, None, a, 1, 4, 4, 32, 8, 3, 3, 1, 1, None) == -2
    assert lib.bcnn_selftest_wait_timeout(0, None) == -1
    assert lib.bcnn_selftest_wait_timeout(1 << 20, None) == -1


def test_prepared_call_takes_what_it_is_preferred_for():
    # The gather's table grows with K: near the largest K one of the tile widths no longer fits shared memory, and the call has to
    # take another.  Rows of an odd, an even and a fourfold number of words around those sizes, both outputs; made-up addresses, so
    # only where no device could run the call: there it gets as far as the driver (ERR_CUDA) or refuses the shape.
    import pytest
    import torch
    from paper_2010_00704_b200 import build, binding
    if torch.cuda.is_available():
        pytest.skip("made-up addresses: only without a device")
    build.build()
    lib = binding.load()
    a = ctypes.c_void_p(4096)
    seen = set()
    for unit, lo, hi in ((1, 8000, 10200), (2, 16000, 20400), (4, 31000, 32768)):          # words of K: the limits lie inside
        for kwords in range(lo, hi + 1, 37 * unit):
            kwords = kwords // unit * unit + (unit if unit < 4 and (kwords // unit) % 2 == 0 else 0)       # exactly `unit` divides it
            K = 32 * kwords
            for M, N in ((1, 64), (700, 256), (4736, 1024), (100000, 512)):
                for fused in (0, 1):
                    st = lib.bcnn_gemm_b1_prepared(a, a, a if fused else None, a, M, N, K, None)
                    preferred = lib.bcnn_prepared_preferred(1, M, 1, K, N, 1, 1, 1, 0, fused)
                    assert st in (binding.ERR_CUDA, binding.ERR_UNSUPPORTED), (M, N, K, fused)
                    assert not preferred or st == binding.ERR_CUDA, (M, N, K, fused)
                    seen.add((fused, st))
    assert len(seen) == 4                                                                    # both answers, both outputs


def test_fc_takes_long_rows_in_large_products():
    # Rows of more than 12800 channels do not fit the kernel that streams the weights: large products of them run in tiles whatever the estimates
    # say, small ones are refused.  Made-up addresses, so only where no device could run the call.
    import pytest
    import torch
    from paper_2010_00704_b200 import build, binding
    if torch.cuda.is_available():
        pytest.skip("made-up addresses: only without a device")
    build.build()
    lib, a = binding.load(), ctypes.c_void_p(4096)
    for B, C, N in ((5, 12808, 5350), (8, 17104, 9000), (16, 32768, 5350), (6, 72108, 8770), (300, 20000, 1000)):
        assert lib.bcnn_fc(a, a, a, a, B, C, N, None) == binding.ERR_CUDA, (B, C, N)
    for B, C, N in ((1, 12804, 100), (4, 40000, 10000)):
        assert lib.bcnn_fc(a, a, a, a, B, C, N, None) == binding.ERR_UNSUPPORTED, (B, C, N)
    assert lib.bcnn_fc(a, a, a, a, 1, 12800, 100, None) == binding.ERR_CUDA


def test_module_engine_takes_wide_branch_modules():
    # per number of branches a module at the end of the module engine's range: expanded weights of one slice of 32 output channels fill
    # shared memory beside what has to lie there for as long
    from paper_2010_00704_b200 import build, binding
    build.build()
    for P, widest in ((4, 2304), (5, 1792), (6, 1472), (7, 1280), (8, 1088), (9, 960), (10, 832), (11, 768), (12, 704), (13, 576)):
        assert binding.bcnn_branches_plan(64, 28, 28, widest, widest, P)[0] == 32, P
        assert binding.bcnn_branches_plan(64, 28, 28, widest, 32, P)[0] == 32, P
        assert binding.bcnn_branches_plan(64, 28, 28, 2 * widest, 64, P)[0] == 0, P
    assert binding.bcnn_branches_plan(64, 28, 28, 896, 896, 9, 3, 3)[0] == 32
    for C in (1024, 2560):                                                          # K of one branch: up to 2560 by the constants
        for P in (1, 2, 3):
            assert binding.bcnn_branches_plan(64, 28, 28, C, C, P)[0] in (32, 64), (P, C)
    assert binding.bcnn_branches_plan(64, 28, 28, 64, 64, 14)[0] == 0
    # the weights as they come do not cost resident slices: P = 2, 256 channels keep all four
    assert binding.bcnn_branches_plan(64, 28, 28, 256, 256, 2)[:2] == (64, 4)
    assert binding.bcnn_branches_plan(64, 28, 28, 128, 128, 9, 3, 3)[:2] == (32, 4)


def test_long_products_stream_where_slices_are_narrow():
    # wide products too long for resident slices of 128 channels: in slices of 64 the weight-stationary engine takes 1.3 to 2.2 times as long
    from paper_2010_00704_b200 import build, binding
    build.build()
    for M, N, K, fused in ((16638, 3584, 4192, True), (17902, 1120, 5632, True), (4096, 4096, 4608, False), (8170, 1008, 4832, False)):
        assert binding.bcnn_auto_engine(1, M, 1, K, N, 1, 1, 1, 0, fused=fused) == "tc_i8", (M, N, K)
    for M, N, K in ((4096, 4096, 2304), (50176, 512, 2304)):
        assert binding.bcnn_auto_engine(1, M, 1, K, N, 1, 1, 1, 0, fused=False) == "tc_ws", (M, N, K)


def test_every_wait_code_has_a_name():
    # the codes as the kernels define them, each in one place
    from paper_2010_00704_b200 import build, binding
    build.build()
    codes = {}
    for src in build.sources():
        for name, code in re.findall(r"\b(ERR_\w+) = (\d{3})\b", open(src).read()):
            assert codes.setdefault(int(code), (src, name)) == (src, name), code
    assert len(codes) >= 37 and {101, 131, 161, 171, 181, 182} <= set(codes)
    for code, where in codes.items():
        assert "timed out" in binding.status_string(code), where
