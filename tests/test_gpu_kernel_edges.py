"""GPU parity at the sizes where a kernel's tiles, remainders and dispatch borders lie, against the same oracles as the
other GPU tests."""
import pytest

import numpy as np
import torch

from paper_2010_00704_b200 import synth
from test_gpu_block import bk, dev, test_avgpool as check_avgpool, test_dwconv3x3_module as check_dwconv   # noqa: F401 (bk: a fixture)
from test_gpu_block import test_fxf_as_shifted_branches as check_shifted, test_parallel_branches as check_branches   # noqa: F401
from test_gpu_parity import run_conv, test_conv_module as check_module   # noqa: F401

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


# several parts per block: one accumulator buffer (nine taps), three (two branches), four (one branch); 32- and 64-channel parts; the
# CUDA-core kernel behind the engine's limit (14 branches)
@pytest.mark.parametrize("shape", [(20, 40, 40, 64, 64, 2), (20, 40, 40, 32, 96, 4), (26, 40, 40, 96, 64, 1), (1, 9, 15, 64, 32, 14)])
def test_branches_many_parts(bk, oracle, shape):
    check_branches(bk, oracle, shape, "full")


# a row tile with more stages than the ring has slots: every slot refilled several times for one part, one or more row tiles a block
@pytest.mark.parametrize("variant", ["full", "no_identity"])
@pytest.mark.parametrize("shape", [(1, 17, 19, 480, 64, 13), (2, 100, 101, 288, 32, 13), (1, 17, 19, 512, 64, 13)])
def test_branches_longer_than_the_ring(bk, oracle, shape, variant):
    B, H, W, C_in, C_out, P = shape
    part, _, row_stages, slots, _ = bk.bcnn_branches_plan(B, H, W, C_in, C_out, P)
    assert part == 32 and row_stages > slots
    check_branches(bk, oracle, shape, variant)


# every number of branches has a kernel of its own; one part a block and several, with and without an identity
@pytest.mark.parametrize("variant", ["full", "no_identity"])
@pytest.mark.parametrize("P", [5, 6, 7, 8, 9, 10, 11, 12, 13])
def test_branches_each_number(bk, oracle, P, variant):
    for shape in ((1, 13, 17, 32, 64, P), (2, 90, 107, 64, 96, P)):
        assert bk.bcnn_branches_plan(*shape)[0] == 32
        check_branches(bk, oracle, shape, variant)


# the widest modules the engine takes: the packed weights lie over all staging tiles (960 channels) or all but the teams' first (1024)
# until they are expanded; tiles behind those are used by the same launch
@pytest.mark.parametrize("variant", ["full", "no_identity", "in_place"])
@pytest.mark.parametrize("shape,early", [((2, 40, 41, 960, 64, 9), 0), ((1, 30, 31, 1472, 32, 6), 0), ((2, 40, 41, 1024, 64, 8), 2), ((1, 26, 27, 768, 96, 9), 2)])
def test_branches_widest(bk, oracle, shape, early, variant):
    B, H, W, C_in, C_out, P = shape
    assert bk.bcnn_branches_plan(B, H, W, C_in, C_out, P)[::4] == (32, early)
    check_branches(bk, oracle, shape, variant)


# many parts a block with all slices resident, so that the packed weights lie under identity tiles that come right behind them
@pytest.mark.parametrize("shape", [(40, 28, 28, 256, 256, 2), (8, 28, 28, 96, 512, 4), (8, 28, 28, 64, 256, 5)])
def test_branches_weights_under_staging_tiles(bk, oracle, shape):
    B, H, W, C_in, C_out, P = shape
    part, resident, _, _, early = bk.bcnn_branches_plan(B, H, W, C_in, C_out, P)
    assert resident >= 3 and early == 2
    check_branches(bk, oracle, shape, "full")


# the CUDA-core kernel: more branches than the engine has accumulators for, several slices of channels, many row tiles;
# and a K beyond the engine's constants, where one branch is compared with another kernel's module besides (for a shorter K both
# calls run on the same engine)
@pytest.mark.parametrize("variant", ["full", "no_identity", "in_place", "no_bits"])
@pytest.mark.parametrize("shape", [(2, 7, 9, 32, 320, 20), (3, 60, 61, 32, 32, 14), (1, 9, 11, 2624, 64, 1)])
def test_branches_cuda_cores(bk, oracle, shape, variant):
    check_branches(bk, oracle, shape, variant)


@pytest.mark.parametrize("reading", ["paper", "zero"])
@pytest.mark.parametrize("shape", [(2, 9, 13, 32, 64, 5), (1, 5, 33, 96, 32, 5)])
def test_shifted_branches_cuda_cores(bk, oracle, shape, reading):
    check_shifted(bk, oracle, shape, reading)


@pytest.mark.parametrize("shape", [(16, 40, 40, 32, 64, 3), (2, 30, 31, 224, 96, 3)])
def test_shifted_branches_many_parts(bk, oracle, shape):
    check_shifted(bk, oracle, shape, "paper")


# the module on the streaming engine: 3 x 3 layers whose resident weights fit beside no producer group (11 stages of 96 channels, 20 of
# 320); one 128-wide tile column and three with a ragged last one, more row tiles than multiprocessors.  32 channels of that K
# fit the weight-stationary engine, one block per multiprocessor
@pytest.mark.parametrize("variant", ["full", "no_identity", "no_bits", "in_place"])
@pytest.mark.parametrize("shape", [(2, 100, 99, 288, 96, 3, 1, 1), (1, 9, 10, 544, 320, 3, 1, 1), (1, 13, 7, 544, 32, 3, 2, 1)])
def test_module_long_k(bk, oracle, shape, variant):
    check_module(bk, oracle, shape, variant)


# packing: pixels that are no whole number of passes (bias in registers or by remainder), NaN and -0, the replicated widths
@pytest.mark.parametrize("shape", [(3, 7, 5, 32, 1), (2, 11, 13, 96, 1), (1, 9, 7, 1056, 1), (40, 28, 28, 160, 1), (2, 5, 9, 8, 4), (2, 9, 5, 64, 2), (1, 7, 9, 128, 3),
                                   (1, 5, 7, 96, 2), (1, 3, 4, 48, 4)])
def test_pack_shapes(bk, oracle, shape):
    B, H, W, C, R = shape
    rng = np.random.default_rng(9500 + sum(shape))
    x, bias = synth.real_input(rng, (B, H, W, C)), synth.real_input(rng, (C * R,))
    x.reshape(-1)[::7], x.reshape(-1)[::11] = -0.0, np.nan
    for b in (bias, None):
        out = torch.empty(B * H * W * C * R // 8, dtype=torch.uint8, device="cuda")
        bk.bcnn_pack(dev(x), None if b is None else dev(b), out, B, H, W, C, R)
        torch.cuda.synchronize()
        want = oracle.binarize(x, b if b is not None else np.zeros(C * R, np.float32), R)
        assert np.array_equal(synth.unpack_bits(out.cpu().numpy().reshape(B, H, W, C * R // 8)), want)


# tiled fp32 product (many images) and one warp per output (few), ragged in every direction
@pytest.mark.parametrize("shape", [(300, 200, 1000), (97, 36, 3000), (3, 2048, 100), (1, 8, 1)])
def test_fc_shapes(bk, oracle, shape):
    B, C, N = shape
    rng = np.random.default_rng(9600 + sum(shape))
    x, w, bias = (rng.standard_normal(s).astype(np.float32) for s in ((B, C), (N, C), (N,)))
    out = torch.empty(B * N, dtype=torch.float32, device="cuda")
    for b in (bias, None):
        bk.bcnn_fc(dev(x), dev(w), None if b is None else dev(b), out, B, C, N)
        torch.cuda.synchronize()
        ref = x.astype(np.float64) @ w.astype(np.float64).T + (0 if b is None else b)
        mag = np.abs(x.astype(np.float64)) @ np.abs(w.astype(np.float64)).T + np.abs(bias)
        assert np.all(np.abs(out.cpu().numpy().reshape(B, N) - ref) <= (C + 76) * 2.0 ** -24 * mag)


# pooling in pixel slices: fewer pixels than slices, channels that are no whole block
@pytest.mark.parametrize("shape", [(2, 1, 1, 8), (3, 5, 7, 264), (1, 14, 14, 2048), (5, 3, 3, 24)])
def test_gap_shapes(bk, oracle, shape):
    B, H, W, C = shape
    x = np.random.default_rng(9700 + sum(shape)).standard_normal(shape).astype(np.float16)
    out = torch.empty(B * C, dtype=torch.float32, device="cuda")
    bk.bcnn_gap(dev(x.view(np.uint8).reshape(-1)), out, B, H, W, C)
    torch.cuda.synchronize()
    mag = np.abs(x.astype(np.float64)).mean(axis=(1, 2))
    assert np.all(np.abs(out.cpu().numpy().reshape(B, C) - oracle.gap(x)) <= (H * W + 15) * 2.0 ** -24 * mag + 1e-30)


# B, H, W, C_in, C_out, k, stride, pad: wide pointwise engine with one and two resident slices (the latter from a dozen row tiles per
# block on), K = 128, 256, 512; halo-tile engine with two and three tiles in flight and 128 channels
@pytest.mark.parametrize("engine,shape", [("tc_pn", (1, 60, 70, 128, 128, 1, 1, 0)), ("tc_pn", (2, 352, 360, 128, 256, 1, 1, 0)), ("tc_pn", (1, 20, 21, 256, 384, 1, 1, 0)),
                                          ("tc_pn", (1, 15, 9, 512, 1024, 1, 1, 0)), ("tc_c3", (9, 64, 64, 64, 64, 3, 1, 1)), ("tc_c3", (9, 64, 64, 32, 128, 3, 1, 1)),
                                          ("tc_c3", (5, 64, 64, 64, 128, 3, 2, 1)), ("tc_i8", (1, 700, 1, 1152, 96, 1, 1, 0)), ("lop3", (1, 9, 11, 96, 70, 1, 1, 0))])
def test_engine_edges(bk, oracle, engine, shape):
    B, H, W, Ci, Co, k, stride, pad = shape
    rng = np.random.default_rng(9800 + sum(shape))
    x, w = synth.pm1(rng, (B, H, W, Ci)), synth.pm1(rng, (Co, k, k, Ci))
    if H * W > 100000:                                  # the packed checker's sums on a sample of rows
        thr = synth.thresholds(rng, Ci, Co)
        got = run_conv(bk, x, w, thr, stride, pad, engine)
        rows = rng.integers(0, H * W, 400)
        want = oracle.threshold(x.reshape(-1, Ci)[rows].astype(np.int32) @ w.reshape(Co, Ci).astype(np.int32).T, thr)
        assert np.array_equal(np.asarray(got).reshape(-1, Co)[rows], want)
        return
    acc = oracle.conv2d(x, w, stride, pad)
    thr = synth.thresholds(rng, k * k * Ci, Co) if Co % 32 == 0 else None
    want = acc if thr is None else oracle.threshold(acc, thr)
    assert np.array_equal(run_conv(bk, x, w, thr, stride, pad, engine), want)


# prepared weights: tiles 256, 128 and 64 wide by the estimate, int32 rows of any width
@pytest.mark.parametrize("M,N,K,fused", [(40000, 256, 2304, True), (12544, 512, 1184, True), (3000, 128, 800, True), (700, 473, 704, False), (20000, 257, 512, False), (5000, 1000, 2400, False)])
def test_prepared_widths(bk, oracle, M, N, K, fused):
    rng = np.random.default_rng(M + N + K)
    A, W = synth.random_bits(rng, (M, K // 8)), synth.random_bits(rng, (N, K // 8))
    thr = synth.thresholds(rng, K, N) if fused else None
    prep = torch.empty(bk.bcnn_prepared_weights_bytes(N, K), dtype=torch.uint8, device="cuda")
    bk.bcnn_prepare_weights(dev(W), prep, N, K)
    out = torch.empty(M * N // 8 if fused else M * N * 4, dtype=torch.uint8, device="cuda")
    bk.bcnn_gemm_b1_prepared(dev(A), prep, None if thr is None else dev(thr), out, M, N, K)
    torch.cuda.synchronize()
    acc = synth.unpack_bits(A).astype(np.float32) @ synth.unpack_bits(W).astype(np.float32).T       # exact: |sums| < 2^24
    if fused:
        assert np.array_equal(synth.unpack_bits(out.cpu().numpy().reshape(M, N // 8)), np.where(acc >= thr, 1, -1))
    else:
        assert np.array_equal(out.cpu().numpy().view(np.int32).reshape(M, N), acc.astype(np.int32))
    assert bk.bcnn_device_error() == 0


# the longest K: the int32 output's 256-wide tiles fit up to 274 176 bits of an odd number of words, and 37 x 4 of them would
# be a whole wave; every output row of a sample
@pytest.mark.parametrize("M,N,K", [(4736, 1024, 274144), (4736, 1024, 274208), (130, 70, 306912)])
def test_prepared_longest_k(bk, oracle, M, N, K):
    rng = np.random.default_rng(M + N + K)
    A, W = synth.random_bits(rng, (M, K // 8)), synth.random_bits(rng, (N, K // 8))
    assert bk.bcnn_prepared_preferred(1, M, 1, K, N, 1, 1, 1, 0, fused=False)
    prep = torch.empty(bk.bcnn_prepared_weights_bytes(N, K), dtype=torch.uint8, device="cuda")
    bk.bcnn_prepare_weights(dev(W), prep, N, K)
    out = torch.empty(M, N, dtype=torch.int32, device="cuda")
    bk.bcnn_gemm_b1_prepared(dev(A), prep, None, out, M, N, K)
    torch.cuda.synchronize()
    rows = np.array([0, 127, 128, M - 1])
    assert np.array_equal(out.cpu().numpy()[rows], oracle.gemm(synth.unpack_bits(A[rows]), synth.unpack_bits(W)))
    assert bk.bcnn_device_error() == 0


# the stem's plain kernel and its table, on both sides of the line between them (148 * 2304 pixels), and with the ring of
# chunks used more than once (148 * 5 * 1984 pixels), a bias for the per-channel path included
@pytest.mark.parametrize("shape,inf", [((1, 9, 7), False), ((1, 576, 592), False), ((1, 577, 592), True), ((1, 579, 591), False), ((1, 1100, 1351), False),
                                       ((1, 1100, 1351), True)])
def test_stem_sizes(bk, oracle, shape, inf):
    B, H, W = shape
    rng = np.random.default_rng(9900 + sum(shape))
    x, bias, w = synth.real_input(rng, (B, H, W, 4)), synth.real_input(rng, (32,)), synth.pm1(rng, (32, 1, 1, 32))
    thr = synth.thresholds(rng, 32, 32)
    if inf:
        bias[5], bias[9] = np.inf, -np.inf
    out = torch.empty(B * H * W * 4, dtype=torch.uint8, device="cuda")
    bk.bcnn_stem_fused(dev(x), dev(bias), dev(synth.pack_bits(w)), dev(thr), out, B, H, W, 4, 8, 32)
    torch.cuda.synchronize()
    want = oracle.threshold(oracle.conv2d(oracle.binarize(x, bias, 8), w, 1, 0), thr)
    assert np.array_equal(synth.unpack_bits(out.cpu().numpy().reshape(B, H, W, 4)), want)


# Engines that refill a stage of shared memory by a bulk copy while the CTA works: many row tiles per CTA, the input in L2 (the
# fastest refill), the call repeated.  A stage handed back too early shows as a few wrong words in some of the launches only (with
# the arrival right behind the wide pointwise engine's loads one launch of fifteen: 200 pass by luck with probability 1e-6).
@pytest.mark.parametrize("engine,shape", [("tc_pn", (1, 333 * 128 + 77, 1, 512, 512, 1, 1, 0)), ("tc_pn", (1, 148 * 9 * 128 + 5, 1, 256, 256, 1, 1, 0)),
                                          ("tc_c3", (16, 128, 128, 64, 64, 3, 1, 1)), ("tc_c3", (8, 160, 176, 32, 64, 3, 2, 1)), ("tc_c3", (16, 128, 128, 64, 128, 3, 2, 1)),
                                          ("tc_pw", (64, 112, 112, 32, 32, 1, 1, 0)), ("tc_pw", (64, 112, 112, 64, 64, 1, 1, 0)), ("tc_pw", (64, 56, 56, 128, 128, 1, 1, 0))])
def test_stages_handed_back_in_every_launch(bk, engine, shape):
    B, H, W, Ci, Co, k, stride, pad = shape
    rng = np.random.default_rng(9950 + sum(shape))
    OH, OW = bk.out_hw(H, W, k, k, stride, pad)
    x, w = dev(synth.random_bits(rng, (B * H * W, Ci // 8))), dev(synth.random_bits(rng, (Co, k * k * Ci // 8)))
    thr = dev(synth.thresholds(rng, k * k * Ci, Co))
    ref, out = (torch.empty(B * OH * OW, Co // 8, dtype=torch.uint8, device="cuda") for _ in range(2))
    bk.bcnn_conv2d_b1_fused(x, w, thr, ref, B, H, W, Ci, Co, k, k, stride, pad, engine=bk.ENGINES["tc_ws"])     # (checked against the oracle elsewhere)
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(200):
        out.fill_(0xA5)
        bk.bcnn_conv2d_b1_fused(x, w, thr, out, B, H, W, Ci, Co, k, k, stride, pad, engine=bk.ENGINES[engine])
        wrong += (out != ref).any()
    assert int(wrong) == 0
    assert bk.bcnn_device_error() == 0


# ... the streaming engine's hand-overs, prepared and raw: pairs of blocks (whose signals cross from one to the other) of one stage a tile and of
# many, 256-wide tiles handed over in halves and in one piece, and raw rows' bit counts, whose places a long walk uses again
@pytest.mark.parametrize("prepared,M,N,K,fused,plan", [(True, 25100, 512, 4608, True, (256, 2, 0, 0)), (True, 76000, 512, 96, True, (256, 2, 0, 0)), (True, 9500, 1500, 8224, False, (256, 2, 0, 0)),
                                                       (True, 50000, 256, 992, True, (256, 1, 0, 0)), (True, 150003, 250, 416, False, (256, 1, 1, 0)),
                                                       (False, 60000, 1024, 96, True, (256, 2, 0, 2)), (False, 9000, 1120, 4640, True, (256, 2, 0, 2)), (False, 5000, 500, 8224, False, (256, 2, 0, 2)),
                                                       (False, 19000, 512, 288, False, (128, 1, 0, 1)), (False, 300000, 64, 288, True, (64, 1, 0, 1))])
def test_streamed_stages_handed_back_in_every_launch(bk, prepared, M, N, K, fused, plan):
    assert stream_plan(bk, prepared, M, N, K, fused)[:4] == plan
    rng = np.random.default_rng(M + N + K)
    x, w, thr = dev(synth.random_bits(rng, (M, K // 8))), dev(synth.random_bits(rng, (N, K // 8))), dev(synth.thresholds(rng, K, N))
    ref, out = (torch.empty(M * N // 8 if fused else M * N * 4, dtype=torch.uint8, device="cuda") for _ in range(2))
    if fused:
        bk.bcnn_gemm_b1_fused(x, w, thr, ref, M, N, K, engine=bk.ENGINES["lop3"])
    else:
        bk.bcnn_gemm_b1(x, w, ref, M, N, K, engine=bk.ENGINES["lop3"])
    prep = torch.empty(bk.bcnn_prepared_weights_bytes(N, K), dtype=torch.uint8, device="cuda")
    bk.bcnn_prepare_weights(w, prep, N, K)
    torch.cuda.synchronize()
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(200):
        out.fill_(0xA5)
        if prepared:
            bk.bcnn_gemm_b1_prepared(x, prep, thr if fused else None, out, M, N, K)
        elif fused:
            bk.bcnn_gemm_b1_fused(x, w, thr, out, M, N, K, engine=bk.ENGINES["tc_i8"])
        else:
            bk.bcnn_gemm_b1(x, w, out, M, N, K, engine=bk.ENGINES["tc_i8"])
        wrong += (out != ref).any()
    assert int(wrong) == 0
    assert bk.bcnn_device_error() == 0


# ... and the stem, seventeen chunks a CTA through its ring of five, against the two separate calls
def test_stem_stages_handed_back_in_every_launch(bk):
    B, H, W = 100, 224, 224
    rng = np.random.default_rng(9960)
    x = torch.randn(B * H * W * 4, device="cuda", generator=torch.Generator(device="cuda").manual_seed(9960))
    bias, w, thr = dev(synth.real_input(rng, (32,))), dev(synth.random_bits(rng, (32, 4))), dev(synth.thresholds(rng, 32, 32))
    bits, ref, out = (torch.empty(B * H * W * 4, dtype=torch.uint8, device="cuda") for _ in range(3))
    bk.bcnn_pack(x, bias, bits, B, H, W, 4, 8)
    bk.bcnn_conv2d_b1_fused(bits, w, thr, ref, B, H, W, 32, 32, 1, 1, 1, 0, engine=bk.ENGINES["lop3"])
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(200):
        out.fill_(0xA5)
        bk.bcnn_stem_fused(x, bias, w, thr, out, B, H, W, 4, 8, 32)
        wrong += (out != ref).any()
    assert int(wrong) == 0
    assert bk.bcnn_device_error() == 0


# the module's sign threshold and PReLU on values where a rounding, a sign of zero, an infinity or a NaN could go the other way: identities
# and next biases from lists of such values in all combinations, on 32- and 64-channel parts with a half-empty last one
@pytest.mark.parametrize("has_nb", [True, False])
@pytest.mark.parametrize("P", [1, 2, 3, 4, 6, 11])
@pytest.mark.parametrize("shape", [(1, 11, 13, 96), (1, 120, 161, 96)])
def test_module_special_values(bk, oracle, shape, P, has_nb):
    B, H, W, C = shape
    rng = np.random.default_rng(41 + P)
    inf, nan, tiny = np.inf, np.nan, 2.0 ** -24                                  # tiny: the smallest fp16 number
    ids = np.array([0.0, -0.0, 1.0, -1.0, tiny, -tiny, 65504.0, -65504.0, inf, -inf, nan, 0.5, -2.0, 1000.0, -1000.0, 6e-5], np.float16)
    nbs = np.array([0.0, -0.0, 1e-45, -1e-45, tiny, -tiny, 0.7 * tiny, -0.7 * tiny, 1.0, -1.0, 1.0 + 2.0 ** -23, -1.0 - 2.0 ** -23, 65504.0, -65504.0,
                    65520.0, -65520.0, 1e30, -1e30, inf, -inf, nan, 0.3, -0.3, 2.0], np.float32)
    slopes = np.array([1.0, 0.25, 0.0, -0.0, -0.5, 2.0, 1e-30, inf, -inf, nan], np.float32)
    x, w = synth.pm1(rng, (B, H, W, P * 32)), synth.pm1(rng, (P, C, 32))
    scale = rng.choice(np.array([0.0, 1.0, -1.0, 1e-6, 1e30], np.float32), (P, C), p=[0.6, 0.1, 0.1, 0.1, 0.1])
    shift = rng.choice(np.array([0.0, -0.0, 1.0, -tiny], np.float32), (P, C))
    slope, nb = rng.choice(slopes, C), rng.choice(nbs, C)
    ident = rng.choice(ids, (B, H, W, C))
    accs = np.stack([oracle.conv2d(np.ascontiguousarray(x[..., 32 * p:32 * p + 32]), w[p].reshape(C, 1, 1, 32), 1, 0) for p in range(P)])
    want_y, want_s = oracle.conv_module_branches(accs, scale, shift, ident, slope, nb if has_nb else None)
    y = torch.empty(want_y.size, dtype=torch.float16, device="cuda")
    bits = torch.empty(want_y.size // 8, dtype=torch.uint8, device="cuda")
    bk.bcnn_conv2d_b1_branches(dev(synth.pack_bits(x)), dev(synth.pack_bits(w)), dev(scale), dev(shift), None, dev(ident), dev(slope), dev(nb) if has_nb else None,
                               y, bits, B, H, W, 32, C, P)
    torch.cuda.synchronize()
    got = y.cpu().numpy().reshape(want_y.shape)
    # a NaN's payload is not defined, everything else is
    assert np.array_equal(np.isnan(got), np.isnan(want_y))
    assert np.array_equal(np.where(np.isnan(got), 0, got.view(np.uint16)), np.where(np.isnan(want_y), 0, want_y.view(np.uint16)))
    assert np.array_equal(synth.unpack_bits(bits.cpu().numpy().reshape(B, H, W, C // 8)), want_s)
    assert bk.bcnn_device_error() == 0


def stream_plan(bk, prepared, M, N, K, fused):
    """Channels of a tile, blocks on one, 1 where it is handed over in one piece, whose bits are counted (0 none, 1 weights, 2 rows), stages, tiles of a block."""
    return bk.bcnn_stream_plan(prepared, 1, M, 1, K, N, 1, 1, 1, 0, fused)


# two blocks on a tile of 256 rows x 256 columns, packed: three waves of tiles with a K of 4096 bits and more, and nine to eleven with a short
# one; the last row tile and the last columns part empty, an odd number of 128-column groups, K with a tail of every length in its last
# stage.  (The two int32 products are whole rows on single blocks.)
@pytest.mark.parametrize("M,N,K,fused", [(25100, 512, 4608, True), (29000, 480, 4128, True), (14336, 1000, 4192, False), (40000, 1152, 288, True),
                                         (9500, 1100, 4448, False), (30011, 640, 4352, True), (152000, 256, 96, True)])
def test_prepared_block_pairs(bk, oracle, M, N, K, fused):
    assert stream_plan(bk, True, M, N, K, fused)[:3] == ((256, 2, 0) if fused else (256, 1, 1))
    test_prepared_widths(bk, oracle, M, N, K, fused)


# ... and int32 ones, as 16-bit pairs beside the next tile's MMAs (K <= 32767) and straight out of the accumulator; eleven tiles of nine stages
@pytest.mark.parametrize("M,N,K,fused", [(9500, 1500, 8224, False), (12300, 900, 10272, False), (9500, 1100, 32800, False), (40000, 1280, 2080, True)])
def test_prepared_block_pairs_int32(bk, oracle, M, N, K, fused):
    assert stream_plan(bk, True, M, N, K, fused)[:3] == (256, 2, 0)
    test_prepared_widths(bk, oracle, M, N, K, fused)


# 256-wide tiles handed over in halves: one to five stages (none, one and two of them split at either end), three tiles per block
@pytest.mark.parametrize("K", [32, 256, 288, 512, 768, 992, 1056])
def test_prepared_split_tiles(bk, oracle, K):
    assert stream_plan(bk, True, 50000, 256, K, True) == (256, 1, 0, 0, (K + 255) // 256, 3)
    test_prepared_widths(bk, oracle, 50000, 256, K, True)


# int32 products of one stage: a wave of 64-wide tiles, and more on 128-wide ones, ragged in rows and columns; up to 64 columns
# the narrow tile at any number of rows
@pytest.mark.parametrize("M,N,K", [(1000, 500, 256), (5301, 860, 32), (6001, 801, 160), (20000, 300, 256), (101003, 64, 256), (150000, 40, 32)])
def test_prepared_one_stage_int32(bk, oracle, M, N, K):
    assert stream_plan(bk, True, M, N, K, False)[:2] == (64 if M == 1000 or N <= 64 else 128, 1)
    test_prepared_widths(bk, oracle, M, N, K, False)


# int32 rows of no whole sectors: tiles down their columns where the output stays in the cache, and whole rows by 256-wide tiles in one piece, K of
# one stage, two and several
@pytest.mark.parametrize("M,N,K", [(40000, 364, 64), (20000, 255, 288), (30100, 397, 1184), (2500, 2300, 96), (300, 1021, 4640), (262200, 131, 256), (150003, 250, 416), (135000, 253, 2336)])
def test_prepared_ragged_int32_rows(bk, oracle, M, N, K):
    test_prepared_widths(bk, oracle, M, N, K, False)


# ... and tiles across their columns: outputs of 2^25 values and more, three, eight and 74 columns of tiles, rows left over in the last round of row
# tiles, K of one stage, two and several
@pytest.mark.parametrize("M,N,K", [(100003, 364, 64), (100000, 380, 1184), (34000, 1021, 288), (9000, 9393, 96)])
def test_prepared_tiles_across_columns(bk, oracle, M, N, K):
    assert stream_plan(bk, True, M, N, K, False)[:4] == (128, 1, 0, 0)
    test_prepared_widths(bk, oracle, M, N, K, False)


# the tiled product with its K over two, four and eight blocks (the last of them without a chunk), ragged in images, outputs and K; tiles of 32 and 64
# outputs in one wave, alone on their multiprocessors, and in several, two on each; few images, tiled and streamed
@pytest.mark.parametrize("shape", [(64, 2048, 100), (97, 1156, 130), (130, 516, 700), (200, 2052, 1000), (300, 264, 65), (61, 1100, 513), (256, 2048, 10),
                                   (64, 160, 500), (250, 36, 2001), (201, 264, 2999), (129, 516, 1001), (255, 128, 4001),
                                   (215, 516, 656), (98, 388, 2401), (4, 2956, 42), (2, 2328, 1146)])
def test_fc_split(bk, oracle, shape):
    test_fc_shapes(bk, oracle, shape)


# rows longer than the streaming kernel holds, where its estimate would be the smaller
@pytest.mark.parametrize("shape", [(5, 12808, 5350), (16, 13004, 2700)])
def test_fc_long_rows(bk, oracle, shape):
    test_fc_shapes(bk, oracle, shape)


# pooling by 8 and 16 channel groups of few images, by 32 and 16 where a slice has three pixels at most
@pytest.mark.parametrize("shape", [(8, 10, 10, 192), (1, 13, 11, 264), (20, 9, 9, 1600), (14, 2, 2, 1112), (3, 4, 6, 520), (3, 5, 5, 520), (2, 6, 8, 136)])
def test_gap_few_images(bk, oracle, shape):
    test_gap_shapes(bk, oracle, shape)


# raw weights on the streaming engine: pairs of blocks (both outputs, K of 32 to 4640 bits with every tail, columns of a half-empty tile, words by
# 16, 8 and 4 bytes; int32 of more than 16 bits), 128-wide tiles that count their weights' bits or their rows' and 64-wide ones, of one stage and
# of several, and on each more tiles in a block's walk than bit counts are kept for (10, 11, 13)
@pytest.mark.parametrize("M,N,K,fused,plan", [(4096, 4096, 1184, True, (256, 2, 0, 2)), (9000, 1120, 4640, True, (256, 2, 0, 2)), (2048, 1000, 4128, False, (128, 1, 0, 2)),
                                              (20000, 512, 32, True, (256, 2, 0, 2)), (20000, 512, 288, True, (256, 2, 0, 2)), (12544, 512, 2112, True, (256, 2, 0, 2)),
                                              (8200, 4000, 4608, False, (256, 2, 0, 2)), (300, 992, 9216, True, (64, 1, 0, 1)), (20, 64, 960, True, (64, 1, 0, 1)),
                                              (5000, 70, 4000, False, (64, 1, 0, 1)), (40000, 192, 256, False, (64, 1, 0, 1)),
                                              (60000, 1024, 96, True, (256, 2, 0, 2)), (60000, 1024, 288, True, (256, 2, 0, 2)), (5000, 1000, 33056, False, (256, 2, 0, 2)),
                                              (300000, 64, 32, True, (64, 1, 0, 1)), (270000, 50, 288, False, (64, 1, 0, 1)),
                                              (2001, 2048, 32, True, (128, 1, 0, 1)), (100000, 352, 32, False, (128, 1, 0, 1)), (100001, 352, 288, False, (128, 1, 0, 1)),
                                              (40003, 96, 288, True, (128, 1, 0, 1)), (19000, 128, 2400, True, (128, 1, 0, 2)), (100001, 352, 2080, False, (128, 1, 0, 2))])
def test_streamed_raw_weights(bk, oracle, M, N, K, fused, plan):
    assert stream_plan(bk, False, M, N, K, fused)[:4] == plan
    rng = np.random.default_rng(M + N + K)
    A, W = synth.random_bits(rng, (M, K // 8)), synth.random_bits(rng, (N, K // 8))
    thr = synth.thresholds(rng, K, N) if fused else None
    out = torch.empty(M * N // 8 if fused else M * N * 4, dtype=torch.uint8, device="cuda")
    if fused:
        bk.bcnn_gemm_b1_fused(dev(A), dev(W), dev(thr), out, M, N, K, engine=bk.ENGINES["tc_i8"])
    else:
        bk.bcnn_gemm_b1(dev(A), dev(W), out, M, N, K, engine=bk.ENGINES["tc_i8"])
    torch.cuda.synchronize()
    acc = synth.unpack_bits(A).astype(np.float32) @ synth.unpack_bits(W).astype(np.float32).T       # exact: |sums| < 2^24
    if fused:
        assert np.array_equal(synth.unpack_bits(out.cpu().numpy().reshape(M, N // 8)), np.where(acc >= thr, 1, -1))
    else:
        assert np.array_equal(out.cpu().numpy().view(np.int32).reshape(M, N), acc.astype(np.int32))
    assert bk.bcnn_device_error() == 0


# ... and convolutions with padding, strides and odd pixel words, against the CUDA-core engine
@pytest.mark.parametrize("fused", [True, False])
@pytest.mark.parametrize("shape", [(16, 28, 29, 160, 512, 3, 1, 1), (40, 27, 27, 96, 1024, 3, 2, 1), (8, 30, 30, 256, 992, 5, 1, 2), (30, 15, 14, 512, 640, 1, 2, 0), (2, 9, 9, 64, 96, 3, 1, 1)])
def test_streamed_raw_convolutions(bk, oracle, shape, fused):
    B, H, W, C_in, C_out, k, stride, pad = shape
    rng = np.random.default_rng(C_in + C_out)
    K = k * k * C_in
    x, w = dev(synth.random_bits(rng, (B, H, W, C_in // 8))), dev(synth.random_bits(rng, (C_out, K // 8)))
    thr = dev(synth.thresholds(rng, K, C_out))
    OH, OW = bk.out_hw(H, W, k, k, stride, pad)
    res = []
    for e in ("tc_i8", "lop3"):
        out = torch.full((B * OH * OW * C_out // 8 * (1 if fused else 32),), 0x5a, dtype=torch.uint8, device="cuda")
        if fused:
            bk.bcnn_conv2d_b1_fused(x, w, thr, out, B, H, W, C_in, C_out, k, k, stride, pad, engine=bk.ENGINES[e])
        else:
            bk.bcnn_conv2d_b1(x, w, out, B, H, W, C_in, C_out, k, k, stride, pad, engine=bk.ENGINES[e])
        torch.cuda.synchronize()
        res.append(out)
    assert torch.equal(res[0], res[1])
    assert bk.bcnn_device_error() == 0
