"""Performance cases: what a user of the library runs, through its public entry points.

A case is a dict of plain values.  ``listed()`` names the fixed ones, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` builds what a program holds before the call (device inputs, packed weights, thresholds, prepared
weights where the library prefers them, a captured chain), ``run(state)`` is one pass, ``work(case)`` the bytes and
operations the pass cannot do without and ``tolerance(case)`` how far another correct implementation may be off.

Kinds of case:

* ``conv``      one binary convolution: k x k, stride 1 or 2, int32 output or packed signs
* ``gemm``      one binary matrix product, int32 or packed, on packed weights (weights that are new on each call) or on
                weights prepared once (a layer that is called again and again)
* ``chain``     a whole network of fused layers with device-resident packed activations, replayed from a CUDA graph (a
                server) or enqueued call by call
* ``block``     the residual path of the paper's building block on real-valued maps: binary 1x1 module, depth-wise 3x3
                module, binary 1x1 module; a down-sampling block also replicates its channels and pools its identity path
* ``branches``  one convolution module with P parallel binary branches, or the nine taps of a binary 3x3 convolution
* ``head``      global average pooling and the fully connected layer
* ``pack``      binarization of a real map: bias, sign, channel replication
"""
import math

import numpy as np
import torch

from paper_2010_00704_b200 import binding as bk
from paper_2010_00704_b200.chain import FusedChain
from paper_2010_00704_b200.workloads import BACKBONE18, BLOCK_STACK, ConvLayer

DEV = "cuda"


def listed():
    return [
        # one image through one layer: the smallest call, latency of the launch and of one pass over the layer
        dict(name="conv_single_3x3", kind="conv", B=1, H=32, W=32, c_in=128, c_out=128, k=3, stride=1, pad=1, out="int32"),
        # a down-sampling layer near the input: large map, few channels
        dict(name="conv_down_112", kind="conv", B=64, H=112, W=112, c_in=32, c_out=64, k=3, stride=2, pad=1, out="bits"),
        # a layer with odd extents and channel counts that are no powers of two (a detector's map, a pruned network)
        dict(name="conv_ragged", kind="conv", B=5, H=45, W=61, c_in=96, c_out=160, k=3, stride=1, pad=1, out="bits"),
        # matrix product whose weights are new on each call, packed result
        dict(name="gemm_4096", kind="gemm", M=4096, N=4096, K=4608, out="bits", prepared=False),
        # the sweep's largest product, integer result, weights laid out once
        dict(name="gemm_16384", kind="gemm", M=16384, N=16384, K=9216, out="int32", prepared=True),
        # the whole backbone: training-size batch, and a single image (a latency-bound server)
        dict(name="backbone_b256", kind="chain", net="backbone18", B=256, size=224, graph=True),
        dict(name="backbone_b1", kind="chain", net="backbone18", B=1, size=224, graph=True),
        # the four-layer residual stack, enqueued call by call
        dict(name="block_stack_b128", kind="chain", net="block_stack", B=128, size=28, graph=False),
        # the paper's own network: its level-2 down-sampling block, a two-branch module of level 3, its head
        dict(name="block_down_112", kind="block", B=64, size=112, c=128, r=2, s=2),
        dict(name="branches_p2_28", kind="branches", B=64, size=28, c=256, p=2, k=1),
        dict(name="head_b256", kind="head", B=256, size=7, c=1024, n=1000),
        # a real-valued map enters the binary part of a network
        dict(name="pack_28", kind="pack", B=128, size=28, c_in=256, r=1),
    ]


# ---- drawn cases -------------------------------------------------------------------------------------

def _log(rng, lo, hi):
    """Integer spread evenly over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_conv(rng):
    k = rng.choice((1, 3, 3, 5))
    out = rng.choice(("bits", "bits", "int32"))
    return dict(kind="conv", B=_log(rng, 1, 256), H=_log(rng, 7, 224), W=_log(rng, 7, 224), c_in=32 * _log(rng, 1, 16),
                c_out=32 * _log(rng, 1, 16) if out == "bits" else _log(rng, 10, 512), k=k, stride=rng.choice((1, 1, 2)), pad=k // 2, out=out)


def _draw_gemm(rng):
    out = rng.choice(("bits", "int32"))
    return dict(kind="gemm", M=_log(rng, 1, 16384), N=32 * _log(rng, 1, 512) if out == "bits" else _log(rng, 10, 16384),
                K=32 * _log(rng, 1, 288), out=out, prepared=rng.random() < 0.5)


def _draw_chain(rng):
    if rng.random() < 0.7:
        return dict(kind="chain", net="backbone18", B=_log(rng, 1, 256), size=32 * rng.randint(3, 7), graph=rng.random() < 0.5)
    return dict(kind="chain", net="block_stack", B=_log(rng, 1, 256), size=2 * rng.randint(4, 14), graph=rng.random() < 0.5)


def _draw_block(rng):
    r, s = rng.choice(((1, 1), (1, 1), (2, 2)))
    return dict(kind="block", B=_log(rng, 1, 256), size=s * _log(rng, 4, 56), c=64 * _log(rng, 1, 16), r=r, s=s)


def _draw_branches(rng):
    p, k = rng.choice(((2, 1), (2, 1), (3, 1), (4, 1), (9, 3)))
    return dict(kind="branches", B=_log(rng, 1, 256), size=_log(rng, 7, 112), c=32 * _log(rng, 1, 16), p=p, k=k)


def _draw_head(rng):
    return dict(kind="head", B=_log(rng, 1, 256), size=rng.randint(4, 14), c=8 * _log(rng, 8, 256), n=_log(rng, 10, 4000))


def _draw_pack(rng):
    c_in, r = rng.choice(((32 * _log(rng, 1, 32), 1), (4, 8), (8, 4), (16, 2), (32, 2), (64, 4)))
    return dict(kind="pack", B=_log(rng, 1, 256), size=_log(rng, 7, 224), c_in=c_in, r=r)


def draw(rng):
    make = rng.choice((_draw_conv, _draw_conv, _draw_conv, _draw_gemm, _draw_gemm, _draw_chain, _draw_chain, _draw_block, _draw_block,
                       _draw_branches, _draw_head, _draw_pack))
    while True:
        case = make(rng)
        w = work(case)
        if w["bytes"] <= 4e8 and w["flops"] <= (1e11 if case["kind"] == "branches" else 1e12):
            return case


# ---- what a program holds before the call ------------------------------------------------------------

def _layer(case):
    return ConvLayer("layer", case["H"], case["W"], case["c_in"], case["c_out"], case["k"], case["stride"], case["pad"])


def _chain_layers(case):
    """The network's layers at the case's input size (the tables are written for 224 and 28 pixels)."""
    base, layers = (224, BACKBONE18) if case["net"] == "backbone18" else (28, BLOCK_STACK)
    return [ConvLayer(l.name, l.H * case["size"] // base, l.W * case["size"] // base, l.C_in, l.C_out, l.k, l.stride, l.pad) for l in layers]


class _Maker:
    """Device tensors from one seed, with the distributions the path meets: fair sign bits, standard normal maps and
    biases, batch norms that bring a K-term sum back to unit variance, thresholds uniform on [-K/4, K/4]."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)

    def bits(self, *shape):
        return torch.randint(0, 256, shape, dtype=torch.uint8, device=DEV, generator=self.g)

    def f32(self, *shape, scale=1.0, mean=0.0):
        return torch.randn(shape, device=DEV, generator=self.g) * scale + mean

    def f16(self, *shape):
        return torch.randn(shape, device=DEV, generator=self.g, dtype=torch.float16)

    def thresholds(self, n, K):
        return torch.randint(-(K // 4), K // 4 + 1, (n,), dtype=torch.int32, device=DEV, generator=self.g)

    def module(self, c, K, p=1):
        """Batch norm (scale, shift), PReLU slope and next bias of a module with c outputs and K-term sums."""
        return dict(scale=self.f32(p, c, scale=K ** -0.5), shift=self.f32(p, c, scale=0.5), slope=self.f32(c, scale=0.05, mean=0.25), nb=self.f32(c, scale=0.5))


def _prepared(w, c_out, K):
    buf = torch.empty(bk.bcnn_prepared_weights_bytes(c_out, K), dtype=torch.uint8, device=DEV)
    return bk.bcnn_prepare_weights(w, buf, c_out, K)


def _empty_out(out, rows, cols):
    return torch.empty(rows, cols, dtype=torch.int32, device=DEV) if out == "int32" else torch.empty(rows, cols // 8, dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    m, kind = _Maker(seed), case["kind"]
    s = dict(case=case, kind=kind)
    if kind == "conv":
        l, B = _layer(case), case["B"]
        fused = case["out"] == "bits"
        s.update(x=m.bits(B, l.H, l.W, l.C_in // 8), w=m.bits(l.C_out, l.k, l.k, l.C_in // 8), thr=m.thresholds(l.C_out, l.K) if fused else None,
                 out=_empty_out(case["out"], l.M(B), l.C_out), args=(B, l.H, l.W, l.C_in, l.C_out, l.k, l.k, l.stride, l.pad), prep=None)
        if bk.bcnn_prepared_preferred(*s["args"], fused=fused):
            s["prep"] = _prepared(s["w"], l.C_out, l.K)
    elif kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        s.update(x=m.bits(M, K // 8), w=m.bits(N, K // 8), thr=m.thresholds(N, K) if case["out"] == "bits" else None,
                 out=_empty_out(case["out"], M, N), args=(M, N, K), prep=None)
        if case["prepared"]:
            s["prep"] = _prepared(s["w"], N, K)
    elif kind == "chain":
        layers, rng = _chain_layers(case), np.random.default_rng(seed)
        ws = [rng.integers(0, 256, (l.C_out, l.k, l.k, l.C_in // 8), dtype=np.uint8) for l in layers]
        ts = [rng.integers(-(l.K // 4), l.K // 4 + 1, l.C_out).astype(np.int32) for l in layers]
        if case["net"] == "backbone18":
            chain = FusedChain(layers, case["B"], ws, ts, real_input_shape=(case["size"], case["size"], 4),
                               bias=rng.standard_normal(32).astype(np.float32), replicate=8)
            chain.x_real.normal_(generator=m.g)
        else:
            chain = FusedChain(layers, case["B"], ws, ts)
            chain.in_bits.random_(0, 256, generator=m.g)
        if case["graph"]:
            chain.capture()
        s.update(chain=chain)
    elif kind == "block":
        B, H, C, R, S = case["B"], case["size"], case["c"], case["r"], case["s"]
        O = (H - 1) // S + 1
        s.update(x=m.f16(B, H, H, C // R), x_bits=m.bits(B, H, H, C // 8), w1=m.bits(C, C // 8), w2=m.bits(C, C // 8), m1=m.module(C, C), m2=m.module(C, C),
                 dw=m.f32(C, 3, 3, scale=1 / 3), md=m.module(C, 1),
                 wide=torch.empty(B, H, H, C, dtype=torch.float16, device=DEV) if R > 1 else None,
                 pooled=torch.empty(B, O, O, C, dtype=torch.float16, device=DEV) if S > 1 else None,
                 y1=torch.empty(B, H, H, C, dtype=torch.float16, device=DEV), yd=torch.empty(B, O, O, C, dtype=torch.float16, device=DEV),
                 yd_bits=torch.empty(B, O, O, C // 8, dtype=torch.uint8, device=DEV), y2=torch.empty(B, O, O, C, dtype=torch.float16, device=DEV),
                 y2_bits=torch.empty(B, O, O, C // 8, dtype=torch.uint8, device=DEV))
    elif kind == "branches":
        B, H, C, P = case["B"], case["size"], case["c"], case["p"]
        s.update(x_bits=m.bits(B, H, H, P * C // 8), w=m.bits(P, C, C // 8), m=m.module(C, P * C, P), identity=m.f16(B, H, H, C),
                 # what a tap outside the image adds: the signs of the branch's biases times its weights, C terms of +-1
                 pad=(2 * torch.randint(0, C + 1, (P, C), device=DEV, generator=m.g) - C).to(torch.int32) if case["k"] > 1 else None,
                 y=torch.empty(B, H, H, C, dtype=torch.float16, device=DEV), y_bits=torch.empty(B, H, H, C // 8, dtype=torch.uint8, device=DEV))
    elif kind == "head":
        B, H, C, N = case["B"], case["size"], case["c"], case["n"]
        s.update(x=m.f16(B, H, H, C), w=m.f32(N, C, scale=C ** -0.5), bias=m.f32(N), pooled=torch.empty(B, C, device=DEV), logits=torch.empty(B, N, device=DEV))
    else:
        B, H, C = case["B"], case["size"], case["c_in"] * case["r"]
        s.update(x=m.f32(B, H, H, case["c_in"]), bias=m.f32(C), out=torch.empty(B, H, H, C // 8, dtype=torch.uint8, device=DEV))
    return s


# ---- one pass ------------------------------------------------------------------------------------------

def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "conv":
        if s["prep"] is not None:
            return bk.bcnn_conv2d_b1_prepared(s["x"], s["prep"], s["thr"], s["out"], *s["args"])
        if s["thr"] is not None:
            return bk.bcnn_conv2d_b1_fused(s["x"], s["w"], s["thr"], s["out"], *s["args"])
        return bk.bcnn_conv2d_b1(s["x"], s["w"], s["out"], *s["args"])
    if kind == "gemm":
        if s["prep"] is not None:
            return bk.bcnn_gemm_b1_prepared(s["x"], s["prep"], s["thr"], s["out"], *s["args"])
        if s["thr"] is not None:
            return bk.bcnn_gemm_b1_fused(s["x"], s["w"], s["thr"], s["out"], *s["args"])
        return bk.bcnn_gemm_b1(s["x"], s["w"], s["out"], *s["args"])
    if kind == "chain":
        return s["chain"].run()
    if kind == "block":
        B, H, C, R, S = case["B"], case["size"], case["c"], case["r"], case["s"]
        O = (H - 1) // S + 1
        identity = s["x"] if R == 1 else bk.bcnn_avgpool(s["x"], s["wide"], B, H, H, C // R, R, 1)
        a, d, b = s["m1"], s["md"], s["m2"]
        # module 1 feeds the depth-wise module, which reads the real map only
        bk.bcnn_conv2d_b1_module(s["x_bits"], s["w1"], a["scale"], a["shift"], identity, a["slope"], None, s["y1"], None, B, H, H, C, C, 1, 1, 1, 0)
        bk.bcnn_dwconv3x3_module(s["y1"], s["dw"], d["scale"], d["shift"], d["slope"], d["nb"], s["yd"], s["yd_bits"], B, H, H, C, 1, S)
        bk.bcnn_conv2d_b1_module(s["yd_bits"], s["w2"], b["scale"], b["shift"], s["yd"], b["slope"], b["nb"], s["y2"], s["y2_bits"], B, O, O, C, C, 1, 1, 1, 0)
        out = dict(y1=s["y1"], yd=s["yd"], y=s["y2"], bits=s["y2_bits"])
        if S > 1:
            out["pooled"] = bk.bcnn_avgpool(s["x"], s["pooled"], B, H, H, C // R, R, S)
        return out
    if kind == "branches":
        B, H, C, P, k, m = case["B"], case["size"], case["c"], case["p"], case["k"], s["m"]
        return bk.bcnn_conv2d_b1_branches(s["x_bits"], s["w"], m["scale"], m["shift"], s["pad"], s["identity"], m["slope"], m["nb"], s["y"], s["y_bits"],
                                          B, H, H, C, C, P, k, k)
    if kind == "head":
        B, H, C, N = case["B"], case["size"], case["c"], case["n"]
        bk.bcnn_gap(s["x"], s["pooled"], B, H, H, C)
        return bk.bcnn_fc(s["pooled"], s["w"], s["bias"], s["logits"], B, C, N), s["pooled"]
    B, H = case["B"], case["size"]
    return bk.bcnn_pack(s["x"], s["bias"], s["out"], B, H, H, case["c_in"], case["r"])


# ---- what a pass cannot do without -----------------------------------------------------------------------

def work(case):
    """Bytes: inputs read once, outputs written once (a block's maps between its calls are outputs of those calls; a
    chain's packed activations between its layers are not counted).  Operations: two per binary or real multiply-add."""
    kind = case["kind"]
    if kind == "conv":
        l, B = _layer(case), case["B"]
        out = l.M(B) * l.C_out * 4 if case["out"] == "int32" else l.out_bits_bytes(B) + 4 * l.C_out
        return dict(bytes=l.in_bytes(B) + l.w_bytes() + out, flops=l.ops(B))
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        out = M * N * 4 if case["out"] == "int32" else M * N // 8 + 4 * N
        return dict(bytes=(M + N) * K // 8 + out, flops=2 * M * N * K)
    if kind == "chain":
        layers, B = _chain_layers(case), case["B"]
        first = B * case["size"] ** 2 * 16 if case["net"] == "backbone18" else layers[0].in_bytes(B)
        return dict(bytes=first + sum(l.w_bytes() + 4 * l.C_out for l in layers) + layers[-1].out_bits_bytes(B), flops=sum(l.ops(B) for l in layers))
    if kind == "block":
        B, H, C, R, S = case["B"], case["size"], case["c"], case["r"], case["s"]
        O = (H - 1) // S + 1
        big, small = B * H * H * C, B * O * O * C
        bits, maps = big // 8 + 3 * small // 8, 2 * big // R + 2 * 2 * big + (3 + 1) * 2 * small
        if R > 1:
            maps += 2 * 2 * big - 2 * big // R
        if S > 1:
            maps += 2 * small + 2 * big // R
        return dict(bytes=bits + maps + C * C // 4 + 80 * C, flops=2 * (big + small) * C + 18 * small)
    if kind == "branches":
        B, H, C, P = case["B"], case["size"], case["c"], case["p"]
        M = B * H * H
        return dict(bytes=M * C * 4 + M * C // 8 + M * P * C // 8 + P * C * C // 8 + (2 * P + 2) * 4 * C, flops=2 * M * C * C * P)
    if kind == "head":
        B, H, C, N = case["B"], case["size"], case["c"], case["n"]
        return dict(bytes=B * H * H * C * 2 + 4 * (B * C + N * C + N + B * N), flops=B * H * H * C + 2 * B * C * N)
    n = case["B"] * case["size"] ** 2 * case["c_in"]
    return dict(bytes=4 * n + n * case["r"] // 8 + 4 * case["c_in"] * case["r"], flops=n * case["r"])


def tolerance(case):
    """Binary products are integers, and the module's steps are single fp32 operations in a stated order: exact.  The
    depth-wise sums (nine fp32 products, stored as fp16) may round the other way on a few elements, and a sign that flips
    with one changes the sums behind it; pooling and the head are fp32 sums."""
    if case["kind"] == "block":
        return {"rel": 3e-4, "max": 0.5, "differ": 1e-4}
    if case["kind"] == "head":
        return {"rel": 1e-5}
    return "exact"
