"""Workloads of the W4A16 layer library, for timing: what a program that quantizes a model's linear
layers, searches their scales and serves them asks of the public entry points.

A case is a dict of plain values.  `listed()` names the ones to look at first, `draw(rng)` gives
more of the same ranges, `prepare` makes what such a program has in hand before the call (inputs,
packed weights, output buffers, a captured decode step), `run` makes one pass.  Shapes are those of
the Llama-2 7B / 13B / 70B linear layers that the tests and the benchmark use, token counts those of
the decode-to-prefill sweep (1 .. 8192) with ragged ones between.  Inputs have the structure that the
method is about: fp16 weights ~ N(0, 0.02^2), activations ~ N(0, 1) in which a seeded 1 % of the input
channels is 20 times larger.
"""
from __future__ import annotations

import math

import torch

from paper_2306_00978_b200 import binding

GROUPS = (64, 128, 256, 512, 1024)
CALIBRATION_TOKENS = 128
# no drawn call multiplies more than the largest listed one
LARGEST_MNK = 8192 * 11008 * 4096


def listed():
    return [
        # one projection for one sequence, called by itself: the smallest call, where the host path counts
        dict(name="linear_4096_4096_m1", kind="linear", M=1, N=4096, K=4096, group=128, alpha=0.5),
        # the linears of a 7B decoder layer for one sequence, replayed as a graph as a decode loop does
        dict(name="layer_7b_m1", kind="layer", M=1, hidden=4096, inter=11008, group=128, alpha=0.5),
        # the same layer for 32 sequences decoded together
        dict(name="layer_7b_m32", kind="layer", M=32, hidden=4096, inter=11008, group=128, alpha=0.5),
        # 70B down projection, 16 sequences: many weight bytes, a long reduction
        dict(name="linear_28672_8192_m16", kind="linear", M=16, N=8192, K=28672, group=128, alpha=0.5),
        # gate / up projection on the dense 3-bit storage, two sequences (a small beam)
        dict(name="int3_4096_11008_m2", kind="int3", M=2, N=11008, K=4096, group=128, alpha=0.5),
        # a short prompt of odd length through the 13B up projection, groups of 64
        dict(name="linear_5120_13824_m100_g64", kind="linear", M=100, N=13824, K=5120, group=64, alpha=0.5),
        # a ragged prompt through a square projection: few tiles for many SMs
        dict(name="linear_4096_4096_m333", kind="linear", M=333, N=4096, K=4096, group=128, alpha=1.0),
        # prefill of 2048 tokens through the 13B down projection
        dict(name="linear_13824_5120_m2048", kind="linear", M=2048, N=5120, K=13824, group=128, alpha=0.5),
        # the largest prefill of the sweep: 8192 tokens through a 7B gate / up projection
        dict(name="linear_4096_11008_m8192", kind="linear", M=8192, N=11008, K=4096, group=128, alpha=0.5),
        # offline: quantize and pack one 7B gate / up projection
        dict(name="quantize_4096_11008", kind="quantize", N=11008, K=4096, group=128, alpha=0.5, bits=4, symmetric=False),
        # offline: the paper's scale search, 20 grid points, 512 calibration tokens
        dict(name="alpha_search_4096_4096_m512", kind="alpha", M=512, N=4096, K=4096, group=128, points=20),
        # offline: clip search over 20 ratios and the 3-bit quantizer that uses its result
        dict(name="clip_search_4096_4096", kind="clip", N=4096, K=4096, group=128, alpha=0.5, bits=3, ratios=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dim(rng, lo=1024, hi=28672):
    """A multiple of 128 (what the layer accepts), spread over the logarithm of the range."""
    return 128 * max(lo // 128, min(hi // 128, _log_int(rng, lo // 128, hi // 128)))


def _group(rng, K, most=1024):
    fits = [g for g in GROUPS if K % g == 0 and g <= most]
    return rng.choice([128] * len(fits) + fits)          # 128 is the paper's setting: half of the draws


def draw(rng):
    kind = rng.choice(["linear"] * 7 + ["layer", "int3", "quantize", "alpha", "clip"])
    alpha = rng.choice([0.5, 0.5, 0.0, 1.0])
    if kind == "layer":
        hidden = _dim(rng, 2048, 8192)
        inter = 128 * int(round(hidden * rng.uniform(2.5, 3.6) / 128))
        return dict(kind=kind, M=_log_int(rng, 1, 64), hidden=hidden, inter=inter, group=_group(rng, math.gcd(hidden, inter), 128), alpha=alpha)
    N, K = _dim(rng), _dim(rng)
    if kind == "linear":
        M = max(1, min(_log_int(rng, 1, 8192), LARGEST_MNK // (N * K)))
        return dict(kind=kind, M=M, N=N, K=K, group=_group(rng, K), alpha=alpha)
    if kind == "int3":
        return dict(kind=kind, M=_log_int(rng, 1, 64), N=N, K=K, group=_group(rng, K), alpha=alpha)
    if kind == "quantize":
        return dict(kind=kind, N=N, K=K, group=_group(rng, K), alpha=rng.choice([0.5, 0.35, 0.0, 1.0]),
                    bits=rng.choice([4, 4, 3]), symmetric=rng.random() < 0.25)
    N, K = min(N, 8192), min(K, 8192)
    if kind == "alpha":
        return dict(kind=kind, M=_log_int(rng, 16, 1024), N=N, K=K, group=_group(rng, K, 128), points=rng.choice([10, 20]))
    return dict(kind=kind, N=N, K=K, group=_group(rng, K, 128), alpha=alpha, bits=rng.choice([3, 4]), ratios=rng.choice([8, 16, 20, 32]))


class _Inputs:
    """Seeded tensors on the device; channels 20 times larger are the same for activations and calibration."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) * 7919 + 17)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda", dtype=torch.float32)

    def weight(self, N, K):
        return (self.normal(N, K) * 0.02).to(torch.float16)

    def gain(self, K):
        gain = torch.ones(K, device="cuda")
        gain[torch.randperm(K, generator=self.g, device="cuda")[: max(1, round(0.01 * K))]] = 20.0
        return gain

    def activations(self, M, gain):
        return (self.normal(M, gain.numel()) * gain).to(torch.float16)

    def act_mean_abs(self, gain):
        return self.activations(CALIBRATION_TOKENS, gain).float().abs().mean(dim=0)


def _packed(inp, N, K, group, alpha, stat, bits=4):
    return (*binding.quantize_pack(inp.weight(N, K), stat, alpha, group, bits=bits), N)


def _prepare_layer(case, inp):
    """The four calls of a decoder layer (q/k/v, o, gate/up, down) on activations that are not yet divided
    by s, captured once; a decode loop writes its activations into `x` and replays."""
    h, f, M, group, alpha = case["hidden"], case["inter"], case["M"], case["group"], case["alpha"]
    calls = []
    for K, widths in ((h, (h, h, h)), (h, (h,)), (h, (f, f)), (f, (h,))):
        gain = inp.gain(K)
        stat = inp.act_mean_abs(gain)
        mats = [_packed(inp, N, K, group, alpha, stat) for N in widths]
        outs = [torch.empty((M, N), dtype=torch.float16, device="cuda") for N in widths]
        calls.append((inp.activations(M, gain), binding.inverse_channel_scale(stat, alpha, K), mats, K, outs))

    def step():
        for x, inv_s, mats, K, outs in calls:
            binding.linear_multi_scaled(x, inv_s, mats, K, group, outs=outs)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()                                            # workspace and device set-up before the capture
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    return dict(case=case, calls=calls, graph=graph, outs=[y for c in calls for y in c[4]])


def prepare(case, seed):
    inp, kind = _Inputs(seed), case["kind"]
    if kind == "layer":
        return _prepare_layer(case, inp)
    N, K = case["N"], case["K"]
    gain = inp.gain(K)
    stat = inp.act_mean_abs(gain)
    if kind in ("linear", "int3"):
        qweight, scales, zeros, _ = _packed(inp, N, K, case["group"], case["alpha"], stat, 3 if kind == "int3" else 4)
        if kind == "int3":
            qweight = binding.pack_int3(qweight, N, K)
        s = binding.channel_scale(stat, case["alpha"], K)
        x = (inp.activations(case["M"], gain).float() / s).to(torch.float16)
        return dict(case=case, x=x, qweight=qweight, scales=scales, zeros=zeros)
    state = dict(case=case, W=inp.weight(N, K), stat=stat)
    if kind == "alpha":
        state["X"] = inp.activations(case["M"], gain)
        state["alphas"] = [i / case["points"] for i in range(case["points"])]
    if kind == "clip":
        state["ratios"] = [1.0 - 0.5 * i / case["ratios"] for i in range(case["ratios"])]
    return state


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "layer":
        state["graph"].replay()
        return state["outs"]
    if kind == "linear":
        return binding.linear(state["x"], state["qweight"], state["scales"], state["zeros"], c["N"], c["K"], c["group"])
    if kind == "int3":
        return binding.linear_int3(state["x"], state["qweight"], state["scales"], state["zeros"], c["N"], c["K"], c["group"])
    if kind == "quantize":
        return binding.quantize_pack(state["W"], state["stat"], c["alpha"], c["group"], bits=c["bits"], symmetric=c["symmetric"])
    if kind == "alpha":
        return binding.search_alpha(state["W"], state["stat"], state["X"], c["group"], state["alphas"])
    ratios = binding.search_clip(state["W"], state["stat"], c["alpha"], c["group"], state["ratios"], bits=c["bits"])
    return (ratios, *binding.quantize_pack(state["W"], state["stat"], c["alpha"], c["group"], clip_ratio=ratios, bits=c["bits"]))


def _packed_bytes(N, K, group, bits=4):
    stored = min(group, 128)
    return N * K * bits / 8 + N * (K / stored) * 2.5      # codes, fp16 scales, 4-bit zero points


def work(case):
    kind = case["kind"]
    if kind == "layer":
        h, f, M, g = case["hidden"], case["inter"], case["M"], case["group"]
        nk = 4 * h * h + 3 * h * f
        packed = 4 * _packed_bytes(h, h, g) + 2 * _packed_bytes(f, h, g) + _packed_bytes(h, f, g)
        # four inputs with their inverse scales, seven outputs
        return dict(bytes=packed + (2 * M + 4) * (3 * h + f) + 2 * M * (5 * h + 2 * f), flops=2 * M * nk)
    N, K, g = case["N"], case["K"], case["group"]
    if kind in ("linear", "int3"):
        M = case["M"]
        return dict(bytes=_packed_bytes(N, K, g, 3 if kind == "int3" else 4) + 2 * M * K + 2 * M * N, flops=2 * M * N * K)
    if kind == "quantize":
        # per weight: scale, two comparisons, quotient, rounding, zero point
        return dict(bytes=2 * N * K + 4 * K + _packed_bytes(N, K, g), flops=6 * N * K)
    if kind == "alpha":
        M, n = case["M"], case["points"]
        return dict(bytes=2 * N * K + 2 * M * K + 4 * K + 4 * n, flops=2 * (n + 1) * M * N * K)
    # per weight and ratio: quotient, rounding, two comparisons, scale, difference, square, sum
    return dict(bytes=2 * N * K + 4 * K + 4 * N * (K / g) + _packed_bytes(N, K, g), flops=8 * N * K * case["ratios"])


def tolerance(case):
    kind = case["kind"]
    if kind in ("quantize", "clip"):
        return "exact"                                    # packed codes, zero points, scales and ratios have one right value
    if kind == "alpha":
        # losses are means of squared output errors: fp16 rounding of the layer's outputs moves them by a few 1e-5
        return dict(rel=1e-3, max=2e-3)
    # an fp16 output is rounded to 2.1e-4 (2-norm); with the fp16 rounding of (q - z) * Delta 2.9e-4 against fp64
    return dict(rel=1e-3, max=8e-3)


def _dequantized(qweight, scales, zeros, N, K, bits=4):
    """(q - z) * Delta in fp64 [N][K], from the packed arrays (layout: include/awq_b200.h)."""
    if bits == 3:
        u = qweight.view(torch.int32).view(-1, 3)
        last = ((u[:, 0] >> 3) & 0x11111111) | ((u[:, 1] >> 2) & 0x22222222) | ((u[:, 2] >> 1) & 0x44444444)
        words = torch.cat([u & 0x77777777, last[:, None]], dim=1).contiguous()
    else:
        words = qweight.view(torch.int32)
    # a word's byte b holds column {0, 2, 1, 3}[b] of its four, rows g (low nibble) and g + 8 (high)
    b = words.view(torch.uint8).view(N // 16, K // 64, 8, 4, 4, 4)[..., [0, 2, 1, 3]]       # band, tile, g, t, j, column
    q = torch.stack([b & 15, b >> 4], dim=1).permute(0, 1, 3, 2, 5, 4, 6).reshape(N, K)     # band, h, g, tile, j, t, column
    stored = scales.shape[1]
    z = zeros.view(N // 32, stored, 2, 8)
    z = torch.stack([z & 15, z >> 4], dim=0).permute(1, 3, 0, 4, 2).reshape(N, stored, 1)   # pair, band, h, g, group
    d = scales.permute(0, 2, 1).reshape(N, stored, 1)
    return ((q.view(N, stored, -1).double() - z.double()) * d.double()).view(N, K)


def _quantized(W, s, group, top=15.0):
    """(q - z) * Delta in fp64 by the quantizer's definition: fp32 w' and quotients, Delta kept in fp16."""
    w = (W.float() * s).view(W.shape[0], -1, group)
    mn, mx = w.amin(dim=2, keepdim=True), w.amax(dim=2, keepdim=True)
    d = ((mx - mn) / torch.full_like(mn, top)).half()
    d = torch.where(torch.isfinite(d) & (d != 0), d, torch.ones_like(d)).float()
    z = torch.round(-mn / d).clamp(0.0, top)
    q = (torch.round(w / d) + z).clamp(0.0, top)
    return ((q - z).double() * d.double()).view(W.shape)


def exact(case, seed):
    """What `run` returns, in 64 bits, from the inputs that `prepare` makes; None where only packed arrays come back."""
    kind = case["kind"]
    if kind in ("quantize", "clip"):
        return None
    state = prepare(case, seed)
    if kind == "layer":
        return [(x.double() * inv_s.double()) @ _dequantized(*m[:3], m[3], K).t() for x, inv_s, mats, K, _ in state["calls"] for m in mats]
    if kind != "alpha":
        packed = (state["qweight"], state["scales"], state["zeros"], case["N"], case["K"])
        return state["x"].double() @ _dequantized(*packed, bits=3 if kind == "int3" else 4).t()
    W, X, stat = state["W"], state["X"], state["stat"]
    target = X.double() @ W.double().t()
    losses = []
    for alpha in state["alphas"]:
        # the statistic is positive and finite here; alpha is an fp32 argument, s an fp32 array
        a32 = torch.tensor(alpha, dtype=torch.float32).double().item()
        s = stat.sqrt() if alpha == 0.5 else (stat.double() ** a32).float()
        y = (X.float() / s).half().double() @ _quantized(W, s, case["group"]).t()
        losses.append(float((y - target).square().mean()))
    return (losses, None)
