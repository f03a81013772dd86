"""The work that users of this library have it do, as measurable cases.

Every case is one pass through the public entry points on resident gradients of M workers:

  step      Quantizer.step: scale agreement, [scale selection and sharing,] quantization, integer
            sum, reconstruction of the average gradient (one training iteration's aggregation)
  train     the single-scale stages called one by one, with the reconstruction fused into the SGD
            update with momentum and weight decay (the paper's optimizer settings)
  randk     GlobalRandK: K coordinates chosen and gathered, quantized, sparse update of the parameters
  gathered  the receiving side of a job spread over processes: the field-wise minimum of the processes'
            packed scale indices, then sum + reconstruction of the level rows of all workers

Ranges: 2 to 64 workers; 10^3 to 3.4*10^8 coordinates, odd counts included; binary32 and bfloat16
gradients; one segment, a layer table, 25 MiB buckets; single scale and 2 to 8 scales; 8-, 6-, 4- and
2-bit levels; 1- to 8-bit indices; L2 and L-inf scales; 16- and 32-bit draws.  Values follow the
recipes of ``workloads.py`` (normal, per-layer spread, Student-t(3), rare large coordinates), made on
the GPU.  Every integer of the path is defined bit for bit, and the scale is a binary64 sum rounded
once to binary32, so results are compared exactly.
"""
import math

import torch

from paper_2109_12497_b200 import binding as B
from paper_2109_12497_b200 import workloads as wl
from paper_2109_12497_b200.pipeline import Quantizer, RandKQuantizer

FMTS = {"i8": (B.UQ_FMT_I8, 127), "i6p": (B.UQ_FMT_I6P, 31), "i4x2": (B.UQ_FMT_I4X2, 7), "i2x4": (B.UQ_FMT_I2X4, 1)}
LEVEL_BITS = {"i8": 8, "i6p": 6, "i4x2": 4, "i2x4": 2}
LR, MU, WD = 0.1, 0.9, 5e-4


def _case(kind, M, d, dtype="f32", values="normal", segments="one", fmt="i8", N=1, ratio=8, idx_bits=0, norm="l2",
          rng_bits=32, K=0, R=1, name=None):
    c = dict(kind=kind, M=M, d=d, dtype=dtype, values=values, segments=segments, fmt=fmt, N=N, ratio=ratio,
             idx_bits=idx_bits, norm=norm, rng_bits=rng_bits, K=K, R=R)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one parameter tensor of a small layer, compressed by itself in a gradient hook: pure latency
        _case("step", 4, 4_099, "bf16", "outliers", "one", "i8", 8, 8, 4, "l2", 16, name="tensor_4k_multi"),
        # the sparsified quantizer of the paper's experiments (K = 10000 of a 25.6 M gradient)
        _case("randk", 8, 25_557_032, K=10_000, name="randk_10k_of_25m"),
        # a small network's whole gradient with its layer table
        _case("step", 8, 100_003, values="layers", segments="layers", name="layers_100k"),
        # workload c1: a small gradient of two workers, max norm
        _case("step", 2, 1 << 20, norm="linf", name="vector_1m"),
        # one 25 MiB bucket of a bfloat16 gradient as a data-parallel framework hands it over
        _case("step", 8, 13_107_200, "bf16", "outliers", name="bucket_25mib"),
        # workload c2: a 25.6 M convolutional gradient, 161 layers, 8-bit levels
        _case("step", 8, 25_557_032, values="layers", segments="layers", name="layers_25m"),
        # workload c3: the same gradient under the multi-scale quantizer, 2-bit shared index
        _case("step", 8, 25_557_032, values="layers", segments="layers", N=4, idx_bits=2, name="layers_25m_multi"),
        # two-scale compressor of the paper's experiments on its 14.7 M gradient, 6-bit wire
        _case("step", 4, 14_728_266, values="layers", segments="layers", fmt="i6p", N=2, ratio=16, idx_bits=1,
              name="layers_15m_two_scale"),
        # 2-bit levels on its 23.5 M gradient, with the optimizer
        _case("train", 8, 23_520_842, values="layers", segments="layers", fmt="i2x4", name="train_24m_2bit"),
        # workload c4: 16 workers, heavy-tailed values, two levels per byte
        _case("step", 16, 1 << 26, values="student_t3", fmt="i4x2", name="vector_64m_4bit"),
        # what one process of a 16-worker job does with the rows and indices that the others sent
        _case("gathered", 16, 25_557_032, values="layers", segments="layers", N=8, idx_bits=4, rng_bits=16, R=4,
              name="gathered_25m"),
        # workload c5: a 335 M bfloat16 gradient in 25 MiB buckets, 8 scales, 16-bit draws
        _case("step", 8, 335_141_888, "bf16", "outliers", "buckets", "i8", 8, 8, 4, "l2", 16, name="buckets_335m_multi"),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["train"] * 2 + ["randk", "gathered"])
    M = rng.choice([2, 3, 4, 4, 5, 8, 8, 8, 8, 12, 16, 16, 32, 64])
    hi = min(1.2e8, 5e8 / M)
    d = int(math.exp(rng.uniform(math.log(1e3), math.log(hi))))
    if rng.random() < 0.3:
        d = -(-d // 4096) * 4096                    # round sizes as well as odd ones
    dtype = rng.choice(["f32", "f32", "bf16"])
    fmt = rng.choice(["i8", "i8", "i8", "i4x2", "i2x4", "i6p"])
    N, ratio, idx_bits = rng.choice([(1, 8, 0), (1, 8, 0), (2, 16, 1), (2, 16, 8), (4, 8, 2), (8, 8, 4)])
    segments = rng.choice(["one", "layers", "buckets"])
    K = R = 0
    if kind == "train":
        N, ratio, idx_bits = 1, 8, 0
    if kind == "randk":
        K, segments = min(d, int(math.exp(rng.uniform(math.log(500), math.log(1e6))))), "one"
    if kind == "gathered":
        R = rng.choice([r for r in (2, 4, 8) if M % r == 0] or [M])
    values = {"layers": "layers"}.get(segments) or rng.choice(["normal", "outliers", "student_t3"])
    return _case(kind, M, d, dtype, values, segments, fmt, N, ratio, idx_bits, rng.choice(["l2", "l2", "l2", "linf"]),
                 rng.choice([16, 32]), K, R)


def _segments(c):
    d = c["d"]
    if c["segments"] == "layers":
        sizes = wl.layer_sizes(d, min(161, max(1, d // 8)), 1002)
        return [0] + [int(x) for x in sizes.cumsum()]
    if c["segments"] == "buckets":
        n = 25 * (1 << 20) // (4 if c["dtype"] == "f32" else 2)
        return list(range(0, d, n)) + [d]
    return None


def _gradients(c, seed, seg):
    """[M, stride] gradients on the GPU, from the seed alone; columns d and up are zero."""
    M, d, stride = c["M"], c["d"], -(-c["d"] // 32) * 32
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = torch.zeros((M, stride), dtype=torch.float32 if c["dtype"] == "f32" else torch.bfloat16, device="cuda")
    scale = None
    if c["values"] == "layers":
        n = len(seg) - 1
        std = 10.0 ** (torch.rand(n, generator=gen, device="cuda") * 4 - 5)
        lengths = torch.tensor([b - a for a, b in zip(seg, seg[1:])], device="cuda")
        scale = torch.repeat_interleave(std, lengths, output_size=d)
    elif c["values"] == "outliers":                  # the same 1 % of the coordinates on every worker
        scale = torch.where(torch.rand(d, generator=gen, device="cuda") < 0.01, 2.0, 0.02)
    for m in range(M):
        x = torch.randn(d, generator=gen, device="cuda")
        if scale is not None:
            x *= scale
        elif c["values"] == "student_t3":
            chi = torch.randn(d, generator=gen, device="cuda").square_()
            for _ in range(2):
                chi += torch.randn(d, generator=gen, device="cuda").square_()
            x /= (chi / 3).clamp_(min=1e-30).sqrt_()
            x *= 1e-3
        else:
            x *= 0.01
        g[m, :d] = x
    return g


def _settings(c):
    fmt, s = FMTS[c["fmt"]]
    return dict(s=s, scales=[s * c["ratio"] ** k for k in range(c["N"])] if c["N"] > 1 else None, fmt=fmt,
                idx_bits=c["idx_bits"], norm=B.UQ_NORM_L2 if c["norm"] == "l2" else B.UQ_NORM_LINF, rng_bits=c["rng_bits"])


def _columns(lev, c, n):
    """The part of the level rows that holds coordinates (units of 8; the 6-bit rows have two planes)."""
    units = -(-n // 8)
    if c["fmt"] != "i6p":
        return lev[:, :units * LEVEL_BITS[c["fmt"]]]
    stride = -(-n // 32) * 32
    return [lev[:, :units * 4], lev[:, stride // 2:stride // 2 + units * 2]]


def prepare(case, seed):
    c, d = case, case["d"]
    dtype = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    seg = _segments(c)
    g = _gradients(c, seed, seg)
    st = {"kind": c["kind"], "g": g, "seed": seed}
    if c["kind"] == "randk":
        q = RandKQuantizer(c["M"], d, c["K"], dtype, **_settings(c))
        st.update(q=q, theta=torch.randn(d, generator=torch.Generator(device="cuda").manual_seed(seed + 1), device="cuda"))
        st["outputs"] = {"theta": st["theta"], "sel": q.sel[:c["K"]], "values": q.inner.out[:c["K"]],
                         "lev": _columns(q.inner.lev, c, c["K"]), "W": q.inner.W, "status": q.status}
        if q.inner.idx is not None:
            st["outputs"]["idx"] = q.inner.idx[:-(-c["K"] // 8) * c["idx_bits"]]
        return st
    q = Quantizer(c["M"], d, dtype, seg, **_settings(c))
    st["q"] = q
    outputs = {"lev": _columns(q.lev, c, d), "W": q.W, "status": q.status}
    if q.idx is not None:
        outputs["idx"] = q.idx[:-(-d // 8) * c["idx_bits"]]
    if c["kind"] == "train":
        gen = torch.Generator(device="cuda").manual_seed(seed + 1)
        st["theta"] = torch.randn(d, generator=gen, device="cuda")
        st["momentum"] = torch.zeros(d, device="cuda")
        outputs.update(theta=st["theta"], momentum=st["momentum"])
    elif c["kind"] == "gathered":
        # what has arrived from the R processes: their level rows and, multi-scale, their packed indices
        q.agree_scale(g)
        if q.multi:
            per = c["M"] // c["R"]
            st["rows"] = torch.zeros((c["R"], q.idx.numel()), dtype=torch.uint8, device="cuda")
            part = B.Layout(per, d, q.stride, dtype, q.layout.seg_off)
            for r in range(c["R"]):
                B.uq_select_scale_multi(part, g[r * per:(r + 1) * per], q.W, q.scales, q.idx_bits, st["rows"][r], q.status)
            B.uq_index_min(st["rows"], q.idx_bits, q.idx)
        q.encode(g, seed)
        st["g"] = None
        outputs = {k: v for k, v in outputs.items() if k == "idx"}
        outputs["out"] = q.out[:d]
    st["outputs"] = outputs
    return st


def run(state):
    kind, q, g = state["kind"], state["q"], state["g"]
    state["seed"] += 1                               # every iteration draws anew
    seed = state["seed"]
    out = state["outputs"]
    if kind == "step":
        out["out"] = q.step(g, seed)
    elif kind == "train":
        q.agree_scale(g)
        q.encode(g, seed)
        q.aggregate_decode_update(state["theta"], state["momentum"], LR, MU, WD)
    elif kind == "randk":
        q.gather(g, seed)
        q.quantize(seed)
        q.update(state["theta"], LR)
    else:
        if q.multi:
            B.uq_index_min(state["rows"], q.idx_bits, q.idx)
        B.uq_decode(q.layout, q.lev, B.UQ_SRC_LEVELS, q.fmt, q.W, q.s, q.scales, q.idx, q.idx_bits, q.out)
    return out


def work(case):
    """Gradients (or rows) read once, levels, indices and results written once; the parameters and the
    momentum are read and written.  No arithmetic is counted: nothing here is a contraction."""
    c, M, d = case, case["M"], case["d"]
    elem = 4 if c["dtype"] == "f32" else 2
    lev, idx = LEVEL_BITS[c["fmt"]] / 8, c["idx_bits"] / 8
    if c["kind"] == "step":
        n = d * (M * (elem + lev) + idx + 4)
    elif c["kind"] == "train":
        n = d * (M * (elem + lev) + idx + 16)
    elif c["kind"] == "randk":
        n = c["K"] * (M * (elem + lev) + idx + 8 + 4 + 8)
    else:
        n = d * (M * lev + (c["R"] + 1) * idx + 4)
    return {"bytes": n, "flops": 0}


def tolerance(case):
    return "exact"
