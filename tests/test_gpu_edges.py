"""The sizes at which the library changes from one kernel, grid or access width to another, each side of the
line against the CPU oracle (parity.py: integers and scale bits equal, values within its derived bound)."""
import numpy as np
import pytest
import torch

from oracle import uq_oracle as o
from paper_2109_12497_b200 import binding as B
from paper_2109_12497_b200 import workloads as wl
from parity import _check_parity, check_parity, ulp_distance

pytestmark = pytest.mark.gpu


# one-kernel step: 8 CTAs up to 1024 units of 8 coordinates, a cluster up to 4096 units, a grid above: of 128
# threads per CTA up to 148 * 128 units, then more, and more than one pass per thread (values read again) beyond one unit
# per register set
@pytest.mark.parametrize("M,d", [(2, 8 * 1024), (2, 8 * 1024 + 1), (2, 8 * 4096), (2, 8 * 4096 + 1), (8, 8 * 4096 - 7), (3, 8 * 4097),
                                 (1, 8 * 4096), (2, 8 * 148 * 128), (1, 8 * 148 * 128 + 1), (5, 8 * 148 * 160 + 9), (8, 8 * 148 * 480 + 1),
                                 (8, 8 * 148 * 512 + 1), (8, 2 * 8 * 148 * 512 + 9)])
@pytest.mark.parametrize("dtype,scales,rng_bits", [(wl.F32, (127,), 16), (wl.BF16, (7, 56), 32), (wl.F32, (7, 56, 448), 32),
                                                   (wl.BF16, (127,), 16)])
def test_one_kernel_step_at_the_edges_of_its_grids(M, d, dtype, scales, rng_bits):
    w = wl.scaled("c3" if len(scales) > 1 else "c1", d, M=M, dtype=dtype, norm=wl.NORM_L2, fmt="i8", s=scales[0],
                  scales=scales, idx_bits=2, rng_bits=rng_bits, segments="one", seed=d)
    assert _check_parity(w, wl.generate(w), None, "one")["q"].one_kernel


# many workers of a small gradient: both sides of the lines between one kernel and one per stage, with the sums (20
# workers or more) and for selection and levels alone (8 or more), with and without a row that d ends in
@pytest.mark.parametrize("M,d", [
    (24, 148 * 4 * 256), (25, 148 * 4 * 256), (64, 148 * 4 * 256), (64, 148 * 4 * 256 + 1), (19, 50_001), (20, 50_001), (20, 239_999),
    (20, 240_001), (32, 93 * 256), (32, 94 * 256), (7, 9_001), (8, 239_999), (8, 240_001), (25, 351 * 256), (25, 352 * 256), (16, 9_001),
    (25, 124_999), (25, 125_001),
])
@pytest.mark.parametrize("name", ["c2", "c3"])
@pytest.mark.parametrize("segments", ["one", "layers161"])
def test_many_workers_of_a_small_gradient(name, d, M, segments):
    w = wl.scaled(name, d, M=M, segments=segments)
    check_parity(w, wl.generate(w))


# norms of large binary32 gradients: four workers' rows per CTA from 148 * 4 * 8 groups of a tile of 8192
# coordinates, with few segments; one row per CTA below.  Maximum exact, Euclidean within one unit in the last place
@pytest.mark.parametrize("M", [2, 5, 8])
@pytest.mark.parametrize("extra", [-8192, 0, 8192 + 1])
@pytest.mark.parametrize("nseg", [1, 7])
def test_norms_of_large_gradients(M, extra, nseg):
    groups = (M + 3) // 4
    d = (148 * 4 * 8 // groups) * 8192 + extra
    stride = (d + 31) // 32 * 32
    g = torch.randn(M, stride, device="cuda", generator=torch.Generator("cuda").manual_seed(d + M))
    seg = None if nseg == 1 else np.array([0, 5, 8192, 8192, 16384 * 3 + 1, d // 2, d - 3, d], dtype=np.int64)
    lay = B.Layout(M, d, stride, torch.float32, None if seg is None else torch.from_numpy(seg).cuda())
    W, status = torch.empty(nseg, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(lay.workspace_bytes(), dtype=torch.uint8, device="cuda")
    g_np = g.cpu().numpy()[:, :d]
    for norm, onorm, ulps in ((B.UQ_NORM_LINF, o.NORM_LINF, 0), (B.UQ_NORM_L2, o.NORM_L2, 1)):
        B.uq_agree_scale(lay, g, norm, W, status, ws)
        assert ulp_distance(W.cpu().numpy(), o.agree_scale(g_np, seg, onorm)).max() <= ulps
    assert int(status.item()) == 0


# norms of small gradients in segments: tiles of 8192 coordinates through shared memory; empty segments, segments of
# one coordinate, more than 32 pieces in a warp's chunk, boundaries around a chunk's end, a ragged last tile, tiles
# without a boundary; and both sides of the line at 512 tiles
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M,d,cuts", [
    (3, 20_003, [*range(1, 81), 255, 256, 256, 256, 257, 511, 513, 1024, 5000, 5003, 20_000, 20_002]),
    (1, 128, [128]), (2, 257, [256]), (7, 4_096, [8, 8, 4_095]),
    (4, 256 * 4096, [3, 700_001]), (4, 256 * 4096 + 1, [3, 700_001]),
])
def test_norms_of_small_gradients_in_segments(dtype, M, d, cuts):
    seg = np.array([0, *cuts, d], dtype=np.int64)
    stride = (d + 31) // 32 * 32
    g = torch.randn(M, stride, device="cuda", generator=torch.Generator("cuda").manual_seed(d)).to(dtype)
    lay = B.Layout(M, d, stride, dtype, torch.from_numpy(seg).cuda())
    W, status = torch.empty(len(seg) - 1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.full((lay.workspace_bytes(),), 0xFF, dtype=torch.uint8, device="cuda")
    g_np = (g if dtype == torch.float32 else g.view(torch.uint16)).cpu().numpy()[:, :d]
    for norm, onorm, ulps in ((B.UQ_NORM_LINF, o.NORM_LINF, 0), (B.UQ_NORM_L2, o.NORM_L2, 1)):
        B.uq_agree_scale(lay, g, norm, W, status, ws)
        assert ulp_distance(W.cpu().numpy(), o.agree_scale(g_np, seg, onorm)).max() <= ulps
    assert int(status.item()) == 0


# a worker's squares are added in an order that does not depend on how many other workers the buffer holds.  One tile's
# squares sum to (2^24 + 1)^2, whose root lies half way between two binary32 values (the even one is 2^24); the
# other squares are 2^-6, a quarter of the last place of that sum: added to it one by one, as lane 0 of the tiles 0, 32,
# 64, .. does, they vanish, and added among themselves first they would tip the root to 2^24 + 2
@pytest.mark.parametrize("M", [1, 2, 3, 8, 16, 17])
def test_order_of_a_sum_does_not_depend_on_the_number_of_workers(M):
    d = 32 * 32 * 8192 + 7
    stride = (d + 31) // 32 * 32
    g = torch.zeros(M, stride, dtype=torch.bfloat16, device="cuda")
    g[:-1] = 0.5
    g[-1, :4] = torch.tensor([2.0 ** 24, 2.0 ** 12, 2.0 ** 12, 1.0])
    g[-1, 32 * 8192:: 32 * 8192] = 0.125
    W, status = torch.empty(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    lay = B.Layout(M, d, stride, torch.bfloat16)
    ws = torch.empty(lay.workspace_bytes(), dtype=torch.uint8, device="cuda")
    B.uq_agree_scale(lay, g, B.UQ_NORM_L2, W, status, ws)
    assert float(W.item()) == 2.0 ** 24 and int(status.item()) == 0


# the same in segments, where the kernel that takes the tiles depends on how many of them there are.  Here every fourth
# tile holds one of the small squares and each lane of the second kernel adds up two tiles, so the lanes' sums
# tip the root: by three units of the last place of the sum, to 2^24 + 2
@pytest.mark.parametrize("M", [1, 8, 9, 64])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_order_of_a_sum_in_segments_does_not_depend_on_the_number_of_workers(M, dtype):
    d = 64 * 8192
    g = torch.zeros(M, d, dtype=dtype, device="cuda")
    g[:-1] = 0.5
    g[-1, :4] = torch.tensor([2.0 ** 24, 2.0 ** 12, 2.0 ** 12, 1.0])
    g[-1, 4 * 8192:: 4 * 8192] = 0.125
    W, status = torch.empty(2, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    lay = B.Layout(M, d, d, dtype, torch.tensor([0, d - 1, d], device="cuda"))
    ws = torch.empty(lay.workspace_bytes(), dtype=torch.uint8, device="cuda")
    B.uq_agree_scale(lay, g, B.UQ_NORM_L2, W, status, ws)
    assert float(W[0].item()) == 2.0 ** 24 + 2 and int(status.item()) == 0


# shared index: 16-, 8- and 4-byte accesses by alignment and length, each number of rows that is unrolled, and more
@pytest.mark.parametrize("offset", [0, 4, 8])
@pytest.mark.parametrize("nbytes", [4, 8, 12, 16, 4096 + 4, 65536 + 16])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 9])
def test_index_min_access_widths(offset, nbytes, R):
    rng = np.random.default_rng(nbytes + R)
    raw = rng.integers(0, 4, size=(R, nbytes * 4), dtype=np.uint8)
    flat = torch.zeros(offset + R * (nbytes + 2 * offset), dtype=torch.uint8, device="cuda")     # row pitch as aligned as the base
    rows = flat[offset:].view(R, nbytes + 2 * offset)
    rows[:, :nbytes] = torch.from_numpy(np.stack([o.pack_index(r, 2) for r in raw])).cuda()
    idx = torch.full((nbytes + 32,), 0xEE, dtype=torch.uint8, device="cuda")
    B.uq_index_min(rows, 2, idx[offset: offset + nbytes], nbytes=nbytes)
    got = idx.cpu().numpy()
    assert np.array_equal(got[offset: offset + nbytes], o.pack_index(o.index_min(raw), 2))
    assert (got[:offset] == 0xEE).all() and (got[offset + nbytes:] == 0xEE).all()


# 8 bf16 workers, selecting: a row's bytes are on their way to shared memory before its scale is known; scales that the
# fast arithmetic cannot take, in the first half of the layers, over more CTAs than the GPU holds at a time
@pytest.mark.parametrize("rng_bits,power", [(16, 110), (32, -98)])
def test_staged_rows_whose_scales_the_fast_forms_cannot_take(rng_bits, power):
    w = wl.scaled("c3", 2_600_003, M=8, dtype=wl.BF16, rng_bits=rng_bits)
    g = wl.generate(w)
    half = wl.segment_offsets(w)[len(wl.segment_offsets(w)) // 2]
    g[:, :half] = wl.f32_to_bf16_bits(wl.bf16_bits_to_f32(g[:, :half]) * np.float32(2.0 ** power))
    check_parity(w, g)


# the levels alone: the workers are dealt out in groups of eight over the grid
@pytest.mark.parametrize("M", [7, 8, 9, 17])
@pytest.mark.parametrize("fmt,s", [("i8", 127), ("i6p", 31), ("i4x2", 7), ("i2x4", 1)])
def test_levels_alone_of_many_workers(M, fmt, s):
    w = wl.scaled("c2", 70_001, M=M, fmt=fmt, s=s, scales=(s,))
    check_parity(w, wl.generate(w))


# the encoder's ways through the workers: straight-line ones by number and element type, and groups of four, two and one
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 6, 7, 9, 15, 16])
@pytest.mark.parametrize("dtype", [wl.F32, wl.BF16])
@pytest.mark.parametrize("rng_bits", [16, 32])
@pytest.mark.parametrize("name,fmt,s", [("c2", "i8", 127), ("c3", "i8", 127), ("c3", "i4x2", 7), ("c3", "i6p", 31)])
def test_encoder_at_every_number_of_workers(name, fmt, s, rng_bits, dtype, M):
    scales = (s, 8 * s, 64 * s) if name == "c3" else (s,)
    w = wl.scaled(name, 9_001, M=M, dtype=dtype, fmt=fmt, s=s, scales=scales, rng_bits=rng_bits)
    check_parity(w, wl.generate(w))


# update of parameters: with 2- and 4-bit levels a thread requests its parameters before the sums; coordinates
# around one thread's 32 and one CTA's share, and none at all in the last vector
@pytest.mark.parametrize("d", [1, 31, 32, 33, 8191, 8193])
@pytest.mark.parametrize("fmt,s", [("i2x4", 1), ("i4x2", 7), ("i6p", 31), ("i8", 127)])
def test_update_at_the_edges_of_its_vectors(d, fmt, s):
    w = wl.scaled("c1", d, M=8, fmt=fmt, s=s, scales=(s,))
    g_np = wl.generate(w)
    r = _check_parity(w, g_np, None, "separate")
    q = r["q"]
    theta = torch.ones(d + 16, device="cuda")
    mom = torch.full((d + 16,), 0.5, device="cuda")
    B.uq_decode_update(q.layout, q.lev, q.fmt, q.W, q.s, q.scales, None, 0, theta[8: 8 + d], mom[8: 8 + d], 0.1, 0.9, 5e-4, None)
    want, want_m = o.sgd_update(r["ref"]["out"], np.ones(d, np.float32), np.full(d, 0.5, np.float32), lr=0.1, mu=0.9, wd=5e-4)
    assert np.array_equal(theta.cpu().numpy()[8: 8 + d], want) and np.array_equal(mom.cpu().numpy()[8: 8 + d], want_m)
    assert (theta[:8] == 1).all() and (theta[8 + d:] == 1).all() and (mom[8 + d:] == 0.5).all()


# 2 binary32 workers, one scale, 32-bit draws: another kernel from 12 000 001 coordinates on
@pytest.mark.parametrize("d", [12_000_000, 12_000_001])
def test_two_workers_on_both_sides_of_the_line(d):
    from paper_2109_12497_b200.pipeline import Quantizer
    q = Quantizer(2, d, torch.float32, [0, 1, 4_000_003, d - 300, d], keep_sums=True)
    g = torch.randn((2, q.stride), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    out = q.step(g, 7).cpu()
    n, lev, S = -(-d // 8) * 8, q.lev.cpu(), q.S.cpu()
    for t in (q.lev, q.out, q.S):
        t.fill_(77)
    q.encode(g, 7)                                                       # stage by stage: levels alone, then the sum
    q.aggregate_decode()
    assert q.status_bits() == 0 and torch.equal(lev[:, :n], q.lev.cpu()[:, :n])
    assert torch.equal(S, q.S.cpu()) and torch.equal(out, q.out.cpu())


# rows of 256 coordinates: the row that d ends in runs as the others do (binary32 steps of 2, 4 and 8 workers), whatever its
# padding holds, and a row's boundaries are counted by its lanes (up to 31) or looked up (32 and more; any number of
# them with 5 binary32 workers and no selection)
@pytest.mark.parametrize("d", [1, 7, 255, 257, 2047, 2048, 4001, 4345, 6009])
@pytest.mark.parametrize("dtype,fmt,s,N,idx_bits,rng_bits", [
    (torch.float32, "i8", 127, 1, 0, 32), (torch.float32, "i4x2", 7, 1, 0, 16), (torch.bfloat16, "i8", 127, 8, 4, 16),
    (torch.float32, "i6p", 31, 2, 1, 32), (torch.bfloat16, "i2x4", 1, 4, 2, 32), (torch.float32, "i8", 127, 3, 8, 32),
    (torch.float32, "i2x4", 1, 1, 0, 32), (torch.float32, "i2x4", 1, 4, 2, 16), (torch.float32, "i4x2", 7, 8, 4, 32),
])
@pytest.mark.parametrize("segments", [False, True])
@pytest.mark.parametrize("M", [2, 4, 5, 8])
def test_rows_that_end_early_or_hold_boundaries(M, d, dtype, fmt, s, N, idx_bits, rng_bits, segments):
    from paper_2109_12497_b200.pipeline import Quantizer
    cuts = [*range(3, 520, 7), 520, 520, 1024, 1500, 2000, 2001, 2009, d - 5, d - 1] if segments else []
    seg = [0, *sorted(min(max(c, 0), d) for c in cuts), d]
    scales = [s * 8 ** k for k in range(N)] if N > 1 else None
    q = Quantizer(M, d, dtype, seg, s=s, scales=scales, idx_bits=idx_bits, rng_bits=rng_bits, keep_sums=True, one_kernel=False,
                  fmt={"i8": B.UQ_FMT_I8, "i4x2": B.UQ_FMT_I4X2, "i2x4": B.UQ_FMT_I2X4, "i6p": B.UQ_FMT_I6P}[fmt])
    gen = torch.Generator("cuda").manual_seed(d)
    g = (torch.randn(M, q.stride, device="cuda", generator=gen) * torch.rand(q.stride, device="cuda", generator=gen) ** 6).to(dtype)
    g[:, d:] = torch.tensor([np.nan, np.inf, -np.inf, 3e38] * 8, device="cuda")[: q.stride - d].to(dtype)
    q.lev.fill_(0x55)
    if q.multi:
        q.idx.fill_(0x55)
    out = q.step(g, 11).cpu().numpy()
    W, lev = q.W.cpu().numpy(), q.lev.cpu().numpy().view(np.uint8)
    assert q.status_bits() == 0
    g_np = g[:, :d].float().cpu().numpy()
    table = None if q.layout.nseg == 1 else np.array(seg, dtype=np.int64)
    assert ulp_distance(W, o.agree_scale(g_np, table, o.NORM_L2)).max() <= 1
    if N > 1:
        idx = o.select_scale_multi(g_np, W, scales, seg_off=table)
        want = o.encode_multi(g_np, W, scales, idx, 11, rng_bits, seg_off=table)
        packed = o.pack_index(np.pad(idx, (0, -d % 8)), idx_bits)       # the last unit's padding: index 0
        assert np.array_equal(q.idx.cpu().numpy()[: len(packed)], packed)
        ref = o.decode(o.aggregate(want), M, W, scales=scales, idx=idx, seg_off=table)
    else:
        want = o.encode_single(g_np, W, s, 11, rng_bits, seg_off=table)
        ref = o.decode(o.aggregate(want), M, W, s=s, seg_off=table)
    unit = np.pad(want, ((0, 0), (0, -d % 8)))                          # the last unit's padding: level 0
    bits = {"i8": lambda x: np.ascontiguousarray(x).view(np.uint8), "i4x2": o.pack_levels_i4, "i2x4": o.pack_levels_i2,
            "i6p": lambda x: o.pack_levels_i6p(x, q.stride)}[fmt](unit)
    n = unit.shape[1]
    parts = [(0, n // 2), (q.stride // 2, n // 4)] if fmt == "i6p" else [(0, bits.shape[1])]
    for a, k in parts:
        assert np.array_equal(lev[:, a: a + k], bits[:, a: a + k])
    assert np.array_equal(q.S.cpu().numpy()[:d], o.aggregate(want)) and np.array_equal(out, ref)
