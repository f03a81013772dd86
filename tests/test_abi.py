"""The C-ABI library loads without a GPU, exports everything include/uq.h declares, and its
host-side argument validation rejects bad calls before any launch."""
import ctypes as C
import re
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

import pytest

from paper_2109_12497_b200 import binding as B
from paper_2109_12497_b200 import build as uq_build
from paper_2109_12497_b200 import pipeline

ROOT = Path(__file__).resolve().parent.parent


@pytest.fixture(scope="module")
def lib():
    uq_build.build()
    return B.lib()


def declared_functions():
    text = (ROOT / "include" / "uq.h").read_text()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(uq_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert set(names) == set(B.EXPORTS)
    for n in names:
        assert getattr(lib, n) is not None


def test_constants_match_the_header():
    text = (ROOT / "include" / "uq.h").read_text()
    for name in ("UQ_OK", "UQ_ERR_BAD_ARG", "UQ_ERR_CUDA", "UQ_ERR_UNSUPPORTED", "UQ_ERR_WORKSPACE",
                 "UQ_F32", "UQ_BF16", "UQ_NORM_LINF", "UQ_NORM_L2", "UQ_FMT_I8", "UQ_FMT_I4X2", "UQ_FMT_I2X4", "UQ_FMT_I6P",
                 "UQ_SRC_LEVELS", "UQ_SRC_SUMS", "UQ_STATUS_NONFINITE", "UQ_STATUS_BAD_SEGMENTS",
                 "UQ_STATUS_SCALE_OVERFLOW", "UQ_STATUS_BAD_INDEX", "UQ_STATUS_TIMEOUT"):
        m = re.search(rf"\b{name}\s*=\s*(\d+)", text)
        assert m and int(m.group(1)) == getattr(B, name), name


def _layout(**kw):
    base = dict(d=1000, worker_stride=1024, seg_off=None, M=2, nseg=1, dtype=B.UQ_F32, worker0=0, coord0=0)
    base.update(kw)
    return B.uq_layout(**base)


def test_sizes(lib):
    L = _layout()
    assert lib.uq_workspace_bytes(C.byref(L)) == 2 * (1 + 1) * 8
    assert lib.uq_index_bytes(C.byref(L), 2) == 256 and lib.uq_index_bytes(C.byref(L), 4) == 512
    assert lib.uq_index_bytes(C.byref(L), 3) == 0
    assert lib.uq_workspace_bytes(C.byref(_layout(worker_stride=1000))) == 0      # not a multiple of 32
    assert lib.uq_version() >= 100
    assert lib.uq_error_string(B.UQ_ERR_BAD_ARG) == b"bad argument"


def test_scratch_of_the_norms_grows_with_the_layout(lib):
    """M * (ceil(d / 8192) + nseg) doubles for every layout: scratch sized for the largest gradient does for all."""
    for M, nseg in ((1, 1), (8, 1), (8, 161), (64, 161), (3, 5000)):
        for d in (1, 8191, 8193, 10304, 100_003, 262_145, 524_288, 524_289, 600_000, 2_000_000, 25_557_032):
            L = _layout(d=d, worker_stride=-(-d // 32) * 32, M=M, nseg=nseg, seg_off=0x10000 if nseg > 1 else None)
            assert lib.uq_workspace_bytes(C.byref(L)) == M * (-(-d // 8192) + nseg) * 8


def test_kernels_behind_the_norms(lib):
    """One kernel, or one per stage for many workers of a small gradient (the count that Quantizer.kernels_per_step reports)."""
    def n(M, d, select, reconstruct, nseg=1):
        return lib.uq_encode_launches(C.byref(_layout(M=M, d=d, worker_stride=-(-d // 32) * 32, nseg=nseg, seg_off=0x10000)), select,
                                      reconstruct)
    assert [n(8, 25_557_032, s, r) for s in (0, 1) for r in (0, 1)] == [1, 1, 1, 1]
    assert [n(64, 50_001, s, r) for s in (0, 1) for r in (0, 1)] == [1, 2, 2, 3]
    assert [n(20, d, 1, 1) for d in (50_001, 239_999, 240_001)] == [3, 3, 1] and n(19, 50_001, 1, 1) == 1
    assert [n(25, d, 1, 1, 7) for d in (50_001, 124_999, 125_001)] == [3, 3, 1] and n(24, 50_001, 1, 1, 7) == 1
    assert [n(32, 256 * k, 1, 1) for k in (93, 94)] == [3, 1] and n(28, 256, 1, 1) == 1
    assert [n(8, d, 1, 0) for d in (239_999, 240_001)] == [2, 1] and n(7, 9_001, 1, 0) == 1
    assert [n(M, 9_001, 1, 0, 7) for M in (15, 16)] == [1, 2]
    assert [n(25, 256 * k, 1, 0) for k in (351, 352)] == [2, 1] and n(8, 0, 1, 1) == 0 and n(65, 100, 0, 1) == 0
    q = pipeline.Quantizer(25, 1000, device="cpu", scales=[127, 1016], idx_bits=2)
    assert [q.kernels_per_step(), pipeline.Quantizer(64, 1001, device="cpu").kernels_per_step(),
            pipeline.Quantizer(8, 1001, device="cpu", one_kernel=False).kernels_per_step()] == [5, 4, 3]


def test_bad_arguments_are_rejected_on_the_host(lib):
    """None of these reaches a launch, so they run without a GPU (pointers are fake but aligned)."""
    p = 0x10000
    ok = _layout()
    bad_layouts = [_layout(M=0), _layout(M=65), _layout(d=-1), _layout(worker_stride=992), _layout(nseg=2),
                   _layout(dtype=5), _layout(worker0=-1), _layout(nseg=0), _layout(coord0=4), _layout(coord0=-8)]
    for L in bad_layouts:
        assert lib.uq_agree_scale(C.byref(L), p, B.UQ_NORM_L2, p, None, p, 1 << 20, None) == B.UQ_ERR_BAD_ARG
        assert lib.uq_encode_single(C.byref(L), p, p, 127, 0, 32, B.UQ_FMT_I8, p, None, None) == B.UQ_ERR_BAD_ARG
    r = C.byref(ok)
    assert lib.uq_agree_scale(r, p, 1, p, None, p, 1 << 20, None) == B.UQ_ERR_BAD_ARG            # norm
    assert lib.uq_agree_scale(r, p, B.UQ_NORM_L2, p, None, p, 8, None) == B.UQ_ERR_WORKSPACE      # too small
    assert lib.uq_agree_scale(r, p, B.UQ_NORM_L2, p, None, None, 1 << 20, None) == B.UQ_ERR_WORKSPACE
    assert lib.uq_agree_scale(r, p + 4, B.UQ_NORM_L2, p, None, p, 1 << 20, None) == B.UQ_ERR_BAD_ARG  # alignment
    for s, fmt in ((0, B.UQ_FMT_I8), (128, B.UQ_FMT_I8), (8, B.UQ_FMT_I4X2), (2, B.UQ_FMT_I2X4), (32, B.UQ_FMT_I6P), (5, 4)):
        assert lib.uq_encode_single(r, p, p, s, 0, 32, fmt, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_encode_single(r, p, p, 127, 0, 24, B.UQ_FMT_I8, p, None, None) == B.UQ_ERR_BAD_ARG  # rng_bits
    assert lib.uq_encode_single(r, p, None, 127, 0, 32, B.UQ_FMT_I8, p, None, None) == B.UQ_ERR_BAD_ARG

    def scales(*v):
        return (C.c_int32 * len(v))(*v)
    for sc, n, bits in ((scales(127, 127), 2, 2), (scales(127, 64), 2, 2), (scales(0, 5), 2, 2),
                        (scales(1, 2, 3, 4, 5), 5, 2), (scales(127, 1016), 2, 3), (scales(127), 0, 2)):
        assert lib.uq_select_scale_multi(r, p, p, sc, n, bits, p, None, None) == B.UQ_ERR_BAD_ARG
        assert lib.uq_encode_multi(r, p, p, sc, n, p, bits, 0, 32, B.UQ_FMT_I8, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_encode_multi(r, p, p, scales(200, 400), 2, p, 2, 0, 32, B.UQ_FMT_I8, p, None, None) \
        == B.UQ_ERR_BAD_ARG                                                                        # s_hat > 127
    assert lib.uq_aggregate(r, p, 7, p, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode(r, p, 2, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode(r, p, B.UQ_SRC_LEVELS, B.UQ_FMT_I8, p, 0, None, 0, None, 0, p, None, None) \
        == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode(r, p, B.UQ_SRC_LEVELS, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p + 4, None, None) \
        == B.UQ_ERR_BAD_ARG


def test_later_entry_points_reject_bad_arguments_on_the_host(lib):
    """The entry points added after the six of the hot path: same rule, nothing is launched."""
    p = 0x10000
    F = C.c_float
    ok, bad = C.byref(_layout()), C.byref(_layout(M=0))
    sc = (C.c_int32 * 2)(127, 1016)
    rows = (C.c_void_p * 2)(p, p)
    assert lib.uq_step(bad, p, B.UQ_NORM_L2, 127, None, 0, 0, 0, 16, B.UQ_FMT_I8, p, None, p, p, None, None, p, 1 << 20,
                       None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_step(ok, p, B.UQ_NORM_L2, 127, None, 0, 0, 0, 16, B.UQ_FMT_I8, p, None, p, p, None, None, p, 8,
                       None) == B.UQ_ERR_WORKSPACE
    small_bytes = lib.uq_workspace_bytes_small()
    assert small_bytes >= 64 + 148 * 8 * 8 * 8
    def small(L, s=127, scales=None, N=0, bits=0, fmt=B.UQ_FMT_I8, out=p, idx=None, ws=small_bytes, status=p):
        return lib.uq_step_small(L, p, B.UQ_NORM_L2, s, scales, N, bits, 0, 16, fmt, p, idx, p, out, None, status, p, ws, None)
    assert small(bad) == B.UQ_ERR_BAD_ARG
    assert small(ok, status=None) == B.UQ_ERR_BAD_ARG                                      # a timeout must be reportable
    assert small(ok, s=128) == B.UQ_ERR_BAD_ARG
    assert small(ok, out=p + 16) == B.UQ_ERR_BAD_ARG                                      # out: 32-byte aligned
    assert small(ok, scales=sc, N=2, bits=3, idx=p) == B.UQ_ERR_BAD_ARG                     # idx_bits
    assert small(ok, scales=sc, N=2, bits=2, idx=None) == B.UQ_ERR_BAD_ARG                  # multi-scale needs idx
    assert small(C.byref(_layout(M=9))) == B.UQ_ERR_UNSUPPORTED
    assert small(ok, s=31, fmt=B.UQ_FMT_I6P) == B.UQ_ERR_UNSUPPORTED
    assert small(ok, ws=64) == B.UQ_ERR_WORKSPACE
    assert small(ok, scales=sc, N=2, bits=2, idx=p, ws=64) == B.UQ_ERR_WORKSPACE
    assert lib.uq_select_encode_multi(ok, p, p, sc, 2, 3, 0, 16, B.UQ_FMT_I8, p, p, None, None) == B.UQ_ERR_BAD_ARG   # idx_bits
    assert lib.uq_select_encode_multi(ok, p, p, sc, 2, 2, 0, 16, B.UQ_FMT_I4X2, p, p, None, None) == B.UQ_ERR_BAD_ARG  # s_hat > 7
    assert lib.uq_select_encode_multi(ok, p, p, sc, 2, 2, 0, 16, B.UQ_FMT_I8, None, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_select_encode_decode_multi(ok, p, p, sc, 2, 3, 0, 16, B.UQ_FMT_I8, p, p, p, None, None) == B.UQ_ERR_BAD_ARG   # idx_bits
    assert lib.uq_select_encode_decode_multi(ok, p, p, sc, 2, 2, 0, 16, B.UQ_FMT_I8, p, p, None, None, None) == B.UQ_ERR_BAD_ARG  # out
    assert lib.uq_select_encode_decode_multi(ok, p, p, sc, 2, 2, 0, 16, B.UQ_FMT_I8, p, p, p + 16, None, None) == B.UQ_ERR_BAD_ARG  # out alignment
    # uq_encode_decode: the checks of the encoders and of uq_decode
    assert lib.uq_encode_decode(ok, p, p, 127, None, 0, None, 0, 0, 24, B.UQ_FMT_I8, p, p, None, None) == B.UQ_ERR_BAD_ARG   # rng_bits
    assert lib.uq_encode_decode(ok, p, p, 128, None, 0, None, 0, 0, 16, B.UQ_FMT_I8, p, p, None, None) == B.UQ_ERR_BAD_ARG   # s > 127
    assert lib.uq_encode_decode(ok, p, p, 127, None, 0, None, 0, 0, 16, B.UQ_FMT_I8, p, None, None, None) == B.UQ_ERR_BAD_ARG  # out
    assert lib.uq_encode_decode(ok, p, p, 127, sc, 2, None, 2, 0, 16, B.UQ_FMT_I8, p, p, None, None) == B.UQ_ERR_BAD_ARG     # idx
    assert lib.uq_encode_decode(ok, p, p, 127, sc, 2, p, 3, 0, 16, B.UQ_FMT_I8, p, p, None, None) == B.UQ_ERR_BAD_ARG        # idx_bits
    assert lib.uq_index_min(p, 0, 64, 64, 2, p, None) == B.UQ_ERR_BAD_ARG                    # R
    assert lib.uq_index_min(p, 2, 64, 62, 2, p, None) == B.UQ_ERR_BAD_ARG                    # whole words
    assert lib.uq_index_min(p, 2, 32, 64, 2, p, None) == B.UQ_ERR_BAD_ARG                    # rows overlap
    assert lib.uq_index_min(p, 2, 64, 64, 3, p, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode_rows(ok, None, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode_rows(ok, rows, 9, p, 127, None, 0, None, 0, p, None, None) == B.UQ_ERR_BAD_ARG
    rows[1] = p + 1
    assert lib.uq_decode_rows(ok, rows, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode_update(ok, p, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p, None, F(float("nan")), F(0), F(0), None,
                                None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_decode_update(ok, p, B.UQ_FMT_I8, p, 127, None, 0, None, 0, p + 4, None, F(0.1), F(0), F(0), None,
                                None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_randk_gather(ok, p, 1001, 0, p, p, 1024, None, None) == B.UQ_ERR_BAD_ARG     # K > d
    assert lib.uq_randk_gather(ok, p, 10, 0, p, p, 40, None, None) == B.UQ_ERR_BAD_ARG         # stride % 32
    assert lib.uq_randk_gather(ok, p, 10, 0, p, p, 0, None, None) == B.UQ_ERR_BAD_ARG          # stride < K
    assert lib.uq_randk_scatter(100, 101, p, p, p, None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_randk_update(100, 10, p, None, p, F(0.1), None, None) == B.UQ_ERR_BAD_ARG
    assert lib.uq_randk_update(100, 10, p, p, p, F(float("nan")), None, None) == B.UQ_ERR_BAD_ARG


def test_step_plan_is_checked_on_the_host(lib):
    """uq_step_run makes the call that its plan describes: the same argument checks, nothing launched."""
    p = 0x10000
    def plan(**kw):
        f = dict(layout=_layout(), norm=B.UQ_NORM_L2, s=127, rng_bits=16, fmt=B.UQ_FMT_I8, W=p, lev=p, out=p, status=p, workspace=p,
                 workspace_bytes=1 << 20)
        f.update(kw)
        return B.uq_step_plan(**f)
    run = lambda q: lib.uq_step_run(C.addressof(q), p, 0, None)
    assert lib.uq_step_run(None, p, 0, None) == B.UQ_ERR_BAD_ARG
    assert run(plan(N=17)) == B.UQ_ERR_BAD_ARG and run(plan(N=-1)) == B.UQ_ERR_BAD_ARG
    assert run(plan(layout=_layout(M=0))) == B.UQ_ERR_BAD_ARG
    assert run(plan(workspace_bytes=8)) == B.UQ_ERR_WORKSPACE
    assert run(plan(one_kernel=1, s=128)) == B.UQ_ERR_BAD_ARG
    assert run(plan(one_kernel=1, workspace_bytes=64)) == B.UQ_ERR_WORKSPACE
    assert run(plan(one_kernel=1, layout=_layout(M=9))) == B.UQ_ERR_UNSUPPORTED
    multi = plan(one_kernel=1, N=2, idx_bits=3, idx=p)                                       # idx_bits
    multi.scales[:2] = [127, 1016]
    assert run(multi) == B.UQ_ERR_BAD_ARG


def test_launches_overlap_only_where_the_kernels_wait():
    """-DUQ_NO_PDL: no launch asks for the overlap with the kernel in front, since no kernel waits for it then."""
    def preprocessed(src, *flags):
        cmd = [uq_build._nvcc(), "-E", "-std=c++17", *flags, "-I", str(uq_build.INCLUDE), "-I", str(uq_build.CSRC),
               str(uq_build.CSRC / src)]
        text = subprocess.run(cmd, capture_output=True, text=True, check=True).stdout
        return re.search(r"programmaticStreamSerializationAllowed\s*=", text), re.search(r'griddepcontrol\.wait;" :::', text)   # (CUDA's own headers spell it without blanks)
    with ThreadPoolExecutor() as pool:
        for asks, waits in pool.map(lambda s: preprocessed(s, "-DUQ_NO_PDL"), uq_build.SOURCES):
            assert not asks and not waits
    asks, waits = preprocessed("uq_small_f32.cu")
    assert asks and waits


def test_binding_fails_loudly_without_the_library(monkeypatch, tmp_path):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", tmp_path / "missing.so")
    with pytest.raises(RuntimeError, match="no CPU fallback"):
        B.lib()


def test_the_package_imports_with_a_torch_built_without_cuda():
    """The layouts, the workloads and the exchange logic are of use without a GPU."""
    code = ("import torch\n"
            "for name in ('_cuda_getDevice', '_cuda_getCurrentRawStream'):\n"
            "    delattr(torch._C, name)\n"
            "from paper_2109_12497_b200 import binding, distributed, pipeline, workloads\n"
            "assert binding.Layout(2, 100, 128, torch.float32).nseg == 1\n")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)


def test_a_tensor_on_another_device_is_refused_before_any_launch():
    """The calls launch on the current device's current stream; the binding refuses, on the host,
    a tensor that lives elsewhere (checked here on the rule itself: no GPU, no launch)."""
    B.require_current_device(0, 0)
    B.require_current_device(3, 3, "g")
    for index, current in ((1, 0), (0, 1), (None, 0)):
        with pytest.raises(ValueError, match="current device"):
            B.require_current_device(index, current, "g")
