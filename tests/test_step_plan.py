"""What the objects of pipeline.py hand to the library, on the host (the calls themselves are replaced by recorders): their
settings, buffers and layout as they are at that call, whatever was assigned or set in place since the last one."""
import ctypes as C
from types import SimpleNamespace

import pytest
import torch

from paper_2109_12497_b200 import binding as B
from paper_2109_12497_b200 import pipeline


class FakeGradients:
    """A tensor as far as step() looks at it, on CUDA device 0."""
    def __init__(self, q):
        self.shape, self.dtype = torch.Size((q.layout.M, q.layout.worker_stride)), q.layout.dtype

    is_contiguous = staticmethod(lambda: True)
    dim = staticmethod(lambda: 2)
    get_device = staticmethod(lambda: 0)
    data_ptr = staticmethod(lambda: 0x1000)


@pytest.fixture
def calls(monkeypatch):
    made = []

    def uq_step_run(address, g, seed, stream):
        made.append(B.uq_step_plan.from_buffer_copy(C.cast(address, C.POINTER(B.uq_step_plan)).contents))
        return B.UQ_OK
    real = B.lib()
    fake = SimpleNamespace(uq_step_run=uq_step_run, **{n: getattr(real, n) for n in (
        "uq_workspace_bytes", "uq_workspace_bytes_small", "uq_index_bytes", "uq_error_string")})
    monkeypatch.setattr(B, "lib", lambda: fake)
    monkeypatch.setattr(pipeline, "_current_device", lambda: 0)
    monkeypatch.setattr(pipeline, "_raw_stream", lambda index: 0)
    return made


def quantizer(**kw):
    q = pipeline.Quantizer(2, 1000, device="cpu", **kw)
    q.device = torch.device("cuda", 0)
    return q


def test_a_step_uses_the_settings_of_its_time(calls):
    q = quantizer(scales=[7, 56], idx_bits=2)
    g = FakeGradients(q)
    q.step(g, 0)
    assert (calls[-1].norm, calls[-1].rng_bits, calls[-1].fmt, calls[-1].one_kernel) == (B.UQ_NORM_L2, 32, B.UQ_FMT_I8, 1)
    assert calls[-1].workspace == q.small_workspace.data_ptr()
    q.norm, q.rng_bits, q.fmt, q.idx_bits, q.one_kernel = B.UQ_NORM_LINF, 16, B.UQ_FMT_I4X2, 4, False
    q.step(g, 0)
    p = calls[-1]
    assert (p.norm, p.rng_bits, p.fmt, p.idx_bits, p.one_kernel) == (B.UQ_NORM_LINF, 16, B.UQ_FMT_I4X2, 4, 0)
    assert p.workspace == q.workspace.data_ptr() and p.workspace_bytes == q.workspace.numel()
    q.scales = [7, 14, 28]
    q.step(g, 0)
    assert calls[-1].N == 3 and list(calls[-1].scales[:3]) == [7, 14, 28]
    single = quantizer()
    single.step(g, 0)
    single.s = 100
    single.step(g, 0)
    assert [p.s for p in calls[-2:]] == [127, 100]


def test_a_step_uses_the_layout_as_it_stands(calls):
    q = quantizer()
    g = FakeGradients(q)
    q.step(g, 0)
    q.layout.c.coord0, q.layout.c.worker0 = 64, 5                 # a gradient handed over piece by piece
    q.step(g, 0)
    assert (calls[-1].layout.coord0, calls[-1].layout.worker0) == (64, 5)
    q.layout = B.Layout(2, 500, 512, torch.float32)
    q.step(FakeGradients(q), 0)
    assert (calls[-1].layout.d, calls[-1].layout.worker_stride) == (500, 512)
    with pytest.raises(ValueError, match="contiguous"):
        q.step(g, 0)                                             # the shape of the layout before


def test_a_step_uses_the_buffers_as_they_are(calls):
    q = quantizer(scales=[127, 1016], idx_bits=2)
    g = FakeGradients(q)
    q.step(g, 0)
    for name in ("W", "idx", "lev", "status", "small_workspace"):
        setattr(q, name, getattr(q, name).clone())
    q.S = torch.zeros(1000, dtype=torch.int32)
    q.out = torch.zeros(1000)
    out = q.step(g, 0)
    p = calls[-1]
    assert (p.W, p.idx, p.lev, p.status, p.S_opt, p.out, p.workspace) == tuple(
        getattr(q, n).data_ptr() for n in ("W", "idx", "lev", "status", "S", "out", "small_workspace"))
    assert out.data_ptr() == q.out.data_ptr()


def test_too_many_scales_are_refused_by_the_library(monkeypatch):
    """N > 16 is the library's argument error, found on the host before anything is launched."""
    monkeypatch.setattr(pipeline, "_current_device", lambda: 0)
    monkeypatch.setattr(pipeline, "_raw_stream", lambda index: 0)
    q = quantizer(scales=[7 * 2 ** k for k in range(17)], idx_bits=8)
    with pytest.raises(B.UqError) as e:
        q.step(FakeGradients(q), 0)
    assert e.value.code == B.UQ_ERR_BAD_ARG


def test_sparse_calls_use_the_buffers_as_they_are(monkeypatch, calls):
    made = {}
    lib = B.lib()
    lib.uq_randk_gather = lambda lay, g, K, seed, sel, gk, gk_stride, status, stream: made.update(
        sel=sel, gk=gk, gk_stride=gk_stride, status=status) or B.UQ_OK
    lib.uq_randk_update = lambda d, K, sel, vals, theta, lr, status, stream: made.update(sel=sel, vals=vals, status=status) or B.UQ_OK
    monkeypatch.setattr(B, "_ptr", lambda t: None if t is None else t.data_ptr())
    monkeypatch.setattr(B, "_stream", lambda: 0)
    monkeypatch.setattr(pipeline.RandKQuantizer, "_mine", lambda self, t, dtype: t.dtype is dtype and t.is_contiguous())
    rq = pipeline.RandKQuantizer(2, 1000, 100, device="cpu")
    g = FakeGradients(SimpleNamespace(layout=rq.dense_layout))
    theta = torch.zeros(1000)
    theta.get_device = lambda: 0
    for _ in range(2):
        for _ in range(2):
            rq.gather(g, 0)
            assert (made["sel"], made["gk"], made["gk_stride"], made["status"]) == (rq.sel.data_ptr(), rq.gk.data_ptr(), 128,
                                                                                      rq.status.data_ptr())
            rq.update(theta, 0.1)
            assert (made["sel"], made["vals"], made["status"]) == (rq.sel.data_ptr(), rq.inner.out.data_ptr(), rq.status.data_ptr())
        rq.sel, rq.gk, rq.status, rq.inner.out = rq.sel.clone(), rq.gk.clone(), rq.status.clone(), rq.inner.out.clone()
    rq.gather(g, 0)
    rq.inner.out = torch.zeros(99)
    with pytest.raises(ValueError, match="vals"):
        rq.update(theta, 0.1)
    rq.sel = torch.zeros(99, dtype=torch.int64)
    with pytest.raises(ValueError, match="sel"):
        rq.gather(g, 0)
