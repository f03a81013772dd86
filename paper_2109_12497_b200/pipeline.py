"""One quantize -> aggregate -> reconstruct step over M resident worker buffers.

``Quantizer`` owns the device buffers of one configuration (scales, scale indices, levels,
scratch, output) and enqueues the C-ABI calls of Algorithm 1 (single-scale) or Algorithm 2
(multi-scale) in order on the current stream.  It holds no arithmetic: each stage is one call
into the CUDA library.
"""
from __future__ import annotations

import ctypes as C
from typing import Optional, Sequence

import numpy as np
import torch

from . import binding as B


_current_device = B._current_device
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)      # (a torch built without CUDA has none)

# Gradients of all workers up to this size take the one-kernel step.  Its time over that of separate kernels at 4, 8, 12 and
# 16 MB, replayed graph, one scale: binary32 1 worker 0.83, 0.83, 1.18, 1.05, 4 workers 0.70, 0.84, 1.23, 0.95, 8 workers
# 0.77, 0.59, 0.73, 0.85; bf16 1 worker 0.92, 1.25, 1.35, 1.32, 4 workers 0.75, 0.86, 1.22, 1.30, 8 workers 0.74, 0.92, 1.20, 1.22.
ONE_KERNEL_MAX_BYTES = 8 << 20


class Quantizer:
    def __init__(self, M: int, d: int, dtype: torch.dtype = torch.float32,
                 seg_off: Optional[Sequence[int]] = None, s: int = 127,
                 scales: Optional[Sequence[int]] = None, fmt: int = B.UQ_FMT_I8, idx_bits: int = 0,
                 norm: int = B.UQ_NORM_L2, rng_bits: int = 32, keep_sums: bool = False,
                 device: str | torch.device = "cuda", fused_select: Optional[bool] = None,
                 one_kernel: Optional[bool] = None):
        B.lib()                                     # fail now if the CUDA library is not built
        dev = torch.device(device)
        if dev.type == "cuda" and dev.index is None:
            dev = torch.device("cuda", torch.cuda.current_device())
        self.device = dev
        self.M, self.d, self.dtype = M, d, dtype
        self.stride = -(-d // 32) * 32
        self.multi = scales is not None and idx_bits != 0
        # multi-scale: whether selection + sharing run inside the encoder's kernel (same bits) instead of as a
        # streaming kernel of their own.  None = the library's own choice (uq_step: inside).
        self.fused_select = None if fused_select is None else bool(fused_select) and self.multi
        self.s = int(scales[0]) if self.multi else int(s)
        self.scales = [int(x) for x in scales] if self.multi else None
        self.fmt, self.idx_bits, self.norm, self.rng_bits = fmt, idx_bits if self.multi else 0, norm, rng_bits
        seg_dev = None
        if seg_off is not None and len(seg_off) > 2:
            seg_dev = torch.as_tensor(np.asarray(seg_off, dtype=np.int64), device=dev)
        self.layout = B.Layout(M, d, self.stride, dtype, seg_dev)
        nseg = self.layout.nseg
        self.W = torch.zeros(nseg, dtype=torch.float32, device=dev)
        self.status = torch.zeros(1, dtype=torch.int32, device=dev)
        # one segment, few workers, and so small that the step is bound by its launches: the whole step as one kernel (uq_step_small).  None = decide by size.
        fits = B.small_step_supported(self.layout, fmt)
        if one_kernel and not fits:
            raise ValueError("uq: the one-kernel step takes one segment, M <= 8 and one-plane level formats")
        self.one_kernel = fits and (one_kernel if one_kernel is not None
                                    else M * d * (4 if dtype == torch.float32 else 2) <= ONE_KERNEL_MAX_BYTES)
        self.workspace = torch.empty(max(8, self.layout.workspace_bytes()), dtype=torch.uint8, device=dev)
        # The one-kernel step keeps its barrier counters in the first bytes of its scratch, wants them
        # zero before the first call and leaves them zero: a buffer of its own, never handed to
        # uq_agree_scale (whose partial sums would overwrite the counters).
        self.small_workspace = (torch.zeros(max(8, B.uq_workspace_bytes_small()), dtype=torch.uint8, device=dev)
                                if self.one_kernel else None)
        self.lev = torch.empty((M, self.layout.level_row_bytes(fmt)), dtype=torch.int8, device=dev)
        self.idx = (torch.empty(max(16, self.layout.index_bytes(self.idx_bits)), dtype=torch.uint8, device=dev)
                    if self.multi else None)
        self.out = torch.empty(max(d, 1), dtype=torch.float32, device=dev)
        self.S = torch.empty(max(d, 1), dtype=torch.int32, device=dev) if keep_sums else None
        self._plan = None                               # the step's arguments, gathered at the next step

    def __setattr__(self, name, value):
        # whatever is assigned, the next step gathers its arguments anew
        object.__setattr__(self, name, value)
        if name != "_plan":
            object.__setattr__(self, "_plan", None)

    # the four stages, each one C-ABI call -------------------------------------------------------
    def agree_scale(self, g: torch.Tensor) -> None:
        B.uq_agree_scale(self.layout, g, self.norm, self.W, self.status, self.workspace)

    def select_scale(self, g: torch.Tensor) -> None:
        B.uq_select_scale_multi(self.layout, g, self.W, self.scales, self.idx_bits, self.idx, self.status)

    def encode(self, g: torch.Tensor, seed: int) -> None:
        if self.multi:
            B.uq_encode_multi(self.layout, g, self.W, self.scales, self.idx, self.idx_bits, seed,
                              self.rng_bits, self.fmt, self.lev, self.status)
        else:
            B.uq_encode_single(self.layout, g, self.W, self.s, seed, self.rng_bits, self.fmt, self.lev,
                               self.status)

    def select_encode(self, g: torch.Tensor, seed: int) -> None:
        """Multi-scale: scale selection, scale sharing and quantization in one call."""
        B.uq_select_encode_multi(self.layout, g, self.W, self.scales, self.idx_bits, seed, self.rng_bits, self.fmt,
                                 self.idx, self.lev, self.status)

    def select_encode_decode(self, g: torch.Tensor, seed: int) -> None:
        """Multi-scale: everything behind the scale agreement in one call."""
        B.uq_select_encode_decode_multi(self.layout, g, self.W, self.scales, self.idx_bits, seed, self.rng_bits,
                                        self.fmt, self.idx, self.lev, self.out, self.status)

    def aggregate_decode(self) -> None:
        B.uq_decode(self.layout, self.lev, B.UQ_SRC_LEVELS, self.fmt, self.W, self.s, self.scales, self.idx,
                    self.idx_bits, self.out, self.S)

    def encode_decode(self, g: torch.Tensor, seed: int) -> None:
        """Quantization, integer aggregation and reconstruction as one call (what the step makes when
        the integer sums are not kept)."""
        B.uq_encode_decode(self.layout, g, self.W, self.s, self.scales, self.idx, self.idx_bits, seed, self.rng_bits,
                           self.fmt, self.lev, self.out, self.status)

    @property
    def selects_inside(self) -> bool:
        """Multi-scale: whether the step's selection runs inside the encoder's kernel."""
        if not self.multi:
            return False
        return self.fused_select is None or self.fused_select

    @property
    def fused_decode(self) -> bool:
        """Whether the step's encoder also aggregates and reconstructs."""
        return self.fused_select is None or self.S is None

    def aggregate_decode_update(self, theta: torch.Tensor, momentum: Optional[torch.Tensor], lr: float,
                                mu: float = 0.0, wd: float = 0.0) -> None:
        """Fused aggregation, reconstruction and SGD step on theta (Algorithm 1/2, last three lines)."""
        B.uq_decode_update(self.layout, self.lev, self.fmt, self.W, self.s, self.scales, self.idx, self.idx_bits,
                           theta, momentum, lr, mu, wd)

    def step(self, g: torch.Tensor, seed: int = 0) -> torch.Tensor:
        """g: [M, stride] gradients of all workers -> the reconstructed average gradient [d]."""
        if self.one_kernel or self.fused_select is None:      # the library's sequence: one trip through the binding
            # every buffer but g is this object's own: their addresses and the settings are gathered in a plan when
            # one of them has been assigned, not marshalled per step (for small gradients the host's share of a step
            # is as long as the GPU's).  The layout is copied each time: its worker0 and coord0 may be set in place.
            call, address, plan, shape, dtype, out = self._plan or self._make_plan()
            plan.layout = self.layout.c
            index = g.get_device()
            if not (g.shape == shape and g.dtype is dtype and g.is_contiguous() and index == self.device.index
                    and index == _current_device()):
                self._check_devices(g)
            rc = call(address, g.data_ptr(), seed, _raw_stream(index))
            if rc != B.UQ_OK:
                raise B.UqError("uq_step_small" if self.one_kernel else "uq_step", rc)
            return out
        # the caller's choice of where selection runs, call by call
        self.agree_scale(g)
        if self.fused_select:                                 # inside the encoder's kernel
            if self.S is None:                                # ... and aggregation + reconstruction too, where it can
                self.select_encode_decode(g, seed)
            else:
                self.select_encode(g, seed)
                self.aggregate_decode()
            return self.out[: self.d]
        if self.multi:
            self.select_scale(g)
        if self.S is None:
            self.encode_decode(g, seed)
        else:
            self.encode(g, seed)
            self.aggregate_decode()
        return self.out[: self.d]

    def _make_plan(self):
        ptr = lambda t: None if t is None else t.data_ptr()
        ws = self.small_workspace if self.one_kernel else self.workspace
        p = B.uq_step_plan(layout=self.layout.c, norm=self.norm, s=self.s, N=len(self.scales) if self.multi else 0,
                           idx_bits=self.idx_bits, rng_bits=self.rng_bits, fmt=self.fmt, one_kernel=int(self.one_kernel),
                           W=ptr(self.W), idx=ptr(self.idx), lev=ptr(self.lev), out=ptr(self.out), S_opt=ptr(self.S),
                           status=ptr(self.status), workspace=ptr(ws), workspace_bytes=ws.numel())
        if self.multi:
            kept = self.scales[: len(p.scales)]         # (the library refuses an N beyond them)
            p.scales[: len(kept)] = kept
        self._plan = (B.lib().uq_step_run, C.addressof(p), p, torch.Size((self.layout.M, self.layout.worker_stride)),
                      self.layout.dtype, self.out[: self.d])
        return self._plan

    def _check_devices(self, g: torch.Tensor) -> None:
        """The checks of the marshalling wrappers for the paths that call the library directly: the
        gradients have the layout's shape, and they, this object's buffers and the current device
        (on whose current stream the kernels are launched) are one and the same device."""
        self.layout.check_g(g)
        if not g.is_cuda:
            raise ValueError("uq: tensors must live on a CUDA device")
        current = torch.cuda.current_device()
        B.require_current_device(g.device.index, current, "g")
        B.require_current_device(self.device.index, current, "the quantizer")

    def kernels_per_step(self) -> int:
        """Kernel launches one step enqueues: norm partials + their sum, and what follows as one kernel or as one per
        stage (the library's choice by size, or the caller's)."""
        if self.one_kernel:
            return 1
        if self.d == 0:
            return 1
        n = 2 + B.lib().uq_encode_launches(self.layout.ref(), self.selects_inside, self.fused_decode)
        return n + (self.multi and not self.selects_inside) + (not self.fused_decode)

    def status_bits(self) -> int:
        """Synchronizes and returns the device status word (0 = clean)."""
        bits = int(self.status.item())
        if bits & B.UQ_STATUS_TIMEOUT and self.small_workspace is not None:   # a barrier wait ran out: its counters are not back at zero
            self.small_workspace.zero_()
        return bits


class RandKQuantizer:
    """GlobalRandKMaxNorm / GlobalRandKMaxNormMultiScale: the K coordinates of this step's shared
    choice are gathered into a compact buffer, the dense quantizer (single- or multi-scale) runs
    on it as one vector, and the K reconstructed values are scattered back."""

    def __init__(self, M: int, d: int, K: int, dtype: torch.dtype = torch.float32, **quantizer_args):
        if not 0 <= K <= d:
            raise ValueError("uq: K must lie in 0..d")
        quantizer_args.pop("seg_off", None)                  # the K-vector is one vector with one scale
        dev = torch.device(quantizer_args.get("device", "cuda"))
        self.M, self.d, self.K = M, d, K
        self.dense_layout = B.Layout(M, d, -(-d // 32) * 32, dtype, None)
        self.inner = Quantizer(M, K, dtype, **quantizer_args)
        self.sel = torch.empty(max(K, 1), dtype=torch.int64, device=dev)
        self.gk = torch.empty((M, self.inner.stride), dtype=dtype, device=dev)
        self.status = self.inner.status
        self._own = None                                     # my buffers' addresses, once a call has checked them

    def __setattr__(self, name, value):
        # whatever is assigned, the next call checks my buffers anew
        object.__setattr__(self, name, value)
        if name != "_own":
            object.__setattr__(self, "_own", None)

    def _mine(self, t: torch.Tensor, dtype: torch.dtype) -> bool:
        """Whether t is contiguous, of that type, and on this object's device, which is the current one (else
        the marshalling wrappers are called, whose checks say what is wrong)."""
        index = t.get_device()
        return t.dtype is dtype and t.is_contiguous() and index == self.inner.device.index and index == _current_device()

    def gather(self, g: torch.Tensor, seed: int) -> None:
        lay, own = self.dense_layout, self._own
        fits = g.shape == (lay.M, lay.worker_stride) and self._mine(g, lay.dtype)
        if own is None or not fits:
            B.uq_randk_gather(lay, g, self.K, seed, self.sel, self.gk, self.status)
            if fits:
                self._own = (self.sel.data_ptr(), self.gk.data_ptr(), self.gk.shape[1], B._ptr(self.status))
            return
        rc = B.lib().uq_randk_gather(lay.ref(), g.data_ptr(), self.K, seed, *own, _raw_stream(g.get_device()))
        if rc != B.UQ_OK:
            raise B.UqError("uq_randk_gather", rc)

    def quantize(self, seed: int) -> torch.Tensor:
        """Agree-scale, [select], encode, aggregate + reconstruct on the compact buffer -> [K] values."""
        return self.inner.step(self.gk, seed)

    def scatter(self, out: torch.Tensor) -> None:
        B.uq_randk_scatter(self.d, self.K, self.sel, self.inner.out, out, self.status)

    def clear(self, out: torch.Tensor) -> None:
        """Zero the entries of ``out`` that the last scatter wrote."""
        B.uq_randk_scatter(self.d, self.K, self.sel, None, out, self.status)

    def update(self, theta: torch.Tensor, lr: float) -> None:
        own, vals = self._own, self.inner.out
        if own is None or not (theta.dim() == 1 and theta.shape[0] >= self.d and self._mine(theta, torch.float32)
                               and vals.dim() == 1 and vals.shape[0] >= self.K and self._mine(vals, torch.float32)):
            B.uq_randk_update(self.d, self.K, self.sel, vals, theta, lr, self.status)
            return
        rc = B.lib().uq_randk_update(self.d, self.K, own[0], vals.data_ptr(), theta.data_ptr(), lr, own[3],
                                     _raw_stream(theta.get_device()))
        if rc != B.UQ_OK:
            raise B.UqError("uq_randk_update", rc)

    def step(self, g: torch.Tensor, out: torch.Tensor, seed: int = 0) -> torch.Tensor:
        """g: [M, stride] gradients -> out (dense [d], zero off the chosen set if it was zero before)."""
        self.gather(g, seed)
        self.quantize(seed)
        self.scatter(out)
        return out

    def kernels_per_step(self) -> int:
        return 2 + self.inner.kernels_per_step() if self.K > 0 else 1

    def status_bits(self) -> int:
        return int(self.status.item())


def from_workload(w, keep_sums: bool = False, device="cuda", fused_select: Optional[bool] = None,
                  one_kernel: Optional[bool] = None) -> Quantizer:
    """A Quantizer configured like a ``workloads.Workload``."""
    from . import workloads as wl
    seg = wl.segment_offsets(w)
    return Quantizer(
        M=w.M, d=w.d, dtype=torch.float32 if w.dtype == wl.F32 else torch.bfloat16, seg_off=seg, s=w.s,
        scales=list(w.scales) if w.quantizer == "multi" else None,
        fmt={"i8": B.UQ_FMT_I8, "i4x2": B.UQ_FMT_I4X2, "i2x4": B.UQ_FMT_I2X4, "i6p": B.UQ_FMT_I6P}[w.fmt], idx_bits=w.idx_bits,
        norm=B.UQ_NORM_L2 if w.norm == wl.NORM_L2 else B.UQ_NORM_LINF, rng_bits=w.rng_bits,
        keep_sums=keep_sums, device=device, fused_select=fused_select, one_kernel=one_kernel)


def randk_from_workload(w, K: int, device="cuda") -> RandKQuantizer:
    """A RandKQuantizer with the quantizer settings of a ``workloads.Workload`` (its segments do
    not apply: the K chosen coordinates form one vector)."""
    from . import workloads as wl
    return RandKQuantizer(
        w.M, w.d, K, torch.float32 if w.dtype == wl.F32 else torch.bfloat16, s=w.s,
        scales=list(w.scales) if w.quantizer == "multi" else None,
        fmt={"i8": B.UQ_FMT_I8, "i4x2": B.UQ_FMT_I4X2, "i2x4": B.UQ_FMT_I2X4, "i6p": B.UQ_FMT_I6P}[w.fmt], idx_bits=w.idx_bits,
        norm=B.UQ_NORM_L2 if w.norm == wl.NORM_L2 else B.UQ_NORM_LINF, rng_bits=w.rng_bits, device=device)
