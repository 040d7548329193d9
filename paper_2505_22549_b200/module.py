"""``DesLoc``: owns nothing but a context handle; holds references to the caller's tensors."""
from __future__ import annotations

import ctypes
from typing import Optional, Sequence

import torch

from . import binding as B

try:
    from . import _native
except ImportError as e:
    raise ImportError(f"the native part of this module is missing ({e}): build it with "
                      "`python -m paper_2505_22549_b200.build`") from e
if _native.torch_version != str(torch.__version__):
    raise ImportError(f"the native part of this module was built for torch {_native.torch_version}, this is torch "
                      f"{torch.__version__}: build it again with `python -m paper_2505_22549_b200.build`")

_entry = lambda f: ctypes.cast(f, ctypes.c_void_p).value
_native.bind(*(_entry(getattr(B.raw_lib(), "desloc_" + n))
               for n in ("step", "step_masked", "step_normclip", "step_diag", "rel_change", "get_diag_norms", "step_host")))

_GRAD_MISFIT = "gradient tensor of wrong dtype, size or layout"
_SNAP_MISFIT = "snapshot tensor of wrong dtype, size or layout"
_HOST_MISFIT = "host gradient tensor of wrong dtype, size, layout or device"


class BoundGrads:
    """Gradient tensors already checked and marshalled (see DesLoc.bind_grads)."""

    def __init__(self, array, keep):
        self.array, self._keep = array, keep
        self.address = ctypes.addressof(array)


class DesLoc:
    """M worker replicas of a tensor list, stepped by the CUDA library.

    x, u, v: lists (one per worker) of lists of CUDA fp32 tensors (one per model tensor),
    updated in place by :meth:`step`.  v is None for SGDM.
    """

    def __init__(self, x: Sequence[Sequence[torch.Tensor]], u, v, *, opt, grad_dtype,
                 beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, clip_rho=0.0,
                 K=(1, 1, 1), flags=0):
        M = len(x)
        numel = [int(t.numel()) for t in x[0]]
        dev = x[0][0].device
        if dev.type != "cuda":
            raise ValueError("DesLoc needs CUDA tensors (there is no CPU path)")
        for arrs in (x, u) + ((v,) if v is not None else ()):
            if len(arrs) != M:
                raise ValueError("x, u, v need one tensor list per worker")
            for lst in arrs:
                if [int(t.numel()) for t in lst] != numel:
                    raise ValueError("every worker needs the same tensor list")
                for t in lst:
                    if t.dtype != torch.float32 or not t.is_contiguous() or t.device != dev:
                        raise ValueError("state tensors must be contiguous fp32 on one device")
        self._keep = (x, u, v)
        self.M, self.numel, self.device = M, numel, dev
        self.grad_dtype = B.DTYPE_BY_NAME.get(grad_dtype, grad_dtype)
        self.cfg = B.make_config(M, numel, opt, grad_dtype, beta1, beta2, eps, weight_decay,
                                 clip_rho, K[0], K[1], K[2], flags)
        flat = lambda a: [t.data_ptr() for lst in a for t in lst]
        self._index = dev.index if dev.index is not None else torch.cuda.current_device()
        self.ctx: Optional[int] = B.desloc_create(
            self.cfg, flat(x), flat(u), flat(v) if v is not None else None, self._index)
        self._tables()

    def _tables(self) -> None:
        # one buffer of pointers per kind of argument, written anew at every call
        self._table = _native.Table(self.numel, self.M)
        self._table2 = _native.Table(self.numel, self.M)

    def bind_grads(self, grads: Sequence[Sequence[torch.Tensor]]):
        """Check a set of gradient tensors once and return a handle every step method accepts in
        place of the nested lists: a loop that reuses its gradient buffers then pays no
        per-step marshalling.  The handle keeps the tensors alive."""
        if isinstance(grads, BoundGrads):
            return grads
        n = self.M * len(self.numel)
        # (a table of its own: another thread may be inside a step, which reads the buffer of self._table with
        # the interpreter's lock released)
        table = _native.Table(self.numel, self.M)
        address = self._fill(table, grads, self.grad_dtype, 0, _GRAD_MISFIT)
        return BoundGrads((ctypes.c_void_p * n).from_buffer_copy((ctypes.c_void_p * n).from_address(address)), grads)

    def _grad_address(self, grads) -> int:
        """Address of the array of gradient pointers, good until the next call of this method."""
        if isinstance(grads, BoundGrads):
            return grads.address
        return self._fill(self._table, grads, self.grad_dtype, 0, _GRAD_MISFIT)

    def _fill(self, table, nested, kind: int, where: int, misfit: str) -> int:
        """Checks and marshals nested lists of tensors into the buffer of `table`; its address.  Objects that are no
        torch.Tensor but answer the same questions go one by one."""
        if not isinstance(nested, (list, tuple)):
            nested = [list(row) for row in nested]
        address = table.fill(nested, kind, where, misfit)
        if address is None:
            want = torch.bfloat16 if kind == B.DESLOC_BF16 else torch.float32
            ptrs = []
            for row in nested:
                for t, n in zip(row, self.numel):
                    if t.dtype != want or t.numel() != n or not t.is_contiguous() or (where == 1 and t.is_cuda):
                        raise ValueError(misfit)
                    ptrs.append(t.data_ptr())
            if len(ptrs) != self.M * len(self.numel):
                raise ValueError("need one gradient list per worker")
            address = table.set(ptrs)
        return address

    def _raise(self, status: int, where: str):
        raise B.DeslocError(status, where, B.desloc_last_cuda_error(self.ctx))

    def step(self, t: int, lr: float, grads, clip_bound: float = 0.0) -> int:
        """Step t on torch's current stream; returns the sync mask."""
        r = _native.step(self.ctx, t, lr, clip_bound, 0.0, self._grad_address(grads), self._index, 0)
        if r < 0:
            self._raise(r, "desloc_step")
        return r

    def step_normclip(self, t: int, lr: float, grads, max_norm: float, clip_bound: float = 0.0) -> int:
        """Step t with norm-based gradient clipping (per worker, over the whole tensor list)."""
        r = _native.step(self.ctx, t, lr, clip_bound, max_norm, self._grad_address(grads), self._index, 1)
        if r < 0:
            self._raise(r, "desloc_step_normclip")
        return r

    def step_diag(self, t: int, lr: float, grads, max_norm: float = 0.0, clip_bound: float = 0.0) -> int:
        """Step t that also accumulates the gradient, parameter and update norms (read them with
        diag_norms()); max_norm > 0 adds norm-based clipping in front."""
        r = _native.step(self.ctx, t, lr, clip_bound, max_norm, self._grad_address(grads), self._index, 2)
        if r < 0:
            self._raise(r, "desloc_step_diag")
        return r

    def diag_norms(self):
        """(per_tensor [3][M][num_tensors], total [3][M]) of the latest step_diag; kind 0 =
        gradient as read, 1 = new parameters, 2 = update d_t.  Waits for the results: what was on the current stream is done."""
        r = _native.diag_norms(self.ctx, self.M, len(self.numel), self._index)
        if isinstance(r, int):
            self._raise(r, "desloc_get_diag_norms")
        return r

    def grad_norms(self):
        """(norms, clip factors) of the latest step_normclip; synchronises the current stream."""
        stream = torch.cuda.current_stream(self.device).cuda_stream
        return B.desloc_get_grad_norms(self.ctx, self.M, stream)

    def rel_change(self, array: int, then: Sequence[Sequence[torch.Tensor]]):
        """Per-worker ||s - then|| / ||then|| against a snapshot (lists like x); waits like diag_norms()."""
        r = _native.rel_change(self.ctx, array, self._fill(self._table2, then, B.DESLOC_F32, 0, _SNAP_MISFIT),
                               self._index, self.M)
        if not isinstance(r, list):
            self._raise(r, "desloc_rel_change")
        return r

    def set_workers(self, x, u, v, first_new: int) -> None:
        """New worker set (lists like the constructor's); workers first_new.. start from the mean
        of the current workers.  Synchronises the current stream."""
        M = len(x)
        for arrs in (x, u) + ((v,) if v is not None else ()):
            if len(arrs) != M or any([int(t.numel()) for t in lst] != self.numel for lst in arrs):
                raise ValueError("every worker needs the same tensor list")
        flat = lambda a: [t.data_ptr() for lst in a for t in lst]
        stream = torch.cuda.current_stream(self.device).cuda_stream
        B.desloc_set_workers(self.ctx, M, first_new, flat(x), flat(u),
                             flat(v) if v is not None else None, stream)
        self._keep = (x, u, v)
        self.M = M
        self._tables()

    def step_host(self, t: int, lr: float, host_grads, dev_grads, clip_bound: float = 0.0) -> int:
        """Step t with gradients in (pinned) host tensors; dev_grads are device staging tensors."""
        hp = self._fill(self._table2, host_grads, self.grad_dtype, 1, _HOST_MISFIT)
        r = _native.step_host(self.ctx, t, lr, clip_bound, hp, self._grad_address(dev_grads), self._index)
        if r < 0:
            self._raise(r, "desloc_step_host")
        return r

    def step_masked(self, mask: int, lr: float, grads, clip_bound: float = 0.0) -> None:
        r = _native.step_masked(self.ctx, mask, lr, clip_bound, self._grad_address(grads), self._index)
        if r < 0:
            self._raise(r, "desloc_step_masked")

    def counters(self):
        return B.desloc_get_counters(self.ctx)

    def launches(self) -> int:
        return B.desloc_get_launch_count(self.ctx)

    def close(self) -> None:
        if self.ctx is not None:
            B.desloc_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass
