"""torch.autograd wrappers over the C ABI (argument marshalling only).

* ``KLDiv.apply(V, W, H)``: d_KL(V, W H) of eq. 1; the backward pass is
  ``dna_kl_backward`` (dW = (1 - Q) H^t, dH = W^t (1 - Q), dV = log(V / Z)).
* ``UnrolledDNAH.apply(V, W, H0, K, every)``: K DNA H half-steps with W held fixed by the
  solve (``dna_step_H_fixed``), returning H_K; the backward pass runs
  ``dna_step_H_adjoint_w`` in reverse, recomputing the states of each segment from
  checkpoints kept every ``every`` steps.  Gradients flow to V, H0 and, when W requires
  one, to W (through every step's Z = W H, A = W^t Q, B = (W o W)^t Qbar and the column
  sums W^t 1 + lambda).

Tensors are CUDA float32 (F32 form) or float64 (F64 form), contiguous, row-major.

Library contexts (their device workspace) are kept per thread and per (N, T, R, form,
device) and bound afresh to the call's tensors each time (``dna_bind`` prepares
everything from them), so repeated calls allocate nothing; a call that fails destroys its
context.  ``release_contexts()`` frees the calling thread's contexts.

Work is queued on the current stream and not waited for (``KLDiv``'s forward waits for its
number): a kept context carries an event after its last call, which the next call's stream
waits for, and every tensor that the queued kernels use is recorded on their stream.
Waiting at the end of each call left the GPU idle while Python prepared the next one
(N=1024 T=4096 R=64: d_KL forward and backward 590 us -> 442, two unrolled steps forward
and backward 1300 -> 925).
"""
from __future__ import annotations

import threading

import torch

from . import _lib as L

_local = threading.local()


def _pool() -> dict:
    pool = getattr(_local, "pool", None)
    if pool is None:
        pool = _local.pool = {}
    return pool


def release_contexts() -> None:
    """Destroy the library contexts this thread keeps for the autograd wrappers."""
    pool = _pool()
    for ctx, _ in pool.values():
        L.dna_destroy(ctx)
    pool.clear()


class _Ctx:
    """A pooled context bound to (V, W, H) for the duration of a ``with`` block, on the
    current stream; ``others`` are further tensors that the block's calls use."""

    def __init__(self, V, W, H, *others):
        N, T = V.shape
        R = W.shape[1]
        dtype = L.DNA_F64 if V.dtype == torch.float64 else L.DNA_F32
        self.key = (N, T, R, dtype, V.device.index)
        if torch.cuda.is_current_stream_capturing():
            # a captured call would replay on a workspace that later calls use too
            raise RuntimeError("the autograd wrappers cannot be captured in a CUDA graph")
        stream = self.stream = torch.cuda.current_stream()
        # taken out while in use (re-entrant calls get their own)
        ctx, self.event = _pool().pop(self.key, (None, None))
        kept = ctx is not None
        if not kept:
            ctx = L.dna_create(N, T, R, L.make_opts(dtype=dtype))
            self.event = torch.cuda.Event()
        self.ctx = ctx
        try:
            if kept:
                # the last call may still use the context's workspace, on whatever stream it
                # ran (an equal handle may be a new stream that took a destroyed one's place)
                stream.wait_event(self.event)
            for t in (V, W, H, *others):
                t.record_stream(stream)
            L.dna_set_stream(ctx, stream)
            L.dna_bind(ctx, V, W, H)
        except BaseException:
            L.dna_destroy(ctx)
            raise

    def __enter__(self):
        return self.ctx

    def __exit__(self, exc_type, exc, tb):
        pool = _pool()
        if exc_type is None and self.key not in pool:
            self.event.record(self.stream)
            pool[self.key] = (self.ctx, self.event)
        else:
            L.dna_destroy(self.ctx)
        return False


class KLDiv(torch.autograd.Function):
    @staticmethod
    def forward(fctx, V, W, H):
        V, W, H = V.contiguous(), W.contiguous(), H.contiguous()
        with _Ctx(V, W, H) as ctx:
            kl = L.dna_kl(ctx)
        fctx.save_for_backward(V, W, H)
        return torch.full((), kl, dtype=torch.float64, device=V.device)

    @staticmethod
    def backward(fctx, grad):
        V, W, H = fctx.saved_tensors
        need_v, need_w, need_h = fctx.needs_input_grad
        dV = torch.empty_like(V) if need_v else None
        dW = torch.empty_like(W) if need_w else None
        dH = torch.empty_like(H) if need_h else None
        with _Ctx(V, W, H) as ctx:
            L.dna_kl_backward(ctx, float(grad), dW, dH, dV)
        return dV, dW, dH


class UnrolledDNAH(torch.autograd.Function):
    @staticmethod
    def forward(fctx, V, W, H0, K: int, every: int = 5):
        V, W = V.contiguous(), W.contiguous()
        H = H0.detach().clone().contiguous()
        T = V.shape[1]
        choices = torch.empty((K, T), dtype=torch.uint8, device=V.device)
        ckpts = []
        with _Ctx(V, W, H) as ctx:
            for k in range(K):
                if k % every == 0:
                    ckpts.append(H.clone())
                L.dna_step_H_fixed(ctx, choices[k])
        fctx.K, fctx.every = K, every
        fctx.save_for_backward(V, W, choices, *ckpts)
        return H

    @staticmethod
    def backward(fctx, grad_HK):
        V, W, choices, *ckpts = fctx.saved_tensors
        K, every = fctx.K, fctx.every
        need_v, need_w = fctx.needs_input_grad[0], fctx.needs_input_grad[1]
        Hbar = grad_HK.contiguous().clone()
        Vbar = torch.zeros_like(V) if need_v else None
        Wbar = torch.zeros_like(W) if need_w else None
        Hrun = ckpts[0].clone()
        with _Ctx(V, W, Hrun, choices, *ckpts) as ctx:
            for seg in reversed(range(len(ckpts))):
                k0, k1 = seg * every, min(seg * every + every, K)
                Hrun.copy_(ckpts[seg])
                states = [ckpts[seg]]
                for _ in range(k0, k1 - 1):           # recompute this segment's states
                    L.dna_step_H_fixed(ctx, None)
                    states.append(Hrun.clone())
                for k in reversed(range(k0, k1)):
                    out = torch.empty_like(Hbar)
                    L.dna_step_H_adjoint_w(ctx, states[k - k0], choices[k], Hbar, out, Vbar,
                                           Wbar)
                    Hbar = out
        return Vbar, Wbar, Hbar, None, None
