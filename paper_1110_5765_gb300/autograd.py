"""Differentiation form: the companded-and-packed product behind
``torch.autograd.Function``.

forward:   C  = op(A) op(B)              through tdgemm (steps a-d)
backward:  dA = dC op(B)^T,  dB = op(A)^T dC
           through the same companded/packed kernels, with the transposes
           expressed as the trans flags of the C ABI (no copies).
The quantizer is straight-through: its derivative is taken as the identity,
so the backward products see the incoming gradient and the saved (unquantized)
inputs; each backward product is companded and packed on its own, with
companders and packing chosen from its own block statistics (Sec. 5, Sec. 6).
Inside CUDA-graph capture the two adjoints of one product run on two streams.

Plans (device workspace) are cached per device, shape, layout and options.  A
plan's calls must not overlap on the device, so each waits for the plan's last
stream where that is another one, and two adjoints that share a plan stay on one
stream.
"""
from __future__ import annotations

import threading

import torch

from .api import Plan

_plans: dict = {}


def _op_layout(X: torch.Tensor):
    """(trans, ld, stored tensor) such that op(stored) == X without copying."""
    r, c = X.shape
    s0, s1 = X.stride()
    if s1 == 1 and s0 >= c:
        return "N", s0, X
    if s0 == 1 and s1 >= r:
        return "T", s1, X.t()
    X = X.contiguous()
    return "N", c, X


_side: dict = {}


def _side_stream(device) -> "torch.cuda.Stream":
    key = torch.device(device).index
    st = _side.get(key)
    if st is None:
        st = torch.cuda.Stream(device=device)
        _side[key] = st
    return st


def _key(A, B, opts):
    """Cache key of the product A B, with the stored operands."""
    tA, lda, As = _op_layout(A)
    tB, ldb, Bs = _op_layout(B)
    return (A.shape[0], B.shape[1], A.shape[1], tA, tB, lda, ldb, A.device.index,
            tuple(sorted(opts.items()))), As, Bs


_creating = threading.Lock()


def _plan_for(key, opts) -> Plan:
    p = _plans.get(key)
    if p is None:
        with _creating:
            p = _plans.get(key)
            if p is None:
                M, N, K, tA, tB, lda, ldb = key[:7]
                p = Plan(M, N, K, transA=tA, transB=tB, lda=lda, ldb=ldb, **opts)
                # the stream that last used the plan (outside capture)
                p._lock, p._last = threading.Lock(), None
                _plans[key] = p
    return p


def clear_plan_cache():
    for p in _plans.values():
        p.close()
    _plans.clear()


def product(A: torch.Tensor, B: torch.Tensor, opts: dict) -> torch.Tensor:
    """C = A B through the library; A, B may be transposed views."""
    key, As, Bs = _key(A, B, opts)
    C = torch.empty((A.shape[0], B.shape[1]), dtype=A.dtype, device=A.device)
    p = _plan_for(key, opts)
    with p._lock:                # (ordering the streams and queueing: one step)
        st = torch.cuda.current_stream(A.device)
        last = p._last
        if last is None or last.cuda_stream != st.cuda_stream:
            # a capture may not wait for work outside it: it begins with the
            # device synchronised, and its replays are the caller's to order
            if not torch.cuda.is_current_stream_capturing():
                if last is not None:
                    st.wait_stream(last)
                p._last = st
        p.run(As, Bs, C, stream=st)
    return C


class TDGemmFn(torch.autograd.Function):
    @staticmethod
    def forward(ctx, A, B, opts):
        ctx.save_for_backward(A, B)
        ctx.opts = opts
        return product(A, B, opts)

    @staticmethod
    def backward(ctx, dC):
        A, B = ctx.saved_tensors
        dC = dC.contiguous()
        need_a, need_b = ctx.needs_input_grad[0], ctx.needs_input_grad[1]
        # two streams only inside CUDA-graph capture: replayed graphs carry no
        # host cost, while in eager mode the extra stream bookkeeping costs
        # more host time than the overlap saves on the device
        # (a square layer of two transposed views: both adjoints have one plan)
        if (not (need_a and need_b) or not torch.cuda.is_current_stream_capturing()
                or _key(dC, B.t(), ctx.opts)[0] == _key(A.t(), dC, ctx.opts)[0]):
            dA = product(dC, B.t(), ctx.opts) if need_a else None
            dB = product(A.t(), dC, ctx.opts) if need_b else None
            return dA, dB, None
        # the two adjoints are independent: dB on a side stream, so one
        # product's latency-bound steps (statistics, fp64 planner, packing)
        # overlap the other's
        cur = torch.cuda.current_stream(dC.device)
        side = _side_stream(dC.device)
        side.wait_stream(cur)
        dA = product(dC, B.t(), ctx.opts)
        with torch.cuda.stream(side):
            dB = product(A.t(), dC, ctx.opts)
        cur.wait_stream(side)
        A.record_stream(side)
        dC.record_stream(side)
        dB.record_stream(cur)
        return dA, dB, None


def tdg_matmul(A: torch.Tensor, B: torch.Tensor, **opts) -> torch.Tensor:
    """Differentiable companded-and-packed A @ B.  ``opts`` are Plan options
    (L, W, dtype, form, target_snr_db / bits, ...)."""
    if "dtype" not in opts:
        opts["dtype"] = "f64" if A.dtype == torch.float64 else "f32"
    return TDGemmFn.apply(A, B, opts)
