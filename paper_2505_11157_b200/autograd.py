"""The operator as differentiable functions over the C-ABI calls, for dropping it into a PyTorch graph.

Nothing is computed here: forward calls ``sna_forward_ex`` (keeping out and lse), backward calls
``sna_backward_ex`` with a workspace tensor; for plain channels-last tensors both calls are made by native code
(csrc_torch/sna_autograd.cpp), for subclasses and under tracing by a Python function.  Tensors are [B, H, nlat, nlon, C] fp32 CUDA, channels last.
"""
from __future__ import annotations

import threading

import torch

from . import sna

try:
    from . import _sna_torch
except ImportError as e:
    raise ImportError("the native autograd function is missing or was built for another PyTorch: build it first "
                      "(python -m paper_2505_11157_b200.build). There is no fallback implementation.") from e


_adoption = threading.Lock()


def _adopt(plan: "sna.Plan"):
    """The native owner of the plan from now on: graphs recorded with it may outlive the Python object."""
    with _adoption:
        if plan.native is None:
            plan.native = _sna_torch.Plan(plan.handle or 0, plan.nlat_in, plan.nlon_in, plan.nlat_out, plan.nlon_out)
        return plan.native


class _SphericalNeighborhoodAttention(torch.autograd.Function):
    @staticmethod
    def forward(ctx, plan: "sna.Plan", q, k, v):
        if q.dtype != torch.float32 or k.dtype != torch.float32 or v.dtype != torch.float32:
            raise ValueError("spherical_neighborhood_attention computes in float32: cast q, k, v first "
                             "(autocast does not apply to this operator)")
        q, k, v = q.contiguous(), k.contiguous(), v.contiguous()
        out, lse = plan.forward(q, k, v, return_lse=True)
        ctx.plan = plan
        ctx.save_for_backward(q, k, v, out, lse)
        return out

    @staticmethod
    def backward(ctx, dout):
        q, k, v, out, lse = ctx.saved_tensors
        dq, dk, dv = ctx.plan.backward(q, k, v, dout.contiguous().float(), out=out, lse=lse)
        return None, dq, dk, dv


_PLAIN = frozenset((torch.Tensor, torch.nn.Parameter))


def spherical_neighborhood_attention(plan: "sna.Plan", q: torch.Tensor, k: torch.Tensor, v: torch.Tensor) -> torch.Tensor:
    """out = NAttn_{S^2}[q, k, v] on the grids and cutoff of ``plan`` (differentiable in q, k, v)."""
    # (a trace would keep the native function's allocations and not its kernel launches)
    if type(q) in _PLAIN and type(k) in _PLAIN and type(v) in _PLAIN and torch._C._get_tracing_state() is None:
        owner = plan.native
        if owner is None:
            owner = _adopt(plan)
        out = _sna_torch.attention(owner, q, k, v)
        if out is not None:
            return out
    return _SphericalNeighborhoodAttention.apply(plan, q, k, v)      # (which says what is wrong with arguments that were refused)


class _SphericalNeighborhoodAttentionCF(torch.autograd.Function):
    @staticmethod
    def forward(ctx, plan: "sna.Plan", heads: int, q, k, v):
        if q.dtype != torch.float32 or k.dtype != torch.float32 or v.dtype != torch.float32:
            raise ValueError("spherical_neighborhood_attention_cf computes in float32: cast q, k, v first")
        out, state = plan.forward_cf(q.contiguous(), k.contiguous(), v.contiguous(), heads)
        ctx.plan, ctx.heads, ctx.state = plan, heads, state
        return out

    @staticmethod
    def backward(ctx, dout):
        dq, dk, dv = ctx.plan.backward_cf(dout.contiguous().float(), ctx.state, ctx.heads)
        return None, None, dq, dk, dv


def spherical_neighborhood_attention_cf(plan: "sna.Plan", q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, heads: int = 1) -> torch.Tensor:
    """The same operator on channels-first tensors [B, heads*C, nlat, nlon], as a 2D convolutional network carries
    them; the layout change runs on the GPU inside the call (differentiable in q, k, v)."""
    return _SphericalNeighborhoodAttentionCF.apply(plan, heads, q, k, v)
