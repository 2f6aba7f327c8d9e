"""Differentiation through the SDDMM / SpMM adjoint pair (Sec. 3.2).

Both operations take or output two dense vectors per nonzero, and each one's
gradient is the other one:

  SpMM   C = S B            dB = S^T dC  (SpMM^T via the transpose plan)
                            ds_e = <dC_i, b_j>  (an SDDMM with unit values)
  SDDMM  c_e = s_e<a_i,b_j>  dA = (S.g) B  (SpMM with values s*g)
                            dB = (S.g)^T A  (SpMM^T with values s*g)
                            ds_e = g_e <a_i, b_j>  (SDDMM with values g)

Every backward step is one of the library's kernels; gradients of BF16 / F16
factors are written in the factor's dtype by the kernel itself (FP32
accumulation inside).  The pattern S is not differentiated; its values are.
"""
from __future__ import annotations

import torch

from . import ops
from .binding import SpkError
from .sparse import CSR


def _vals_or_none(v):
    return v if (v is not None and v.numel() > 0) else None


class SDDMMFunction(torch.autograd.Function):
    @staticmethod
    def forward(ctx, S: CSR, vals, A, B):
        ctx.S = S
        ctx.save_for_backward(vals, A, B)
        return ops.sddmm(S, A, B, _vals_or_none(vals), use_default_vals=False)

    @staticmethod
    def backward(ctx, g):
        vals, A, B = ctx.saved_tensors
        S = ctx.S
        g = g.contiguous().float()
        v = _vals_or_none(vals)
        dvals = dA = dB = None
        if ctx.needs_input_grad[1]:
            dvals = ops.sddmm(S, A, B, g, use_default_vals=False)
        if ctx.needs_input_grad[2]:
            dA = ops.spmm(S, B, v, g, out_dtype=A.dtype, use_default_vals=False)
        if ctx.needs_input_grad[3]:
            dB = ops.spmm_t(S, A, v, g, out_dtype=B.dtype, use_default_vals=False)
        return None, dvals, dA, dB


class SpMMFunction(torch.autograd.Function):
    @staticmethod
    def forward(ctx, S: CSR, vals, B):
        ctx.S = S
        ctx.save_for_backward(vals, B)
        return ops.spmm(S, B, _vals_or_none(vals), use_default_vals=False)

    @staticmethod
    def backward(ctx, dC):
        vals, B = ctx.saved_tensors
        S = ctx.S
        dC = dC.contiguous().float()
        dvals = dB = None
        if ctx.needs_input_grad[1]:
            dvals = ops.sddmm(S, dC, B, use_default_vals=False)
        if ctx.needs_input_grad[2]:
            dB = ops.spmm_t(S, dC, _vals_or_none(vals), out_dtype=B.dtype, use_default_vals=False)
        return None, dvals, dB


def sddmm(S: CSR, A, B, vals=None):
    """Differentiable SDDMM; ``vals`` None means all ones (not differentiated)."""
    if vals is None:
        vals = torch.empty(0, dtype=torch.float32, device=S.device)
    return SDDMMFunction.apply(S, vals, A, B)


def spmm(S: CSR, B, vals=None):
    """Differentiable SpMM (FP32 output)."""
    if vals is None:
        vals = torch.empty(0, dtype=torch.float32, device=S.device)
    return SpMMFunction.apply(S, vals, B)


def _one_pass_rows(row_bytes: int) -> bool:
    """Rows of B that the one-pass kernels may cover.  Others are not tried: the call that refuses them comes after
    its outputs are allocated, 20-40 us of host time."""
    return row_bytes <= 512 and row_bytes % 16 == 0


def _one_pass(S: CSR, heads: int, row_bytes: int, need_dA: bool, need_dB: bool) -> bool:
    """Whether the one-pass backward beats the separate steps, by size.  It saves
    launches, gathers and (several heads) most of the traffic; with one head, on
    large patterns without split rows, each of its two kernels holds more per
    entry in flight and in L2 than the steps do.  Time of the one-pass kernels
    over the steps, GB300, uniform rows of 24 / bipartite of 25: dA and dB, 8M
    entries FP32 K = 16 1.17 / 1.08, K = 64 1.32 / 1.22, BF16 K = 128 1.25 / 1.27;
    16M 1.13-1.36; 2M 0.65-1.1; uniform rows of 8 0.9-1.0 from 128 bytes on.  dB
    alone, 4M FP32 K = 64 1.34 / 1.38, 8M FP32 K = 32 1.19 / 1.11; dA alone, 8M
    K = 16 1.18 / 1.13.  4 heads 0.5-0.95 everywhere; R-MAT (split rows) 0.9-1.15."""
    if not _one_pass_rows(row_bytes):
        return False
    if heads > 1 or S.nnz < 3 << 20 or S.schedule_info()["npieces"] > 0:
        return True
    big = S.nnz >= 6 << 20
    if row_bytes <= 64:
        return not big
    if need_dA:
        return not (need_dB and big and S.nnz >= 12 * S.M)
    return row_bytes < 256 and not big


class GNNLayerFunction(torch.autograd.Function):
    """Y = SpMM(S_e, H) with e = SDDMM(S, H, H): an attention-style graph layer.

    Backward accumulates the three contributions to dH in FP32 inside the
    kernels (accumulate mode) and writes H's dtype once:
      dE_e = <dY_i, h_j>;  dH = (S.dE) H + (S.dE)^T H + S_e^T dY.
    """

    @staticmethod
    def forward(ctx, S: CSR, vals, H):
        v = _vals_or_none(vals)
        e = ops.sddmm(S, H, H, v, use_default_vals=False)
        Y = ops.spmm(S, H, e, use_default_vals=False)
        ctx.S = S
        ctx.save_for_backward(vals, H, e)
        return Y

    @staticmethod
    def backward(ctx, dY):
        vals, H, e = ctx.saved_tensors
        S = ctx.S
        dY = dY.contiguous().float()
        v = _vals_or_none(vals)
        acc = None
        # the steps: FP32 rows of up to 64 bytes on large uniform patterns (16M entries, 24 a row, K = 16: 1 / 1.27 of
        # the one-pass time; 8 a row 1 / 1.01; wider and 16-bit rows gain by the one pass)
        row_bytes = H.size(1) * H.element_size()
        if S.has_schedule and _one_pass_rows(row_bytes) and (H.dtype != torch.float32 or H.size(1) > 16
                                                             or _one_pass(S, 1, row_bytes, True, False)):
            try:                                   # (dE, (S.dE) H) in one pass over S, the two S^T products in another
                acc, ee = ops.fused_grad(S, H, dY, e.reshape(1, -1), None, None, 1, False, 1.0, v)
                ops.spmm_t_pair(S, ee, H, dY, out=acc, accumulate=True)
            except SpkError as err:
                if err.code != "SPK_ERR_UNSUPPORTED":
                    raise
                acc = None
        if acc is None:
            dE = ops.sddmm(S, dY, H, use_default_vals=False)
            acc = ops.spmm(S, H, v, dE, use_default_vals=False)
            ops.spmm_t(S, H, v, dE, out=acc, accumulate=True, use_default_vals=False)
            ops.spmm_t(S, dY, e, out=acc, accumulate=True, use_default_vals=False)
        dH = acc if H.dtype == torch.float32 else ops.cast(acc, H.dtype)
        return None, None, dH


def gnn_layer(S: CSR, H, vals=None):
    if vals is None:
        vals = torch.empty(0, dtype=torch.float32, device=S.device)
    return GNNLayerFunction.apply(S, vals, H)


def _dw_per_head(S, dY, B, dw, heads, Kh):
    for h in range(heads):
        c0 = h * Kh
        ops.sddmm(S, dY[:, c0:c0 + Kh], B[:, c0:c0 + Kh], out=dw[h], use_default_vals=False)


def _fused_backward_steps(S, v, A, B, scores, lse, dY, R, heads, scale, softmax, need_dA, need_dB):
    """dA and dB (FP32; None where not needed) in separate passes: dw by one
    multi-head SDDMM (FP32 operands; one SDDMM per head otherwise, or where no
    multi-head kernel covers K), the score gradient c, dA = one multi-head
    SpMM, dB = two multi-head SpMM^T."""
    Kh = A.size(1) // heads
    w = ops.fused_weights(S, scores, lse, heads, softmax) if softmax else scores
    dw = torch.empty_like(scores)
    if B.dtype == torch.float32 and heads > 1:
        try:                                       # all heads in one pass over the pattern
            ops.sddmm_mh(S, dY, B, heads, out=dw)
        except SpkError as err:                    # no multi-head kernel for this K: one SDDMM per head
            if err.code != "SPK_ERR_UNSUPPORTED":
                raise
            _dw_per_head(S, dY, B, dw, heads, Kh)
    else:
        _dw_per_head(S, dY, B, dw, heads, Kh)
    c = ops.fused_score_grad(S, w, dw, R, heads, softmax, scale, v)
    dA = ops.spmm_mh(S, B, c, heads) if need_dA else None
    dB = None
    if need_dB:
        dB = ops.spmm_t_mh(S, A, c, heads)
        ops.spmm_t_mh(S, dY, w, heads, out=dB, accumulate=True)
    return dA, dB


class FusedMMFunction(torch.autograd.Function):
    """Differentiable FusedMM: per head h, e = scale * s * <A_i, B_j>,
    w = e or its row softmax, Y_i = sum_j w_ij B_j.

    Backward (chain rule, per head; dw_ij = <dY_i, B_j>):
      g = dw, or w * (dw - rowdot_i) with softmax, rowdot_i = sum_j w_ij dw_ij
          = <dY_i, Y_i> (read from the saved output)
      c = scale * s * g;  dA = C B;  dB = C^T A + W^T dY  (C, W: S's pattern
      holding c, w)
    Steps: the row term; one pass over S that gathers B once for dw, the
    weights, c and dA (ops.fused_grad); one pass over S^T that adds both
    products of dB to one output (ops.spmm_t_pair), all heads at once, in
    FP32.  Where those kernels don't cover K, the heads or the alignment, or are
    the slower way (_one_pass), the same steps one by one
    (_fused_backward_steps).  The sparse values are not
    differentiated.
    """

    @staticmethod
    def forward(ctx, S: CSR, vals, A, B, heads: int, scale: float, softmax: bool):
        v = _vals_or_none(vals)
        Y, scores, lse = ops.fusedmm(S, A, B, v, heads=heads, scale=scale, softmax=softmax, want_scores=True,
                                     want_lse=softmax, use_default_vals=False)
        ctx.S, ctx.heads, ctx.scale, ctx.softmax = S, heads, scale, softmax
        ctx.save_for_backward(vals, A, B, Y, scores, lse if softmax else scores[:0])
        return Y

    @staticmethod
    def backward(ctx, dY):
        vals, A, B, Y, scores, lse = ctx.saved_tensors
        S, heads, scale, softmax = ctx.S, ctx.heads, ctx.scale, ctx.softmax
        dY = dY.contiguous().float()
        v = _vals_or_none(vals)
        need_dA, need_dB = ctx.needs_input_grad[2:4]
        R = ops.fused_rowdot(dY, Y, heads) if softmax else None
        done = False
        if _one_pass(S, heads, B.size(1) * B.element_size(), need_dA, need_dB):
            try:
                dA, cw = ops.fused_grad(S, B, dY, scores, lse, R, heads, softmax, scale, v, want_dA=need_dA)
                dB = ops.spmm_t_pair(S, cw, A, dY) if need_dB else None
                done = True
            except SpkError as err:                # no one-pass kernels for this K and these heads
                if err.code != "SPK_ERR_UNSUPPORTED":
                    raise
        if not done:
            dA, dB = _fused_backward_steps(S, v, A, B, scores, lse, dY, R, heads, scale, softmax, need_dA, need_dB)
        if dA is not None and A.dtype != torch.float32:
            dA = ops.cast(dA, A.dtype)
        if dB is not None and B.dtype != torch.float32:
            dB = ops.cast(dB, B.dtype)
        return None, None, dA, dB, None, None, None


def fusedmm(S: CSR, A, B, vals=None, *, heads: int = 1, scale: float = 1.0, softmax: bool = False):
    """Differentiable FusedMM (FP32 output M x K); ``vals`` None means all ones."""
    if vals is None:
        vals = torch.empty(0, dtype=torch.float32, device=S.device)
    return FusedMMFunction.apply(S, vals, A, B, int(heads), float(scale), bool(softmax))


__all__ = ["SDDMMFunction", "SpMMFunction", "GNNLayerFunction", "FusedMMFunction", "sddmm", "spmm", "gnn_layer",
           "fusedmm"]
