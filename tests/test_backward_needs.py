"""The FusedMM and graph-layer backward: only the gradients that are needed are
computed (host logic, with the kernels replaced by a recorder), and the shapes
that the one-pass kernels do not cover get the right values from the separate
steps (GPU, against the FP64 oracle)."""
import types

import numpy as np
import pytest
import torch

import oracle
from helpers import comp_err
from test_gpu_fused_grad import GRAD_TOL, GRAD_TOL_16, _case

import paper_2404_19638_gb300.autograd as ag
from paper_2404_19638_gb300.binding import STATUS, SpkError

DEV = "cuda"
NEEDS = [(True, True), (True, False), (False, True)]


class Recorder:
    """Stands in for the ops module: notes each call, returns host tensors."""

    def __init__(self, covered, M, N, K, nnz, heads):
        self.calls, self.covered, self.shape = [], covered, (M, N, K, nnz, heads)

    def __getattr__(self, name):
        M, N, K, nnz, heads = self.shape

        def call(*args, **kw):
            self.calls.append((name, kw))
            if name == "fused_grad":
                if not self.covered:
                    raise SpkError(next(s for s, c in STATUS.items() if c == "SPK_ERR_UNSUPPORTED"), name, "")
                return torch.zeros(M, K) if kw.get("want_dA", True) else None, torch.zeros(nnz, heads, 2)
            if name in ("spmm_t_pair", "spmm_t_mh"):
                return torch.zeros(N, K)
            if name == "spmm_mh":
                return torch.zeros(M, K)
            if name == "fused_rowdot":
                return torch.zeros(M, heads)
            return torch.zeros(heads, nnz)

        return call


def _pattern(M, nnz, npieces=0):
    return types.SimpleNamespace(M=M, nnz=nnz, has_schedule=True, schedule_info=lambda: {"npieces": npieces})


@pytest.mark.parametrize("need_A,need_B", NEEDS)
@pytest.mark.parametrize("covered,heads", [(True, 2), (False, 2), (False, 1)])
def test_unneeded_gradients_are_not_computed(monkeypatch, covered, heads, need_A, need_B):
    M, N, K, nnz = 5, 4, 8, 7
    rec = Recorder(covered, M, N, K, nnz, heads)
    monkeypatch.setattr(ag, "ops", rec)
    A, B, Y = torch.zeros(M, K), torch.zeros(N, K), torch.zeros(M, K)
    ctx = types.SimpleNamespace(saved_tensors=(torch.empty(0), A, B, Y, torch.zeros(heads, nnz), torch.zeros(M, heads)),
                                S=_pattern(M, nnz), heads=heads, scale=1.0, softmax=True,
                                needs_input_grad=(False, False, need_A, need_B, False, False, False))
    out = ag.FusedMMFunction.backward(ctx, torch.ones(M, K))
    assert (out[2] is not None) == need_A and (out[3] is not None) == need_B
    names = [n for n, _ in rec.calls]
    if covered:
        assert dict(rec.calls)["fused_grad"]["want_dA"] == need_A
        assert names.count("spmm_t_pair") == need_B and "spmm_mh" not in names
    else:
        assert names.count("spmm_mh") == need_A and names.count("spmm_t_mh") == 2 * need_B


@pytest.mark.parametrize("M,nnz,pieces,heads,K,needs,one", [
    (1 << 19, 12 << 20, 0, 1, 64, (True, True), False), (1 << 19, 12 << 20, 9, 1, 64, (True, True), True),
    (1 << 19, 12 << 20, 0, 2, 64, (True, True), True), (1 << 22, 12 << 20, 0, 1, 64, (True, True), True),
    (1 << 22, 12 << 20, 0, 1, 16, (True, True), False), (1 << 18, 4 << 20, 0, 1, 64, (True, True), True),
    (1 << 18, 4 << 20, 0, 1, 64, (False, True), False), (1 << 18, 4 << 20, 0, 1, 32, (False, True), True),
    (1 << 19, 12 << 20, 0, 1, 64, (True, False), True), (1 << 19, 12 << 20, 0, 1, 16, (True, False), False)])
def test_one_pass_or_steps_by_size(monkeypatch, M, nnz, pieces, heads, K, needs, one):
    rec = Recorder(True, 2, 2, K, 1, heads)
    monkeypatch.setattr(ag, "ops", rec)
    X = torch.zeros(2, K)
    ctx = types.SimpleNamespace(saved_tensors=(torch.empty(0), X, X, X, torch.zeros(heads, 1), torch.zeros(2, heads)),
                                S=_pattern(M, nnz, pieces), heads=heads, scale=1.0, softmax=True,
                                needs_input_grad=(False, False, *needs, False, False, False))
    ag.FusedMMFunction.backward(ctx, X)
    assert ("fused_grad" in [n for n, _ in rec.calls]) == one


@pytest.mark.parametrize("K,tried", [(128, True), (132, False), (50, False)])
def test_rows_that_no_one_pass_kernel_covers_are_not_tried(monkeypatch, K, tried):
    rec = Recorder(True, 2, 2, K, 1, 1)
    monkeypatch.setattr(ag, "ops", rec)
    X = torch.zeros(2, K)
    need = (False, False, True, True, False, False, False)
    ctx = types.SimpleNamespace(saved_tensors=(torch.empty(0), X, X, X, torch.zeros(1, 1), torch.zeros(2, 1)),
                                S=_pattern(2, 1), heads=1, scale=1.0, softmax=True, needs_input_grad=need)
    ag.FusedMMFunction.backward(ctx, X)
    assert ("fused_grad" in [n for n, _ in rec.calls]) == tried
    rec.calls.clear()
    monkeypatch.setattr(rec, "sddmm", lambda *a, **k: None, raising=False)
    monkeypatch.setattr(rec, "spmm", lambda *a, **k: X, raising=False)
    ctx = types.SimpleNamespace(saved_tensors=(torch.empty(0), X, torch.zeros(1)), S=_pattern(2, 1))
    ag.GNNLayerFunction.backward(ctx, X)
    assert ("fused_grad" in [n for n, _ in rec.calls]) == tried


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _np(X):
    return X.cpu().numpy() if X.dtype == torch.float32 else X.view(torch.int16).cpu().numpy().view(np.uint16)


# rows over 512 bytes, heads that are no power of two of vectors; then shapes that the one-pass kernels cover
@pytest.mark.gpu
@pytest.mark.parametrize("need_A,need_B", NEEDS)
@pytest.mark.parametrize("softmax", [False, True])
@pytest.mark.parametrize("dt,K,heads", [("f32", 132, 1), ("f32", 72, 2), ("bf16", 264, 1), ("f32", 64, 4), ("bf16", 64, 1)])
def test_fusedmm_gradients_each_and_both(spk, dt, K, heads, softmax, need_A, need_B):
    M, N = 330, 270
    rp, ci, vals, A, B, dY = _case(M, N, K, seed=K + heads)
    A, B, dY = 0.3 * A, 0.3 * B, 0.3 * dY
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    tA, tB = (torch.from_numpy(X).to(DEV) for X in (A, B))
    if dt == "bf16":
        tA, tB = spk.cast(tA, torch.bfloat16), spk.cast(tB, torch.bfloat16)
    fmt = None if dt == "f32" else dt
    args = (rp, ci, _np(tA), _np(tB), dY, vals)
    kw = dict(heads=heads, scale=0.4, softmax=softmax, fmt=fmt)
    ref, den = oracle.fusedmm_grad(*args, **kw), oracle.fusedmm_grad(*args, absmode=True, **kw)
    tA.requires_grad_(need_A)
    tB.requires_grad_(need_B)
    Y = spk.autograd.fusedmm(S, tA, tB, S.vals, heads=heads, scale=0.4, softmax=softmax)
    Y.backward(torch.from_numpy(dY).to(DEV))
    for X, need, r, d in ((tA, need_A, ref[0], den[0]), (tB, need_B, ref[1], den[1])):
        assert (X.grad is not None) == need
        if need:
            assert comp_err(X.grad.float().cpu().numpy(), r, d) <= (GRAD_TOL if dt == "f32" else GRAD_TOL_16)


@pytest.mark.gpu
@pytest.mark.parametrize("K", [32, 48, 64])
@pytest.mark.parametrize("softmax", [False, True])
def test_separate_steps_on_covered_heads(spk, K, softmax):
    """The multi-head dw of the separate steps (K = 32, 64) and one SDDMM a head (48), on shapes that autograd gives
    to the one-pass kernels."""
    M, N, heads = 300, 260, 2
    rp, ci, vals, A, B, dY = _case(M, N, K, seed=K)
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    tA, tB, tY = (torch.from_numpy(X).to(DEV) for X in (A, B, dY))
    Y, sc, lse = spk.fusedmm(S, tA, tB, heads=heads, scale=0.2, softmax=softmax, want_scores=True, want_lse=True)
    R = spk.ops.fused_rowdot(tY, Y, heads) if softmax else None
    dA, dB = ag._fused_backward_steps(S, S.vals, tA, tB, sc, lse, tY, R, heads, 0.2, softmax, True, True)
    kw = dict(heads=heads, scale=0.2, softmax=softmax)
    ref, den = (oracle.fusedmm_grad(rp, ci, A, B, dY, vals, absmode=m, **kw) for m in (False, True))
    for got, r, d in ((dA, ref[0], den[0]), (dB, ref[1], den[1])):
        assert comp_err(got.cpu().numpy(), r, d) <= GRAD_TOL


@pytest.mark.gpu
@pytest.mark.parametrize("K", [7, 50, 64, 132])
def test_gnn_layer_gradient(spk, K):
    """The graph layer on widths with and without one-pass kernels."""
    M = 310
    rp, ci, vals, H, _, dY = _case(M, M, K, seed=K)
    H = 0.3 * H
    S = spk.CSR(rp, ci, (M, M), torch.from_numpy(vals), device=DEV, chunk_work=96)
    tH = torch.from_numpy(H).to(DEV).requires_grad_()
    spk.autograd.gnn_layer(S, tH, S.vals).backward(torch.from_numpy(dY).to(DEV))
    ref = oracle.gnn_grad(rp, ci, H, dY, vals)
    den = oracle.gnn_grad(rp, ci, np.abs(H), np.abs(dY), np.abs(vals))
    assert comp_err(tH.grad.cpu().numpy(), ref, den) <= GRAD_TOL
