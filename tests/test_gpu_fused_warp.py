"""FusedMM and its backward, one warp per chunk: widths around every copy width,
rows shorter than a batch (more row starts than the rows of A copied with it),
rows that end on batch, tile and chunk edges, heads, value forms and
infinities.  Against the FP64 oracle (forward) and against the same steps as
separate kernels (backward), at the componentwise FP32 gate."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, comp_err

pytestmark = pytest.mark.gpu
DEV = "cuda"
DTS = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _pattern(kind, M, N, seed):
    """Row pointers and columns: degrees 0-3 (``short``), multiples of the batch
    sizes (``edges``), one long row among empty ones (``long``), or mixed."""
    g = np.random.default_rng(seed)
    deg = {"short": g.integers(0, 4, M), "edges": g.choice([0, 8, 16, 31, 32, 33, 64], M), "mixed": g.integers(0, 60, M),
           "long": np.where(np.arange(M) == M // 2, 1500, (np.arange(M) % 9 == 0) * 2)}[kind]
    rp = np.zeros(M + 1, np.int32)
    np.cumsum(deg, out=rp[1:])
    return rp, g.integers(0, N, rp[-1]).astype(np.int32)


def _operands(dt, M, N, K, seed):
    g = torch.Generator().manual_seed(seed)
    A, B = (0.5 * torch.randn(n, K, generator=g) for n in (M, N))
    A, B = A.to(DTS[dt]).to(DEV), B.to(DTS[dt]).to(DEV)
    return A, B, torch.randn(M, K, generator=g).to(DEV)


def _np(X):
    return X.cpu().numpy() if X.dtype == torch.float32 else X.view(torch.int16).cpu().numpy().view(np.uint16)


SHAPES = [("f32", K, h) for K, h in ((4, 1), (8, 2), (16, 4), (20, 1), (32, 8), (48, 3), (64, 1), (64, 16), (100, 1),
                                     (128, 1), (128, 32), (96, 2))] + \
         [(dt, K, h) for dt in ("bf16", "f16") for K, h in ((8, 1), (16, 2), (24, 3), (64, 4), (72, 1), (128, 2), (256, 1),
                                                           (256, 32))]


@pytest.mark.parametrize("dt,K,heads", SHAPES)
@pytest.mark.parametrize("kind", ["short", "edges", "long"])
def test_forward(spk, dt, K, heads, kind):
    M, N = 260, 190
    rp, ci = _pattern(kind, M, N, K + heads)
    A, B, _ = _operands(dt, M, N, K, K)
    vals = np.random.default_rng(K).uniform(0.5, 1.5, ci.size).astype(np.float32)
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    fmt = None if dt == "f32" else dt
    for softmax in (False, True):
        Y, sc, lse = spk.fusedmm(S, A, B, heads=heads, scale=0.3, softmax=softmax, want_scores=True, want_lse=True)
        kw = dict(heads=heads, scale=0.3, softmax=softmax, fmt_a=fmt, fmt_b=fmt)
        Yr, scr, lser = oracle.fusedmm(rp, ci, _np(A), _np(B), vals, **kw)
        Ya, _, _ = oracle.fusedmm(rp, ci, _np(A), _np(B), vals, absmode=True, **kw)
        assert comp_err(Y.cpu().numpy(), Yr, Ya) <= TOL
        D = K // heads
        for h in range(heads):
            s = slice(h * D, (h + 1) * D)
            den = 0.3 * oracle.sddmm(rp, ci, np.ascontiguousarray(_np(A)[:, s]), np.ascontiguousarray(_np(B)[:, s]), vals,
                                     fmt_a=fmt, fmt_b=fmt, absmode=True)
            assert comp_err(sc[h].cpu().numpy(), scr[h], den) <= TOL
        if softmax:
            got, fin = lse.cpu().numpy(), np.isfinite(lser)
            assert np.array_equal(np.isfinite(got), fin)
            assert np.max(np.abs(got[fin] - lser[fin]) / (1 + np.abs(lser[fin])), initial=0.0) <= TOL


@pytest.mark.parametrize("dt,K,heads", SHAPES)
@pytest.mark.parametrize("kind,with_vals,softmax", [("short", False, True), ("edges", True, False), ("mixed", True, True),
                                                     ("long", False, False)])
def test_backward_equals_separate_steps(spk, dt, K, heads, kind, with_vals, softmax):
    M, N = 240, 210
    rp, ci = _pattern(kind, M, N, K + heads)
    A, B, dY = _operands(dt, M, N, K, K + 1)
    g = np.random.default_rng(K)
    v = torch.from_numpy(g.uniform(0.5, 1.5, ci.size).astype(np.float32)).to(DEV) if with_vals else None
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=96)
    S.transpose_plan(96)
    kw = dict(heads=heads, scale=0.3, softmax=softmax)
    Y, sc, lse = spk.fusedmm(S, A, B, v, want_scores=True, want_lse=True, use_default_vals=False, **kw)
    R = spk.ops.fused_rowdot(dY, Y, heads) if softmax else None
    nhv = K // heads // (4 if dt == "f32" else 8)
    if heads > 1 and nhv & (nhv - 1):                  # 12 vectors a head do not halve: refused
        with pytest.raises(spk.SpkError):
            spk.ops.fused_grad(S, B, dY, sc, lse, R, heads, softmax, 0.3, v)
        return
    dA, cw = spk.ops.fused_grad(S, B, dY, sc, lse, R, heads, softmax, 0.3, v)
    dB = spk.ops.spmm_t_pair(S, cw, A, dY)
    base = torch.ones_like(dB)
    spk.ops.spmm_t_pair(S, cw, A, dY, out=base, accumulate=True)
    # FP64 chain rule from the same scores, lse and row term; den: the magnitudes that each entry adds up
    rows = torch.from_numpy(np.repeat(np.arange(M), np.diff(rp))).to(DEV)
    cols = torch.from_numpy(ci).long().to(DEV)
    D = K // heads
    for h in range(heads):
        s = slice(h * D, (h + 1) * D)
        Bh, Ah, Yh = B[:, s].double(), A[:, s].double(), dY[:, s].double()
        x = sc[h].double()
        w = torch.exp(x - lse[rows, h].double()) if softmax else x
        ww = w * (1 + (x - lse[rows, h].double()).abs()) if softmax else w.abs()      # exp widens its argument's error
        r = R[rows, h].double() if softmax else torch.zeros_like(x)
        dw, adw = (Yh[rows] * Bh[cols]).sum(1), (Yh[rows] * Bh[cols]).abs().sum(1)
        sv = 0.3 * (v.double() if v is not None else torch.ones_like(x))
        c, ac = (sv * w * (dw - r), sv * ww * (adw + r.abs())) if softmax else (sv * dw, sv * adw)
        got = cw[:, h].double()
        assert comp_err(got[:, 0].cpu().numpy(), c.cpu().numpy(), ac.cpu().numpy()) <= TOL
        assert comp_err(got[:, 1].cpu().numpy(), w.cpu().numpy(), ww.cpu().numpy()) <= TOL

        def scatter(n, idx, t):
            return torch.zeros(n, D, dtype=torch.float64, device=DEV).index_add_(0, idx, t).cpu().numpy()

        assert comp_err(dA[:, s].cpu().numpy(), scatter(M, rows, c[:, None] * Bh[cols]),
                        scatter(M, rows, ac[:, None] * Bh[cols].abs())) <= TOL
        ref = scatter(N, cols, c[:, None] * Ah[rows] + w[:, None] * Yh[rows])
        den = scatter(N, cols, ac[:, None] * Ah[rows].abs() + ww[:, None] * Yh[rows].abs())
        assert comp_err(dB[:, s].cpu().numpy(), ref, den) <= TOL
        assert comp_err(base[:, s].cpu().numpy(), ref + 1, den + 1) <= TOL
    assert torch.equal(cw, spk.ops.fused_grad(S, B, dY, sc, lse, R, heads, softmax, 0.3, v)[1])


def test_uncovered_shapes_are_refused_and_fall_back(spk):
    M, N = 150, 140
    rp, ci = _pattern("mixed", M, N, 3)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    for dt, K, heads in (("f32", 132, 1), ("f32", 72, 2), ("bf16", 264, 1)):
        A, B, dY = _operands(dt, M, N, K, 4)
        A.requires_grad_(); B.requires_grad_()
        Y, sc, _ = spk.fusedmm(S, A.detach(), B.detach(), heads=heads, want_scores=True)
        with pytest.raises(spk.SpkError):
            spk.ops.fused_grad(S, B.detach(), dY, sc, None, None, heads, False, 1.0)
        out = spk.autograd.fusedmm(S, A, B, heads=heads, scale=1.0)
        out.backward(dY)
        assert A.grad.shape == A.shape and torch.isfinite(A.grad.float()).all() and torch.isfinite(B.grad.float()).all()


def test_infinities_stay_in_their_rows(spk):
    M, N, K = 120, 100, 64
    rp, ci = _pattern("mixed", M, N, 9)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    A, B, _ = _operands("f32", M, N, K, 2)
    B[7, 3], B[9, 0] = float("inf"), float("nan")
    hit = np.zeros(M, bool)
    hit[np.repeat(np.arange(M), np.diff(rp))[(ci == 7) | (ci == 9)]] = True
    for softmax in (False, True):
        Y, _, _ = spk.fusedmm(S, A, B, softmax=softmax)
        O, _, _ = spk.fusedmm(S, A, B, softmax=softmax, tune={"vecs_per_lane": 1})
        ok = ~torch.from_numpy(hit).to(DEV)
        assert torch.isfinite(Y[ok]).all()
        torch.testing.assert_close(Y[ok], O[ok], rtol=1e-5, atol=1e-5)
