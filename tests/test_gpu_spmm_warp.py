"""SpMM, one warp per chunk: row widths around every copy width and K block,
partial batches and index tiles, values in every form the entry point takes.
Every output element adds its nonzeros in slot order, so the balanced default
equals the register path bit for bit, and both match the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, comp_err, edge_pattern

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _factor(spk, dt, n, K, g):
    X = torch.from_numpy(g.standard_normal((n, K)).astype(np.float32)).to(DEV)
    if dt == "e4m3":
        q, s = spk.quantize_e4m3_rows(X)
        return q, s, dict(fmt_b=None, b_scale=s.cpu().numpy()), q.view(torch.uint8).cpu().numpy()
    if dt == "f32":
        return X, None, {}, X.cpu().numpy()
    q = spk.cast(X, torch.bfloat16 if dt == "bf16" else torch.float16)
    return q, None, dict(fmt_b=dt), q.view(torch.int16).cpu().numpy().view(np.uint16)


# bytes of a row: 16, below / at / above each of 32, 64, 128, 256, 512, and two K blocks with a ragged second
WIDTHS = [("f32", K) for K in (4, 8, 12, 16, 20, 32, 36, 64, 68, 128, 132, 260)] + \
         [(dt, K) for dt in ("bf16", "f16") for K in (8, 24, 32, 64, 72, 128, 136, 256, 264)] + \
         [("e4m3", K) for K in (16, 32, 48, 128, 144, 512, 528)]


@pytest.mark.parametrize("dt,K", WIDTHS)
def test_row_widths(spk, dt, K):
    M, N = 310, 270
    rp, ci = edge_pattern(M, N, K, long_row=700)
    g = np.random.default_rng(K)
    vals = g.uniform(-1, 1, ci.size).astype(np.float32)
    B, s, kw, Bn = _factor(spk, dt, N, K, g)
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    C = spk.spmm(S, B, b_scale=s)
    if dt == "e4m3":
        kw.pop("fmt_b")
    ref, den = (oracle.spmm(rp, ci, Bn, vals, absmode=m, **kw) for m in (False, True))
    assert comp_err(C.cpu().numpy(), ref, den) <= TOL
    assert torch.equal(C, spk.spmm(S, B, b_scale=s, tune={"variant": 3}))


@pytest.mark.parametrize("W", [32, 33, 64, 512])
@pytest.mark.parametrize("mode", ["plain", "none", "vals2_only", "both", "shifted", "accumulate", "bf16", "f16_accumulate",
                                  "transpose", "transpose_none", "strided"])
def test_values_outputs_and_chunks(spk, mode, W):
    M, N, K = 500, 390, 48
    rp, ci = edge_pattern(M, N, 5 * W, long_row=1500)
    g = np.random.default_rng(W)
    nnz = ci.size
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=W)
    P = S.transpose_plan(W)
    B = torch.from_numpy(g.standard_normal((N, K + 8)).astype(np.float32)).to(DEV)
    B = B[:, 4:4 + K] if mode == "strided" else B[:, :K].contiguous()
    A = torch.from_numpy(g.standard_normal((M, K)).astype(np.float32)).to(DEV)
    v = torch.from_numpy(g.uniform(-1, 1, nnz + 1).astype(np.float32)).to(DEV)
    v1, v2 = v[:nnz].contiguous(), torch.flip(v, (0,))[:nnz].contiguous()
    args = {"none": (None, None), "vals2_only": (None, v2), "both": (v1, v2), "shifted": (v[1:], None),
            "transpose_none": (None, None)}.get(mode, (v1, None))
    got = []
    for tune in (None, {"variant": 3}):
        kw = dict(tune=tune)
        if mode in ("bf16", "f16_accumulate"):
            kw["out_dtype"] = torch.bfloat16 if mode == "bf16" else torch.float16
        if mode in ("accumulate", "f16_accumulate"):
            kw["out"] = (A if mode == "accumulate" else A.half()).clone()
            kw.update(accumulate=True)
        if mode.startswith("transpose"):
            got.append(spk.spmm_t(S, A, *args, plan=P, **kw))
        else:
            got.append(spk.spmm(S, B, *args, **kw))
    assert torch.equal(got[0], got[1])
    if mode in ("plain", "strided"):
        Bn = B.cpu().numpy()
        ref, den = (oracle.spmm(rp, ci, Bn.copy(), v1.cpu().numpy(), absmode=m) for m in (False, True))
        assert comp_err(got[0].cpu().numpy(), ref, den) <= TOL


def test_infinities_and_nan_stay_in_their_rows(spk):
    M, N, K = 200, 150, 64
    rp, ci = edge_pattern(M, N, 77, long_row=300)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    B = torch.randn(N, K, device=DEV)
    B[3, 5], B[10, 0], B[11, 63] = float("inf"), float("nan"), -float("inf")
    C, R = spk.spmm(S, B), spk.spmm(S, B, tune={"variant": 1})
    assert torch.equal(torch.isnan(C), torch.isnan(R)) and torch.equal(torch.isinf(C), torch.isinf(R))
    fin = torch.isfinite(R)
    torch.testing.assert_close(C[fin], R[fin], rtol=1e-5, atol=1e-4)


@pytest.mark.parametrize("dt,K", [("f32", 32), ("bf16", 64), ("e4m3", 48), ("f32", 260)])
@pytest.mark.parametrize("both", [False, True])
def test_transpose_gathers_values_through_the_plan(spk, dt, K, both):
    """S^T Y takes the values through the slot permutation while it loads its
    index tiles; the register path reads them permuted into the workspace."""
    M, N = 330, 401
    rp, ci = edge_pattern(M, N, K + 5, long_row=900)
    g = np.random.default_rng(K)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    P = S.transpose_plan(64)
    Y, s, _, _ = _factor(spk, dt, M, K, g)
    v = [torch.from_numpy(g.uniform(-1, 1, ci.size).astype(np.float32)).to(DEV) for _ in range(2)]
    args = (v[0], v[1]) if both else (None, v[1])
    got = [spk.spmm_t(S, Y, *args, y_scale=s, plan=P, tune=t) for t in (None, {"variant": 3})]
    assert torch.equal(got[0], got[1])
