"""SDDMM and SpMM on rows that 16 bytes do not divide (copies of 8 and 4 bytes):
widths around the vector, lane and block sizes, operands at odd offsets and
strides, every value and output form.  SpMM adds its nonzeros in slot order on
every path, so it equals the register path bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, comp_err, edge_pattern

pytestmark = pytest.mark.gpu
DEV = "cuda"
DTS = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _np(X):
    X = X.contiguous()
    return X.cpu().numpy() if X.dtype == torch.float32 else X.view(torch.int16).cpu().numpy().view(np.uint16)


# FP32 1..4 elements past each block; 16-bit even widths; odd 16-bit widths stay on the element path
WIDTHS = [("f32", K) for K in (1, 2, 3, 5, 7, 9, 14, 17, 31, 33, 50, 63, 65, 66, 99, 127, 129, 130, 257)] + \
         [(dt, K) for dt in ("bf16", "f16") for K in (2, 6, 9, 18, 30, 34, 50, 66, 100, 126, 130, 250, 258)]


@pytest.mark.parametrize("dt,K", WIDTHS)
@pytest.mark.parametrize("view", ["whole", "shifted"])
def test_widths(spk, dt, K, view):
    M, N, pad = 300, 260, 2 if view == "shifted" else 0
    rp, ci = edge_pattern(M, N, K, long_row=700)
    g = np.random.default_rng(K)
    A, B = (torch.from_numpy(g.standard_normal((n, K + 2 * pad)).astype(np.float32)).to(DEV).to(DTS[dt])[:, pad:pad + K]
            for n in (M, N))
    vals = g.uniform(-1, 1, ci.size).astype(np.float32)
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    fmt = None if dt == "f32" else dt
    e = spk.sddmm(S, A, B)
    ref, den = (oracle.sddmm(rp, ci, _np(A), _np(B), vals, fmt_a=fmt, fmt_b=fmt, absmode=m) for m in (False, True))
    assert comp_err(e.cpu().numpy(), ref, den) <= TOL
    if dt != "f32":
        Af = A.float()
        e = spk.sddmm(S, Af, B)
        assert comp_err(e.cpu().numpy(), ref, den) <= TOL
    C = spk.spmm(S, B)
    ref, den = (oracle.spmm(rp, ci, _np(B), vals, fmt_b=fmt, absmode=m) for m in (False, True))
    assert comp_err(C.cpu().numpy(), ref, den) <= TOL
    assert torch.equal(C, spk.spmm(S, B, tune={"variant": 3}))


@pytest.mark.parametrize("K", [3, 50, 131])
@pytest.mark.parametrize("mode", ["none", "both", "accumulate", "bf16", "f16_accumulate", "transpose", "strided_out"])
def test_values_and_outputs(spk, K, mode):
    M, N = 310, 290
    rp, ci = edge_pattern(M, N, K, long_row=900)
    g = np.random.default_rng(K)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    B = torch.from_numpy(g.standard_normal((N, K)).astype(np.float32)).to(DEV)
    A = torch.from_numpy(g.standard_normal((M, K)).astype(np.float32)).to(DEV)
    v1, v2 = (torch.from_numpy(g.uniform(-1, 1, ci.size).astype(np.float32)).to(DEV) for _ in range(2))
    args = {"none": (None, None), "both": (v1, v2), "transpose": (v1, v2)}.get(mode, (v1, None))
    got = []
    for tune in (None, {"variant": 3}):
        kw = dict(tune=tune)
        if mode in ("bf16", "f16_accumulate"):
            kw["out_dtype"] = torch.bfloat16 if mode == "bf16" else torch.float16
        if mode in ("accumulate", "f16_accumulate"):
            kw.update(out=(A if mode == "accumulate" else A.half()).clone(), accumulate=True)
        if mode == "strided_out":
            kw["out"] = torch.zeros(M, K + 3, device=DEV)[:, 1:1 + K]
        got.append(spk.spmm_t(S, A, *args, **kw) if mode == "transpose" else spk.spmm(S, B, *args, **kw))
    assert torch.equal(got[0], got[1])


def test_rows_of_few_entries(spk):
    """More row starts in a batch than rows of A copied with it."""
    M, N, K = 900, 700, 50
    g = np.random.default_rng(1)
    rp = np.zeros(M + 1, np.int32)
    np.cumsum(g.integers(0, 3, M), out=rp[1:])
    ci = g.integers(0, N, rp[-1]).astype(np.int32)
    S = spk.CSR(rp, ci, (M, N), device=DEV)
    A, B = (torch.from_numpy(g.standard_normal((n, K)).astype(np.float32)).to(DEV) for n in (M, N))
    e = spk.sddmm(S, A, B).cpu().numpy()
    ref, den = (oracle.sddmm(rp, ci, _np(A), _np(B), absmode=m) for m in (False, True))
    assert comp_err(e, ref, den) <= TOL
