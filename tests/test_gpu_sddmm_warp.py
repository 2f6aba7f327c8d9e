"""SDDMM, one warp per chunk: row widths around every lane layout, rows of one
entry up to rows longer than a chunk (more row starts in a batch than copied A
rows, none at all), partial batches, and every dtype pair."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, comp_err, edge_pattern
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _pattern(kind, M, N, seed):
    if kind == "edge":
        return edge_pattern(M, N, seed, long_row=700)
    deg = {"ones": 1, "twos": 2, "fives": 5}[kind]
    g = np.random.default_rng(seed)
    return synth.csr_from_coo(np.repeat(np.arange(M), deg), g.integers(0, N, deg * M), M, N)


def _factor(spk, dt, n, K, g):
    X = torch.from_numpy(g.standard_normal((n, K)).astype(np.float32)).to(DEV)
    if dt == "e4m3":
        q, s = spk.quantize_e4m3_rows(X)
        return q, s, q.view(torch.uint8).cpu().numpy(), s.cpu().numpy()
    if dt == "f32":
        return X, None, X.cpu().numpy(), None
    q = spk.cast(X, torch.bfloat16 if dt == "bf16" else torch.float16)
    return q, None, q.view(torch.int16).cpu().numpy().view(np.uint16), None


CASES = [(a, b, K) for a, b, Ks in (("f32", "f32", (4, 12, 16, 20, 32, 64, 68, 128, 132, 256)),
                                    ("bf16", "bf16", (8, 32, 40, 64, 128, 136, 256)), ("f16", "f16", (24, 64, 128)),
                                    ("f32", "bf16", (8, 64, 72, 128, 256)), ("f32", "f16", (64, 128)),
                                    ("e4m3", "e4m3", (16, 64, 128, 144, 256))) for K in Ks]


@pytest.mark.parametrize("kind", ["edge", "ones", "twos", "fives"])
@pytest.mark.parametrize("a,b,K", CASES)
def test_widths_and_row_lengths(spk, a, b, K, kind):
    M, N = 290, 240
    rp, ci = _pattern(kind, M, N, K)
    g = np.random.default_rng(K + 1)
    vals = g.uniform(-1, 1, ci.size).astype(np.float32)
    A, sa, An, san = _factor(spk, a, M, K, g)
    B, sb, Bn, sbn = _factor(spk, b, N, K, g)
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    out = spk.sddmm(S, A, B, a_scale=sa, b_scale=sb)
    kw = dict(a_scale=san, b_scale=sbn) if a == "e4m3" else {k: v for k, v in (("fmt_a", a), ("fmt_b", b)) if v != "f32"}
    ref, den = (oracle.sddmm(rp, ci, An, Bn, vals, absmode=m, **kw) for m in (False, True))
    assert comp_err(out.cpu().numpy(), ref, den) <= TOL
    # the register path forms every dot in the same order
    assert torch.equal(out, spk.sddmm(S, A, B, a_scale=sa, b_scale=sb, tune={"variant": 3}))


@pytest.mark.parametrize("mode", ["none", "vals2_only", "both", "shifted"])
def test_value_forms(spk, mode):
    M, N, K = 300, 310, 64
    rp, ci = edge_pattern(M, N, 9, long_row=1100)
    nnz = ci.size
    g = np.random.default_rng(3)
    S = spk.CSR(rp, ci, (M, N), device=DEV, chunk_work=64)
    A, B = (torch.from_numpy(g.standard_normal((n, K)).astype(np.float32)).to(DEV) for n in (M, N))
    v = torch.from_numpy(g.uniform(-1, 1, nnz + 1).astype(np.float32)).to(DEV)
    v1, v2 = v[:nnz].contiguous(), torch.flip(v, (0,))[:nnz].contiguous()
    args = {"none": (None, None), "vals2_only": (None, v2), "both": (v1, v2), "shifted": (v[1:], None)}[mode]
    assert torch.equal(spk.sddmm(S, A, B, *args), spk.sddmm(S, A, B, *args, tune={"variant": 3}))
