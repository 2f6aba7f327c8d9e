"""FusedMM row softmax with masked entries: values of -inf, or the lowest float,
make scores of -inf, which weigh nothing wherever they stand in a row."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"
# Scores are sums of 16 to 64 products of factors in [0.3, 0.6): above 1 (times the lowest float: -inf), at most 23, off by at most
# 64 * 2^-24 * 23 = 9e-5 and its double where two are subtracted; 2e-4 relative in the weights, as much in Y (below 0.6) and lse.
ATOL = 2e-4


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


def _rows():
    """Lengths and masked entries: runs of masked entries at the start, the end and in the middle of short, long
    and split rows, all of a row, none, and random halves."""
    rng = np.random.default_rng(5)
    masks = []
    for n in [1, 2, 3, 5, 8, 15, 16, 17, 31, 32, 33, 40, 64, 300, 700]:
        for k in range(6):
            m = np.zeros(n, bool)
            if k < 4:
                m[(slice(0, n // 2 + 1), slice(n // 2, n), slice(0, n), slice(0, n - 1))[k]] = True
            elif k == 4:
                m = rng.random(n) < 0.5
            masks.append(m)
    return [masks[i] for i in rng.permutation(len(masks))]


@pytest.mark.parametrize("fill", [-np.inf, np.finfo(np.float32).min])
@pytest.mark.parametrize("dt,heads,tune", [
    (torch.float32, 1, None), (torch.float32, 4, None), (torch.bfloat16, 1, None), (torch.bfloat16, 2, None),
    (torch.float32, 1, {"group_lanes": 8, "vecs_per_lane": 2, "unroll": 4}), (torch.float32, 2, {"vecs_per_lane": 1})])
def test_masked_entries_weigh_nothing(spk, dt, heads, tune, fill):
    K, N, masks = 64, 900, _rows()
    M = len(masks)
    rng = np.random.default_rng(K + heads)
    rp = np.cumsum([0] + [m.size for m in masks]).astype(np.int32)
    ci = np.concatenate([np.sort(rng.choice(N, m.size, replace=False)) for m in masks]).astype(np.int32)
    vals = np.where(np.concatenate(masks), fill, 1.0).astype(np.float32)
    A, B = (torch.from_numpy(rng.uniform(0.3, 0.6, (n, K)).astype(np.float32)).to(dt) for n in (M, N))
    S = spk.CSR(rp, ci, (M, N), torch.from_numpy(vals), device=DEV, chunk_work=96)
    Y, _, lse = spk.fusedmm(S, A.to(DEV), B.to(DEV), heads=heads, softmax=True, want_lse=True, tune=tune)
    Y, lse, Kh = Y.cpu().double(), lse.cpu().double(), K // heads
    for r, m in enumerate(masks):
        cols = torch.from_numpy(ci[rp[r]:rp[r + 1]]).long()
        keep = cols[~torch.from_numpy(m)]
        for h in range(heads):
            a, b = A[r, h * Kh:(h + 1) * Kh].double(), B[keep, h * Kh:(h + 1) * Kh].double()
            y = Y[r, h * Kh:(h + 1) * Kh]
            if keep.numel() == 0:
                assert not y.any() and lse[r, h] == -np.inf
                continue
            e = b @ a
            assert abs(lse[r, h] - torch.logsumexp(e, 0)) <= ATOL
            assert (y - torch.softmax(e, 0) @ b).abs().max() <= ATOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("tune", [None, {"group_lanes": 8, "vecs_per_lane": 2, "unroll": 4}, {"vecs_per_lane": 1}])
def test_rows_with_a_nan_or_infinite_score_are_zeros(spk, bad, tune):
    """Such a row has no softmax: zeros, with an lse of -inf, in short, long and split rows; the others are untouched."""
    K, N, lens = 64, 900, [1, 5, 16, 40, 300, 700] * 2
    rng = np.random.default_rng(1)
    rp = np.cumsum([0] + lens).astype(np.int32)
    ci = np.concatenate([np.sort(rng.choice(N, n, replace=False)) for n in lens]).astype(np.int32)
    A, B = (torch.from_numpy(rng.uniform(0.3, 0.6, (n, K)).astype(np.float32)).to(DEV) for n in (len(lens), N))
    vals = np.ones(ci.size, np.float32)
    run = lambda: spk.fusedmm(spk.CSR(rp, ci, (len(lens), N), torch.from_numpy(vals), device=DEV, chunk_work=96), A, B,
                              softmax=True, want_lse=True, tune=tune)
    Y0, _, l0 = run()
    for r in range(6):
        vals[rp[r] + rng.integers(lens[r])] = bad
    Y, _, lse = run()
    assert not Y[:6].any() and (lse[:6] == -np.inf).all()
    assert torch.equal(Y[6:], Y0[6:]) and torch.equal(lse[6:], l0[6:])
