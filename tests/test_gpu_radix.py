"""Coordinates -> CSR -> transpose plan at the sizes where the radix sort's tiles
end (4096 pairs a tile, 512 a warp), for digits that are all equal, all
different or skewed, against NumPy's stable sorts."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def spk():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2404_19638_gb300 as m
    return m


@pytest.mark.parametrize("nnz", [1, 31, 33, 511, 513, 4095, 4096, 4097, 12289])
@pytest.mark.parametrize("M,N,kind", [(1, 1, "flat"), (300, 1, "flat"), (1, 70000, "flat"), (5000, 70000, "flat"),
                                       (70000, 257, "skew"), (1 << 17, 1 << 17, "one"), (900, 1 << 24, "flat")])
def test_orders(spk, nnz, M, N, kind):
    g = np.random.default_rng(nnz + M)
    def draw(n):
        if kind == "one":
            return np.full(nnz, n - 1)
        return g.integers(0, n, nnz) if kind == "flat" else np.minimum(g.zipf(1.3, nnz) - 1, n - 1)
    r, c = draw(M).astype(np.int32), draw(N).astype(np.int32)
    v = g.standard_normal(nnz).astype(np.float32)
    S = spk.CSR.from_coo(torch.from_numpy(r).to(DEV), torch.from_numpy(c).to(DEV), (M, N), torch.from_numpy(v).to(DEV))
    order = np.lexsort((np.arange(nnz), c, r))
    keep = np.ones(nnz, bool)
    keep[1:] = (r[order][1:] != r[order][:-1]) | (c[order][1:] != c[order][:-1])
    order = order[keep]
    ci, rows = c[order], r[order]
    rp = np.searchsorted(rows, np.arange(M + 1))
    assert np.array_equal(S.rowptr.cpu().numpy(), rp) and np.array_equal(S.colidx.cpu().numpy(), ci)
    assert np.array_equal(S.vals.cpu().numpy(), v[order])
    colptr, rowidx, perm = (x.cpu().numpy() for x in S.transpose_plan().arrays())
    p = np.argsort(ci, kind="stable")
    assert np.array_equal(perm[:p.size], p) and np.array_equal(rowidx[:p.size], rows[p])
    assert np.array_equal(colptr, np.searchsorted(ci[p], np.arange(N + 1)))
