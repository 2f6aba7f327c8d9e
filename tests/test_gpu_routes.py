"""Which calls reach which kernel: sizes at the limits of the one-warp-per-chunk
kernels, where another route answers."""
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


@pytest.mark.parametrize("K", [65535 * 128, 65535 * 128 + 4])
def test_spmm_rows_around_the_grid_limit(spk, K):
    """65,535 K blocks of 512 bytes, and one vector more.  One entry a row: exactly the product."""
    rp, ci = np.array([0, 1, 1, 2], np.int32), np.array([1, 0], np.int32)
    v = torch.tensor([0.75, -3.0], device=DEV)
    S = spk.CSR(rp, ci, (3, 2), v, device=DEV)
    g = torch.Generator(device=DEV).manual_seed(0)
    B = torch.randn(2, K, generator=g, device=DEV)
    C = spk.spmm(S, B)
    assert torch.equal(C[0], v[0] * B[1]) and torch.equal(C[2], v[1] * B[0]) and not C[1].any()
    X = spk.spmm_t(S, C)
    assert torch.equal(X[1], v[0] * C[0]) and torch.equal(X[0], v[1] * C[2])


@pytest.mark.parametrize("dt,K", [(torch.float32, 18), (torch.float32, 50), (torch.float32, 64), (torch.bfloat16, 50)])
def test_default_tune_runs_the_default_kernel(spk, dt, K):
    """A tune from tune_default, or one that names a compiled shape the kernel has no use for, gives the bits of
    the call without a tune.  (The element path adds a dot's products in another order than the warp kernel.)"""
    g = torch.Generator(device=DEV).manual_seed(K)
    M, N, nnz = 900, 700, 12_000
    rows = torch.randint(M, (nnz,), generator=g, device=DEV).int()
    cols = torch.randint(N, (nnz,), generator=g, device=DEV).int()
    S = spk.CSR.from_coo(rows, cols, (M, N), torch.rand(nnz, generator=g, device=DEV))
    A, B = (torch.randn(n, K, generator=g, device=DEV).to(dt) for n in (M, N))
    code = 0 if dt == torch.float32 else 1
    e, C, X = spk.sddmm(S, A, B), spk.spmm(S, B), spk.spmm_t(S, A)
    assert torch.equal(e, spk.sddmm(S, A, B, tune=S.tune_default(0, code, K)))
    assert torch.equal(C, spk.spmm(S, B, tune=S.tune_default(1, code, K)))
    assert torch.equal(X, spk.spmm_t(S, A, tune=S.tune_default(2, code, K)))
    if K % 4:
        assert torch.equal(e, spk.sddmm(S, A, B, tune={"variant": 2, "group_lanes": 16, "vecs_per_lane": 1, "unroll": 4}))


def _skewed(spk, M, nnz, seed=0):
    """Few rows and columns with many entries (u^3 draws), split rows among them."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rows, cols = ((torch.rand(nnz, generator=g, device=DEV) ** 3 * M).int().clamp_(max=M - 1) for _ in range(2))
    return spk.CSR.from_coo(rows, cols, (M, M), torch.rand(nnz, generator=g, device=DEV))


def _time(fn, n=8):
    fn()
    best = float("inf")
    for _ in range(5):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        for _ in range(n):
            fn()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("dt,K", [(torch.float32, 66), (torch.float32, 99), (torch.float32, 257), (torch.bfloat16, 130)])
def test_wide_ragged_rows_are_no_slower_than_the_element_path(spk, dt, K):
    """Rows of many 4- or 8-byte parts on a large skewed pattern (variant 3 is the element path): the small copies
    took 1.8 to 3.3 times its time there."""
    S = _skewed(spk, 1 << 17, 3_000_000)
    B = torch.randn(S.N, K, device=DEV).to(dt)
    assert _time(lambda: spk.spmm(S, B)) <= 1.25 * _time(lambda: spk.spmm(S, B, tune={"variant": 3}))


@pytest.mark.parametrize("nnz,same", [(20_000, False), (1_000_000, True)])
def test_wide_odd_sddmm_changes_path_with_the_size(spk, nnz, same):
    """FP32 rows of 65 elements: small copies up to 2^19 entries, the element path (another order of adding) above."""
    S = _skewed(spk, 1 << 14, nnz)
    A, B = (torch.randn(S.M, 65, device=DEV) for _ in range(2))
    e, r = spk.sddmm(S, A, B), spk.sddmm(S, A, B, tune={"variant": 3})
    assert torch.equal(e, r) == same
    torch.testing.assert_close(e, r, rtol=1e-4, atol=1e-4)


def test_spmm_t_on_large_patterns_is_no_slower_than_permuted_values(spk):
    """8M entries of uniform columns, values and rows of Y larger than L2: against the values gathered into CSC order
    first and an SpMM on the transposed pattern (the gather inside the SpMM took 1.5 times as long)."""
    M, d, K = 333_000, 24, 64
    g = torch.Generator(device=DEV).manual_seed(3)
    rp = (torch.arange(M + 1, device=DEV) * d).int()
    ci = torch.randint(M, (M * d,), generator=g, device=DEV).int()
    v = torch.rand(M * d, generator=g, device=DEV)
    S = spk.CSR(rp, ci, (M, M), v)
    colptr, rowidx, perm = (t.clone() for t in S.transpose_plan().arrays())
    T = spk.CSR(colptr, rowidx, (M, M))
    Y = torch.randn(M, K, device=DEV)
    p = perm.long()
    assert torch.equal(spk.spmm_t(S, Y), spk.spmm(T, Y, v[p]))
    assert _time(lambda: spk.spmm_t(S, Y)) <= 1.15 * _time(lambda: spk.spmm(T, Y, v[p]))


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("tune", [None, {"group_lanes": 8, "vecs_per_lane": 1, "unroll": 8}])
def test_batch_runs_six_ctas_an_sm(spk, dt, tune):
    """Neither BF16 operands nor a shape named for SpMM (one routine per row width) cost resident warps."""
    S = _skewed(spk, 3000, 40_000)
    B = torch.randn(S.N, 32, device=DEV).to(dt)
    out = torch.empty(S.M, 32, device=DEV)
    b = spk.Batch([spk.Item(spk.OP_SPMM, S, B, out, tune=tune)])
    b.run()
    assert torch.equal(out, spk.spmm(S, B))
    default = b.info()
    b.set_registers(80)
    assert b.info() == default
    b.set_registers(96)
    assert b.info()["ctas"] < default["ctas"]


@pytest.mark.parametrize("odt", [torch.bfloat16, torch.float16])
def test_empty_rows_of_16_bit_outputs(spk, odt):
    """4M rows with 1M entries: rows without entries are written as fast in 16 bits as in FP32 (1.65 times that
    when the output type was looked up at every row, 1.2 without)."""
    g = torch.Generator(device=DEV).manual_seed(1)
    M, N, n, K = 4_000_000, 200_000, 1_000_000, 16
    rows = torch.sort(torch.randint(M, (n,), generator=g, device=DEV)).values
    rp = torch.searchsorted(rows, torch.arange(M + 1, device=DEV)).int()
    S = spk.CSR(rp, torch.randint(N, (n,), generator=g, device=DEV).int(), (M, N))
    B = torch.randn(N, K, generator=g, device=DEV)
    C, H = torch.empty(M, K, device=DEV), torch.full((M, K), float("nan"), device=DEV, dtype=odt)
    full = _time(lambda: spk.spmm(S, B, out=C))
    assert _time(lambda: spk.spmm(S, B, out=H)) <= 1.4 * full
    assert torch.equal(H, C.to(odt))


def _rows_of(spk, M, d, seed=3):
    """M rows of exactly d entries, uniform columns."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rp = (torch.arange(M + 1, device=DEV) * d).int()
    ci = torch.randint(M, (M * d,), generator=g, device=DEV).int()
    return spk.CSR(rp, ci, (M, M), torch.rand(M * d, generator=g, device=DEV))


@pytest.mark.parametrize("K", [4, 12, 16])
def test_narrow_rows_on_regular_patterns(spk, K):
    """FP32 rows of up to 64 bytes, 8M entries, 24 a row: as fast as the row-split kernel (the warp kernel took twice
    its time), and the bits of the balanced register path in every form that a call can have."""
    S = _rows_of(spk, 333_000, 24)
    wide = torch.randn(S.N, K + 4, device=DEV)
    B, v2, reg = wide[:, :K], torch.rand(S.nnz, device=DEV), {"variant": 3}
    assert torch.equal(spk.spmm(S, B), spk.spmm(S, B, tune=reg))
    assert torch.equal(spk.spmm(S, B, vals2=v2), spk.spmm(S, B, vals2=v2, tune=reg))
    assert torch.equal(spk.spmm(S, B, out_dtype=torch.bfloat16), spk.spmm(S, B, out_dtype=torch.bfloat16, tune=reg))
    C, D = torch.ones(S.M, K, device=DEV), torch.ones(S.M, K, device=DEV)
    spk.spmm(S, B, out=C, accumulate=True)
    spk.spmm(S, B, out=D, accumulate=True, tune=reg)
    assert torch.equal(C, D)
    assert _time(lambda: spk.spmm(S, B)) <= 1.25 * _time(lambda: spk.spmm(S, B, tune={"variant": 1}))


def test_fusedmm_on_regular_and_random_rows(spk):
    """One head, FP32, K = 64, 24 entries a row: with rows of one length the lane groups keep in step and run (the warp
    kernel took 1.2 to 1.3 times as long), with random lengths the warp kernel does."""
    lanes, K = {"group_lanes": 8, "vecs_per_lane": 2, "unroll": 4}, 64
    S = _rows_of(spk, 333_000, 24)
    A, B = (0.2 * torch.randn(S.M, K, device=DEV) for _ in range(2))
    f = lambda S, tune=None: spk.fusedmm(S, A, B, softmax=True, want_lse=True, tune=tune)
    for x, y in zip(f(S), f(S, lanes)):
        assert x is y is None or torch.equal(x, y)
    assert _time(lambda: f(S)) <= 1.1 * _time(lambda: f(S, lanes))
    g = torch.Generator(device=DEV).manual_seed(5)
    rows, cols = (torch.randint(S.M, (S.nnz,), generator=g, device=DEV).int() for _ in range(2))
    R = spk.CSR.from_coo(rows, cols, (S.M, S.M), torch.rand(S.nnz, generator=g, device=DEV))
    for x, y in zip(f(R), f(R, lanes)):
        if x is not None:
            torch.testing.assert_close(x, y, rtol=2e-4, atol=2e-5)
    assert _time(lambda: f(R)) <= _time(lambda: f(R, lanes))


def test_spmm_t_with_two_value_arrays(spk):
    """2.5M entries, 25 a row, FP32 K = 64: a second array doubles what competes with the rows for L2 when both are
    gathered through the permutation (1.6 times the time of one array); put in order first they take 1.37 times."""
    g = torch.Generator(device=DEV).manual_seed(3)
    M, N, d, K = 100_000, 20_000, 25, 64
    rp = (torch.arange(M + 1, device=DEV) * d).int()
    ci = torch.randint(N, (M * d,), generator=g, device=DEV).int()
    S = spk.CSR(rp, ci, (M, N))
    v, w = (torch.rand(M * d, generator=g, device=DEV) for _ in range(2))
    vw, Y = v * w, torch.randn(M, K, device=DEV)
    assert torch.equal(spk.spmm_t(S, Y, v, w), spk.spmm_t(S, Y, vw))
    assert _time(lambda: spk.spmm_t(S, Y, v, w)) <= 1.5 * _time(lambda: spk.spmm_t(S, Y, vw))
