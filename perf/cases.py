"""Performance cases: the work that a program hands to this framework.

A case names an operation (``op``), the dtype of its dense factors, a pattern
family with its sizes (``pattern``, ``M``, ``N``, ``nnz``) and the width ``K``:

  step       SDDMM followed by SpMM on the same operands (one iteration of the
             paper's Compute phase)
  spmm_grad  SpMM forward and backward, gradients of B and of the values
  gnn_grad   the graph layer (SDDMM -> SpMM on one H) forward and backward
  attn       FusedMM with row softmax, forward only (serving)
  attn_grad  FusedMM with row softmax, forward and backward
  batch      SDDMM and SpMM of many small matrices in one captured launch
  plan       coordinates -> CSR with its balanced schedule -> transpose plan

Patterns: ``er`` (uniform columns, the same number in nearly every row),
``rmat`` (power-law graph, a, b, c, d = .57, .19, .19, .05) and ``bip``
(bipartite, row and column weights Zipf(1.1) clipped to [1, 20000]).  All have
exactly ``nnz`` distinct entries, sorted by row and column.
"""
import math

import torch

import paper_2404_19638_gb300 as spk

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "e4m3": torch.float8_e4m3fn}
BYTES = {"f32": 4, "bf16": 2, "f16": 2, "e4m3": 1}
BATCH_K = (16, 32, 64)


def listed():
    def case(name, op, dtype, pattern, M, N, nnz, K, heads=1):
        return {"name": name, "op": op, "dtype": dtype, "pattern": pattern, "M": M, "N": N, "nnz": nnz, "K": K,
                "heads": heads}

    return [
        # the smallest call: one small sparse block a step, where launches and latency count
        case("step_tiny_f32", "step", "f32", "er", 4096, 4096, 65536, 32),
        # a power-law graph at its ordinary size, full precision
        case("step_rmat20_f32", "step", "f32", "rmat", 1 << 20, 1 << 20, 16_086_730, 64),
        # the same graph with BF16 factors
        case("step_rmat20_bf16", "step", "bf16", "rmat", 1 << 20, 1 << 20, 16_086_730, 64),
        # recommender: tall user-item matrix, wide embeddings; the largest single step
        case("step_rec_bf16", "step", "bf16", "bip", 2_000_000, 500_000, 50_000_000, 128),
        # recommender scoring on FP8 embeddings with per-row scales
        case("step_rec_e4m3", "step", "e4m3", "bip", 500_000, 125_000, 12_500_000, 128),
        # odd sizes: rectangular, a width that no 16-byte vector divides
        case("step_ragged_f32", "step", "f32", "er", 120_011, 75_503, 2_400_131, 50),
        # one training step of a graph convolution with learned edge weights, a mid-size graph
        case("spmm_grad_f32", "spmm_grad", "f32", "rmat", 200_000, 200_000, 3_100_000, 32),
        # one training step of the graph layer on a large graph, BF16 features
        case("gnn_grad_bf16", "gnn_grad", "bf16", "rmat", 1 << 22, 1 << 22, 33_000_000, 64),
        # one training step of graph attention, 4 heads
        case("attn_grad_f32", "attn_grad", "f32", "rmat", 1 << 20, 1 << 20, 16_086_730, 64, 4),
        # serving graph attention, one head, BF16 features
        case("attn_bf16", "attn", "bf16", "rmat", 1 << 20, 1 << 20, 16_086_730, 64, 1),
        # many uneven matrices (n log-uniform up to M, half er, half rmat, K of 16, 32 or 64) in one launch
        case("batch_f32", "batch", "f32", "mixed", 200_000, 32, 0, 0),
        # a new graph arrives as coordinates: CSR, schedule and transpose plan before the first step
        case("plan_coo", "plan", "f32", "rmat", 1 << 19, 1 << 19, 8_000_000, 1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "spmm_grad", "gnn_grad", "attn", "attn_grad", "batch", "plan"])
    if op == "batch":
        return {"op": op, "dtype": rng.choice(["f32", "bf16"]), "pattern": "mixed", "M": _log(rng, 20_000, 200_000),
                "N": rng.randint(4, 32), "nnz": 0, "K": 0, "heads": 1}
    pattern = rng.choice(["er", "rmat", "bip"] if op in ("step", "plan") else ["er", "rmat"])
    M = _log(rng, 2_000, 2_000_000)
    N = M if op == "gnn_grad" or pattern == "rmat" else min(2_000_000, max(1_000, int(M * rng.uniform(0.25, 2.0))))
    deg = rng.uniform(3.0, 32.0)
    dtype = {"step": rng.choice(["f32", "f32", "bf16", "bf16", "f16", "e4m3"]), "spmm_grad": rng.choice(["f32", "bf16"]),
             "gnn_grad": rng.choice(["f32", "bf16"]), "attn": rng.choice(["f32", "bf16", "f16"]),
             "attn_grad": rng.choice(["f32", "bf16"]), "plan": "f32"}[op]
    heads = 1
    if op == "plan":
        K = 1
    elif op in ("attn", "attn_grad"):
        heads = rng.choice([1, 2, 4])
        K = heads * rng.choice([16, 32, 64] if heads < 4 else [8, 16, 32])
    else:
        K = rng.choice([16, 32, 48, 64, 64, 96, 128, 128, rng.randint(1, 140)])
    most = {"step": 40_000_000, "spmm_grad": 16_000_000, "gnn_grad": 16_000_000, "attn": 16_000_000,
            "attn_grad": 12_000_000, "plan": 16_000_000}[op]
    nnz = max(1, min(int(M * deg), most, M * N // 8, 50_000_000 * 128 // max(K, 1)))
    return {"op": op, "dtype": dtype, "pattern": pattern, "M": M, "N": N, "nnz": nnz, "K": K, "heads": heads}


# ------------------------------------------------------------------ inputs
def _keys(g, pattern, M, N, n, weights):
    """n coordinates row * N + column (repeats among them)."""
    dev = g.device
    if pattern == "er":
        base = torch.arange(n, device=dev) * M // n if n >= M else torch.randint(M, (n,), generator=g, device=dev)
        return base * N + torch.randint(N, (n,), generator=g, device=dev)
    if pattern == "bip":
        def pick(cum, size):
            u = torch.rand(n, generator=g, device=dev, dtype=torch.float64) * cum[-1]
            return torch.searchsorted(cum, u, right=True).clamp_(max=size - 1)
        return pick(weights[0], M) * N + pick(weights[1], N)
    scale = max(1, math.ceil(math.log2(max(M, N))))
    keys, have = [], 0
    while have < n:
        m = n - have if M == N == 1 << scale else int((n - have) * 1.3) + 1024
        r = torch.zeros(m, dtype=torch.int32, device=dev)
        c = torch.zeros(m, dtype=torch.int32, device=dev)
        for level in range(scale):
            u = torch.rand(m, generator=g, device=dev)
            bit = 1 << (scale - 1 - level)
            r += (u >= 0.76).int() * bit
            c += (((u >= 0.57) & (u < 0.76)) | (u >= 0.95)).int() * bit
        ok = (r < M) & (c < N)
        k = (r.long() * N + c)[ok][: n - have]
        keys.append(k)
        have += k.numel()
    return torch.cat(keys)


def _pattern(g, pattern, M, N, nnz):
    """(rows, cols) of exactly nnz distinct entries, sorted by row and column."""
    weights = None
    if pattern == "bip":
        weights = [torch.rand(size, generator=g, device=g.device, dtype=torch.float64).pow(-10.0).floor()
                   .clamp(1, 20_000).cumsum(0) for size in (M, N)]
    keys = torch.unique(_keys(g, pattern, M, N, nnz, weights))
    while keys.numel() < nnz:
        more = int((nnz - keys.numel()) * 1.25) + 1024
        keys = torch.unique(torch.cat([keys, _keys(g, "rmat" if pattern == "rmat" else pattern, M, N, more, weights)]))
    if keys.numel() > nnz:
        drop = torch.randperm(keys.numel(), generator=g, device=g.device)[: keys.numel() - nnz]
        keep = torch.ones(keys.numel(), dtype=torch.bool, device=g.device)
        keep[drop] = False
        keys = keys[keep]
    rows = torch.div(keys, N, rounding_mode="floor")
    return rows, keys - rows * N


def _rowptr(rows, M):
    ptr = torch.zeros(M + 1, dtype=torch.int64, device=rows.device)
    torch.cumsum(torch.bincount(rows, minlength=M), 0, out=ptr[1:])
    return ptr.int()


def _normal(g, shape, std=1.0):
    return torch.randn(shape, generator=g, device=g.device) * std


def _values(g, n):
    return torch.rand(n, generator=g, device=g.device) * 2 - 1


def _e4m3(X):
    """Per-row FP8 codes and scales (amax / 448)."""
    amax = X.abs().amax(dim=1)
    scale = torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))
    return (X / scale[:, None]).clamp(-448.0, 448.0).to(torch.float8_e4m3fn), scale


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + 17)


def _batch_sizes(case):
    """n, K, nonzeros a row and pattern of each matrix: n log-uniform in [1000, M], the first half er with 4..32 a row."""
    count = case["N"]
    for m in range(count):
        u, v = (m * 0.6180339887 + 0.13) % 1.0, (m * 0.7548776662 + 0.37) % 1.0
        er = m < count // 2
        yield int(1000 * (case["M"] / 1000) ** u), BATCH_K[int(3 * v)], 4 + int(29 * (1.0 - v)) if er else 15, "er" if er else "rmat"


def _batch_inputs(case, seed):
    """The matrices of a batch: rows, cols, n, values, A, B each."""
    g = _generator(seed)
    out = []
    for n, K, deg, pattern in _batch_sizes(case):
        rows, cols = _pattern(g, pattern, n, n, n * deg)
        A, B = (_normal(g, (n, K)).to(DTYPES[case["dtype"]]) for _ in range(2))
        out.append((rows, cols, n, _values(g, rows.numel()), A, B))
    return out


def _inputs(case, seed):
    """Everything a pass reads, as plain tensors."""
    g = _generator(seed)
    op, M, N, K, dt = case["op"], case["M"], case["N"], case["K"], DTYPES[case["dtype"]]
    rows, cols = _pattern(g, case["pattern"], M, N, case["nnz"])
    x = {"rows": rows, "cols": cols}
    if op == "plan":                                   # unordered, a twentieth of the coordinates twice
        n = rows.numel()
        twice = torch.randperm(n, generator=g, device=g.device)[: n // 20]
        x["order"] = torch.cat([torch.arange(n, device=g.device), twice])[
            torch.randperm(n + n // 20, generator=g, device=g.device)]
        x["vals"] = _values(g, n + n // 20)
        return x
    x["vals"] = None if op in ("gnn_grad", "attn", "attn_grad") else (
        torch.randint(1, 6, (rows.numel(),), generator=g, device=g.device).float() if case["pattern"] == "bip"
        else _values(g, rows.numel()))
    if op == "gnn_grad":
        x["A"] = x["B"] = _normal(g, (N, K), 0.1).to(dt)
    elif case["dtype"] == "e4m3":
        x["A"], x["a_scale"] = _e4m3(_normal(g, (M, K)))
        x["B"], x["b_scale"] = _e4m3(_normal(g, (N, K)))
    else:
        if op != "spmm_grad":
            x["A"] = _normal(g, (M, K)).to(dt)
        x["B"] = _normal(g, (N, K)).to(dt)
    if op.endswith("_grad"):
        x["dY"] = _normal(g, (M, K))
    return x


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        items, outs = [], []
        for rows, cols, n, vals, A, B in _batch_inputs(case, seed):
            S = spk.CSR(_rowptr(rows, n), cols.int(), (n, n), vals)
            e = torch.empty(S.nnz, dtype=torch.float32, device=S.device)
            C = torch.empty((n, B.size(1)), dtype=torch.float32, device=S.device)
            items += [spk.Item(spk.OP_SDDMM, S, B, e, A=A), spk.Item(spk.OP_SPMM, S, B, C)]
            outs += [e, C]
        batch = spk.Batch(items)
        batch.capture()
        return {"op": op, "batch": batch, "outs": outs}
    x = _inputs(case, seed)
    if op == "plan":
        order = x["order"]
        return {"op": op, "rows": x["rows"][order].int(), "cols": x["cols"][order].int(), "vals": x["vals"],
                "shape": (case["M"], case["N"])}
    S = spk.CSR(_rowptr(x["rows"], case["M"]), x["cols"].int(), (case["M"], case["N"]), x["vals"])
    if op.endswith("_grad"):
        S.transpose_plan()
    state = {"op": op, "S": S, "heads": case["heads"], "scale": 1.0 / math.sqrt(case["K"] / case["heads"])}
    for name in ("A", "B", "a_scale", "b_scale", "dY"):
        state[name] = x.get(name)
    if op == "spmm_grad":
        state["vals"] = x["vals"].requires_grad_()
        state["B"].requires_grad_()
    elif op == "gnn_grad":
        state["B"].requires_grad_()
    elif op == "attn_grad":
        state["A"].requires_grad_()
        state["B"].requires_grad_()
    return state


def run(state):
    op = state["op"]
    if op == "batch":
        state["batch"].replay()
        return state["outs"]
    if op == "plan":
        S = spk.CSR.from_coo(state["rows"], state["cols"], state["shape"], state["vals"])
        return [S.rowptr, S.colidx, S.vals, *S.transpose_plan().arrays()]
    S, A, B = state["S"], state["A"], state["B"]
    if op == "step":
        return {"sddmm": spk.sddmm(S, A, B, a_scale=state["a_scale"], b_scale=state["b_scale"]),
                "spmm": spk.spmm(S, B, b_scale=state["b_scale"])}
    if op == "attn":
        return spk.fusedmm(S, A, B, heads=state["heads"], scale=state["scale"], softmax=True)[0]
    if op == "spmm_grad":
        Y = spk.autograd.spmm(S, B, state["vals"])
        dB, dvals = torch.autograd.grad(Y, [B, state["vals"]], state["dY"])
        return {"Y": Y.detach(), "dB": dB, "dvals": dvals}
    if op == "gnn_grad":
        Y = spk.autograd.gnn_layer(S, B)
        return {"Y": Y.detach(), "dH": torch.autograd.grad(Y, B, state["dY"])[0]}
    Y = spk.autograd.fusedmm(S, A, B, heads=state["heads"], scale=state["scale"], softmax=True)
    dA, dB = torch.autograd.grad(Y, [A, B], state["dY"])
    return {"Y": Y.detach(), "dA": dA, "dB": dB}


# ------------------------------------------------------------------ work
def _pair_work(M, N, nnz, K, elt):
    pattern = 4 * (M + 1) + 8 * nnz                    # row pointers, columns, values
    scales = 4 * (M + N) if elt == 1 else 0
    sddmm = pattern + 4 * nnz + (M + N) * K * elt + scales
    spmm = pattern + N * K * elt + 4 * M * K + scales
    return sddmm + spmm, 4 * nnz * K


def work(case):
    op, M, N, nnz, K = case["op"], case["M"], case["N"], case["nnz"], case["K"]
    elt = BYTES[case["dtype"]]
    pattern = 4 * (M + 1) + 4 * nnz
    if op == "step":
        b, f = _pair_work(M, N, nnz, K, elt)
    elif op == "batch":
        each = [_pair_work(n, n, n * deg, k, elt) for n, k, deg, _ in _batch_sizes(case)]
        b, f = sum(w[0] for w in each), sum(w[1] for w in each)
    elif op == "plan":                                 # coordinates in; CSR, values, transpose plan out
        b, f = 12 * (nnz + nnz // 20) + 4 * (M + 1) + 8 * nnz + 4 * (N + 1) + 8 * nnz, 0
    elif op == "attn":
        b, f = pattern + (M + N) * K * elt + 4 * M * K, 4 * nnz * K
    elif op == "spmm_grad":                            # values, B, dY in; Y, dB, dvalues out
        b, f = pattern + 8 * nnz + 2 * N * K * elt + 8 * M * K, 6 * nnz * K
    elif op == "gnn_grad":                             # H, dY in; Y, dH out
        b, f = pattern + 2 * N * K * elt + 8 * M * K, 12 * nnz * K
    else:                                              # A, B, dY in; Y, dA, dB out
        b, f = pattern + 2 * (M + N) * K * elt + 8 * M * K, 12 * nnz * K
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit results
def _sddmm64(rows, cols, A, B):
    out = torch.empty(rows.numel(), dtype=torch.float64, device=rows.device)
    step = max(1, (1 << 28) // A.size(1))
    for i in range(0, rows.numel(), step):
        out[i:i + step] = (A[rows[i:i + step]] * B[cols[i:i + step]]).sum(1)
    return out


def _spmm64(rows, cols, vals, shape, B):
    """C = S B; rows need not be sorted."""
    out = torch.zeros((shape[0], B.size(1)), dtype=torch.float64, device=B.device)
    step = max(1, (1 << 28) // B.size(1))
    for i in range(0, rows.numel(), step):
        out.index_add_(0, rows[i:i + step], B[cols[i:i + step]] * vals[i:i + step, None])
    return out


def exact(case, seed):
    op, M, N, heads = case["op"], case["M"], case["N"], case["heads"]
    if op == "batch":
        out = []
        for rows, cols, n, vals, A, B in _batch_inputs(case, seed):
            A, B, v = A.double(), B.double(), vals.double()
            out += [_sddmm64(rows, cols, A, B) * v, _spmm64(rows, cols, v, (n, n), B)]
        return out
    x = _inputs(case, seed)
    if op == "plan":                                   # whole numbers and copied values
        return None
    rows, cols = x["rows"], x["cols"]
    v = torch.ones(rows.numel(), dtype=torch.float64, device=rows.device) if x["vals"] is None else x["vals"].double()
    A = x["A"].double() if "A" in x else None
    B = x["B"].double()
    if "a_scale" in x:
        A, B = A * x["a_scale"].double()[:, None], B * x["b_scale"].double()[:, None]
    if op == "step":
        return {"sddmm": _sddmm64(rows, cols, A, B) * v, "spmm": _spmm64(rows, cols, v, (M, N), B)}
    dY = x["dY"].double() if "dY" in x else None
    if op == "spmm_grad":
        return {"Y": _spmm64(rows, cols, v, (M, N), B), "dB": _spmm64(cols, rows, v, (N, M), dY),
                "dvals": _sddmm64(rows, cols, dY, B)}
    if op == "gnn_grad":
        e = _sddmm64(rows, cols, B, B)
        dE = _sddmm64(rows, cols, dY, B)
        dH = _spmm64(rows, cols, dE, (M, N), B) + _spmm64(cols, rows, dE, (N, M), B) + _spmm64(cols, rows, e, (N, M), dY)
        return {"Y": _spmm64(rows, cols, e, (M, N), B), "dH": dH}
    Kh = case["K"] // heads
    scale = 1.0 / math.sqrt(Kh)
    Y, dA, dB = (torch.zeros((n, case["K"]), dtype=torch.float64, device=rows.device) for n in (M, M, N))
    for h in range(heads):
        s = slice(h * Kh, (h + 1) * Kh)
        e = _sddmm64(rows, cols, A[:, s], B[:, s]) * scale
        top = torch.full((M,), -math.inf, dtype=torch.float64, device=rows.device)
        top.scatter_reduce_(0, rows, e, "amax")
        w = torch.exp(e - top[rows])
        w /= torch.zeros(M, dtype=torch.float64, device=rows.device).index_add_(0, rows, w)[rows]
        Y[:, s] = _spmm64(rows, cols, w, (M, N), B[:, s])
        if op == "attn":
            continue
        dw = _sddmm64(rows, cols, dY[:, s], B[:, s])
        dot = torch.zeros(M, dtype=torch.float64, device=rows.device).index_add_(0, rows, w * dw)
        c = scale * w * (dw - dot[rows])
        dA[:, s] = _spmm64(rows, cols, c, (M, N), B[:, s])
        dB[:, s] = _spmm64(cols, rows, c, (N, M), A[:, s]) + _spmm64(cols, rows, w, (N, M), dY[:, s])
    return Y if op == "attn" else {"Y": Y, "dA": dA, "dB": dB}
