"""Performance cases: what a user of this library has it do, through the public entry points.

A case is one call, or one short sequence of calls, that a program makes again
and again on objects that it keeps (a permuted handle, a batch, a server), or,
for the two preprocessing cases, the calls that it makes once per matrix:

  spmv     y = A x, in the original or the permuted space, on a handle that the
           library tuned (autotune=True), as the bench and the server make them
  spmm     Y = A X with k right-hand sides, rows of X and Y padded to 16 bytes
           (as the header advises) or not
  batch    one batched run over many uneven matrices, each with its own k
  serve    a trace of SpMV, SpMM and power-iteration requests through Server.run
  power    20 steps of power iteration with the Rayleigh quotient of every step
  prep     both random permutations and the permuted CSR of a new matrix
  entropy  the block-grid entropy of a handle and its hierarchical map

Matrices are the library's own synthetic workloads: block-diagonal (4096 rows,
FP64), power-law rows clustered near the diagonal (2^20 rows), the 5-point
Laplacian (up to 4096 x 4096 grid points), Poisson rows with uniform columns
(the batched and served sets).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_00106_gb300 import maxe, serve
from paper_2308_00106_gb300 import workloads as W

VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
VECTOR_BYTES = {"f64": 8, "f32": 4, "bf16": 4}
VECTOR = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}
ZIPF_S, ZIPF_CAP = 1.5, 1000
POWER_STEPS = 20


def listed():
    return [
        # the smallest call: one FP64 product of the 4096-row block-diagonal matrix in the original
        # space, the inner step of a user's own solver on a small system
        {"name": "spmv_blockdiag_4k_f64", "kind": "spmv", "matrix": "blockdiag", "n": 4096, "lam": 0.0,
         "dtype": "f64", "order": "rc", "space": "original"},
        # the headline: iterative use of a permuted power-law matrix, vectors kept in the permuted space
        {"name": "spmv_powerlaw_1m_f32", "kind": "spmv", "matrix": "powerlaw", "n": 1 << 20, "lam": 0.0,
         "dtype": "f32", "order": "rc", "space": "permuted"},
        # the whole method in the paper's precision: x permuted, product, y scattered back
        {"name": "spmv_powerlaw_1m_f64_orig", "kind": "spmv", "matrix": "powerlaw", "n": 1 << 20, "lam": 0.0,
         "dtype": "f64", "order": "rc", "space": "original"},
        # the largest single product: the 16.8M-row stencil after its rows and columns were permuted
        {"name": "spmv_laplacian_4096_f32", "kind": "spmv", "matrix": "laplacian", "n": 4096, "lam": 0.0,
         "dtype": "f32", "order": "rc", "space": "permuted"},
        # a block of right-hand sides on the stencil in natural order (the plain handle)
        {"name": "spmm_laplacian_2048_f32_k16", "kind": "spmm", "matrix": "laplacian", "n": 2048, "lam": 0.0,
         "dtype": "f32", "order": "natural", "space": "permuted", "k": 16, "pad": True},
        # BF16 values, four right-hand sides, the permuted stencil called in the original space
        {"name": "spmm_laplacian_2048_bf16_k4", "kind": "spmm", "matrix": "laplacian", "n": 2048, "lam": 0.0,
         "dtype": "bf16", "order": "rc", "space": "original", "k": 4, "pad": True},
        # odd sizes: a k that is no multiple of the vector width in plain contiguous tensors
        {"name": "spmm_poisson_100003_f32_k7", "kind": "spmm", "matrix": "poisson", "n": 100_003, "lam": 20.0,
         "dtype": "f32", "order": "rc", "space": "permuted", "k": 7, "pad": False},
        # the batched workload: 256 uneven matrices, 1 to 16 right-hand sides each, one run
        {"name": "batch_256_f32", "kind": "batch", "count": 256, "rows_lo": 1000, "rows_hi": 200_000, "kmax": 16,
         "dtype": "f32"},
        # a burst of requests to a server of resident matrices (half FP32, half BF16 values)
        {"name": "serve_12", "kind": "serve", "count": 12, "rows_lo": 10_000, "rows_hi": 600_000, "requests": 24,
         "kmax": 32},
        # power iteration on one served matrix
        {"name": "power_300k_f32", "kind": "power", "n": 300_007, "lam": 20.0, "dtype": "f32"},
        # preprocessing of a new matrix: the cost that reuse has to pay back
        {"name": "prep_powerlaw_1m_f32", "kind": "prep", "matrix": "powerlaw", "n": 1 << 20, "lam": 0.0,
         "dtype": "f32", "cols": True},
        # scoring a permutation: the 64 x 64 grid entropy and its 8 x 8 hierarchical map
        {"name": "entropy_powerlaw_1m", "kind": "entropy", "matrix": "powerlaw", "n": 1 << 20, "lam": 0.0,
         "dtype": "f32", "order": "rc", "grid": 64, "levels": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, kinds, most_nnz=48_000_000):
    m = rng.choice(kinds)
    if m == "blockdiag":
        return {"matrix": m, "n": 16 * _log_int(rng, 64, 256), "lam": 0.0}
    if m == "powerlaw":
        return {"matrix": m, "n": _log_int(rng, 20_000, 1 << 20), "lam": 0.0}
    if m == "laplacian":
        return {"matrix": m, "n": _log_int(rng, 60, min(3000, int(math.sqrt(most_nnz / 5)))), "lam": 0.0}
    n = _log_int(rng, 1000, min(3_000_000, most_nnz // 8))
    lam = round(rng.uniform(5.0, min(50.0, most_nnz / n)), 3)
    return {"matrix": m, "n": n, "lam": lam}


def draw(rng):
    kind = rng.choice(["spmv", "spmv", "spmv", "spmm", "spmm", "batch", "serve", "power", "prep", "entropy"])
    dtype = rng.choice(["f64", "f32", "bf16"])
    order = rng.choice(["rc", "rc", "natural"])
    if kind == "spmv":
        m = _draw_matrix(rng, ["blockdiag", "powerlaw", "laplacian", "poisson"])
        return {"kind": kind, **m, "dtype": dtype, "order": order, "space": rng.choice(["original", "permuted"])}
    if kind == "spmm":
        m = _draw_matrix(rng, ["laplacian", "poisson"], most_nnz=12_000_000)
        return {"kind": kind, **m, "dtype": dtype, "order": order, "space": rng.choice(["original", "permuted"]),
                "k": _log_int(rng, 2, 32), "pad": rng.random() < 0.7}
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 4, 200), "rows_lo": 1000,
                "rows_hi": _log_int(rng, 10_000, 200_000), "kmax": rng.randint(1, 16), "dtype": dtype}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(2, 12), "rows_lo": 10_000,
                "rows_hi": _log_int(rng, 50_000, 600_000), "requests": rng.randint(3, 20), "kmax": rng.randint(2, 32)}
    if kind == "power":
        return {"kind": kind, "n": _log_int(rng, 2000, 600_000), "lam": round(rng.uniform(5.0, 40.0), 3),
                "dtype": dtype}
    m = _draw_matrix(rng, ["powerlaw", "laplacian", "poisson"], most_nnz=24_000_000)
    if kind == "prep":
        return {"kind": kind, **m, "dtype": dtype, "cols": rng.random() < 0.7}
    grid = rng.randint(8, 128)
    return {"kind": kind, **m, "dtype": dtype, "order": order, "grid": grid, "levels": rng.choice([2, 4, 8])}


# ------------------------------------------------------------------ inputs

def _matrix(case, seed):
    if case["matrix"] == "blockdiag":
        return W.blockdiag(seed, n=case["n"], dtype=case["dtype"]).to("cuda")
    if case["matrix"] == "powerlaw":
        return W.powerlaw(seed, n=case["n"], dtype=case["dtype"], device="cuda")
    if case["matrix"] == "laplacian":
        return W.laplacian5(case["n"], case["dtype"], "cuda")
    return W.poisson_uniform(seed, case["n"], case["lam"], case["dtype"], "cuda")


def _perms(A, seed, order):
    if order == "natural":
        return None, None
    return maxe.maxe_build_permutation(seed, A.rows, 0), maxe.maxe_build_permutation(seed, A.cols, 1)


def _rand(seed, shape, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype) * 2 - 1


def _padded(n, k, dtype, pad):
    """Zeroed n x k rows, padded to whole 16 bytes when pad."""
    v = 16 // torch.empty(0, dtype=dtype).element_size()
    ld = (k + v - 1) // v * v if pad else k
    return torch.zeros(n, ld, dtype=dtype, device="cuda")[:, :k]


def _rhs(case, A, seed):
    X = _padded(A.cols, case["k"], VECTOR[case["dtype"]], case["pad"])
    X.copy_(_rand(seed + 17, (A.cols, case["k"]), VECTOR[case["dtype"]]))
    return X


def _batch_set(case, seed):
    """Matrices like the batched workload's (rows log-uniform, Poisson row lengths): the sizes and the numbers
    of right-hand sides are the workload's own, the entries are the seed's."""
    rng = np.random.default_rng(2308)
    rows = np.exp(rng.uniform(math.log(case["rows_lo"]), math.log(case["rows_hi"]), case["count"])).round()
    lams = rng.uniform(8.0, 64.0, case["count"])
    ks = rng.integers(1, case["kmax"] + 1, case["count"])
    mats = [W.poisson_uniform(seed * 1000 + m, int(rows[m]), float(lams[m]), case["dtype"], "cuda")
            for m in range(case["count"])]
    return mats, [int(k) for k in ks]


def _batch_rhs(case, A, k, seed, i):
    dt = VECTOR[case["dtype"]]
    X = _padded(A.cols, k, dt, k > 1)
    X.copy_(_rand(seed + 1000 + i, (A.cols, k), dt))
    return X


def _batch_ld(case, k):
    v = 16 // VECTOR_BYTES[case["dtype"]]
    return 1 if k == 1 else (k + v - 1) // v * v


def _serve_set(case, seed):
    """Matrices like the served workload's, sizes fixed as above."""
    rng = np.random.default_rng(2309)
    rows = np.exp(rng.uniform(math.log(case["rows_lo"]), math.log(case["rows_hi"]), case["count"])).round()
    lams = rng.uniform(5.0, 50.0, case["count"])
    return [W.poisson_uniform(seed * 1000 + m, int(rows[m]), float(lams[m]), "f32" if m % 2 == 0 else "bf16", "cuda")
            for m in range(case["count"])]


def _trace(case, seed):
    """One mix of requests, all there at the start; their vectors are the seed's."""
    trace = serve.make_trace(case["requests"], case["count"], math.inf, 2308, kmax=case["kmax"])
    for i, r in enumerate(trace):
        r.seed = seed * 1000 + i
    return trace


def _prep_matrix(case, seed):
    """One matrix whatever the seed (many permutations of it are drawn, as in the paper's protocol), other values."""
    A = _matrix(case, 2308)
    A.val = _rand(seed + 5, A.nnz, torch.float32).to(A.val.dtype)
    return A


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("spmv", "spmm"):
        A = _matrix(case, seed)
        rperm, cperm = _perms(A, seed, case["order"])
        s["h"] = maxe.from_csr(A, rperm, cperm, autotune=True)
        s["permuted"] = case["space"] == "permuted"
        dt = VECTOR[case["dtype"]]
        if kind == "spmv":
            s["x"] = _rand(seed + 17, A.cols, dt)
            s["y"] = torch.empty(A.rows, dtype=dt, device="cuda")
        else:
            s["X"] = _rhs(case, A, seed)
            s["Y"] = _padded(A.rows, case["k"], dt, case["pad"])
    elif kind == "batch":
        mats, ks = _batch_set(case, seed)
        # all results in one buffer, item after item
        lds = [_batch_ld(case, k) for k in ks]
        sizes = [A.rows * ld for A, ld in zip(mats, lds)]
        align = 4 if case["dtype"] != "f64" else 2
        starts = np.concatenate([[0], np.cumsum([(z + align - 1) // align * align for z in sizes])])
        s["out"] = torch.zeros(int(starts[-1]), dtype=VECTOR[case["dtype"]], device="cuda")
        s["handles"], items = [], []
        for i, (A, k) in enumerate(zip(mats, ks)):
            rperm, cperm = _perms(A, seed + i, "rc")
            h = maxe.from_csr(A, rperm, cperm)
            Y = s["out"][int(starts[i]):int(starts[i]) + sizes[i]].view(A.rows, lds[i])[:, :k]
            X = _batch_rhs(case, A, k, seed, i)
            s["handles"].append(h)
            items.append((h, X[:, 0] if k == 1 else X, Y[:, 0] if k == 1 else Y, False))
        s["batch"] = maxe.Batch(len(items))
        s["batch"].set(items)
    elif kind == "serve":
        s["server"] = serve.Server(_serve_set(case, seed), seed=seed)
        s["trace"] = _trace(case, seed)
    elif kind == "power":
        A = W.poisson_uniform(seed, case["n"], case["lam"], case["dtype"], "cuda")
        rperm, cperm = _perms(A, seed, "rc")
        s["h"] = maxe.from_csr(A, rperm, cperm, autotune=True)
        s["v0"] = _rand(seed + 17, A.rows, VECTOR[case["dtype"]])
    elif kind == "prep":
        s["A"] = _prep_matrix(case, seed)
        s["seed"] = seed
        s["cols"] = case["cols"]
    else:
        A = _matrix(case, seed)
        rperm, cperm = _perms(A, seed, case["order"])
        s["h"] = maxe.from_csr(A, rperm, cperm)
        s["grid"] = min(case["grid"], A.rows)
        s["levels"] = case["levels"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "spmv":
        return maxe.maxe_spmv(s["h"], s["x"], s["y"], permuted=s["permuted"])
    if kind == "spmm":
        return maxe.maxe_spmm(s["h"], s["X"], s["Y"], permuted=s["permuted"])
    if kind == "batch":
        s["batch"].run()
        return s["out"]
    if kind == "serve":
        reqs = [serve.clone_request(r) for r in s["trace"]]
        s["server"].run(reqs, keep_results=True)
        return [r.result if r.kind != "power" else r.result[:2] for r in reqs]
    if kind == "power":
        lam, v, hist = maxe.maxe_power_iteration(s["h"], s["v0"], POWER_STEPS, history=True)
        return {"lambda": lam, "v": v, "history": hist}
    if kind == "prep":
        A = s["A"]
        rperm = maxe.maxe_build_permutation(s["seed"], A.rows, 0)
        cperm = maxe.maxe_build_permutation(s["seed"], A.cols, 1) if s["cols"] else None
        h = maxe.from_csr(A, rperm, cperm)
        rowptr, col, val, _, _ = h.csr()
        rowptr.handle = h  # the three are views of the handle's arrays: they live as long as it does
        return {"rowptr": rowptr, "col": col, "val": val, "rperm": rperm, "cperm": cperm}
    H, counts = maxe.maxe_nnz_entropy(s["h"], s["grid"], s["grid"])
    return {"H": H, "counts": counts, "map": maxe.maxe_entropy_levels(counts, s["levels"])}


# ------------------------------------------------------------------ work

def _zipf_mean():
    k = np.arange(1, ZIPF_CAP + 1, dtype=np.float64)
    p = k ** -ZIPF_S
    return float((k * p).sum() / p.sum())


def _size(case):
    """(rows, expected nonzeros)."""
    n = case["n"]
    if case.get("matrix") == "blockdiag":
        return n, 0.02 * 16 * (n // 16) ** 2 + 2000
    if case.get("matrix") == "powerlaw":
        return n, n * _zipf_mean()
    if case.get("matrix") == "laplacian":
        return n * n, 5.0 * n * n - 4 * n
    return n, n * case["lam"]


def _product(rows, nnz, dtype, k=1):
    """Bytes and operations of Y = A X on a square matrix, every byte once."""
    vb, xb = VALUE_BYTES[dtype], VECTOR_BYTES[dtype]
    return nnz * (4 + vb) + 4 * (rows + 1) + 2 * rows * k * xb, 2 * nnz * k


def work(case):
    kind = case["kind"]
    if kind in ("spmv", "spmm"):
        rows, nnz = _size(case)
        b, f = _product(rows, nnz, case["dtype"], case.get("k", 1))
        if case["order"] == "rc" and case["space"] == "original":
            b += 8 * rows  # both permutations
    elif kind == "batch":
        rng = np.random.default_rng(2308)  # the expected matrix of the set, over many draws
        rows = np.exp(rng.uniform(math.log(case["rows_lo"]), math.log(case["rows_hi"]), 4096))
        per = [_product(r, 36.0 * r, case["dtype"], (case["kmax"] + 1) / 2) for r in rows]
        b, f = (case["count"] * float(np.mean([p[q] for p in per])) for q in (0, 1))
    elif kind == "serve":
        rng = np.random.default_rng(2308)
        rows = np.exp(rng.uniform(math.log(case["rows_lo"]), math.log(case["rows_hi"]), 4096))
        b = f = 0.0
        # 60% SpMV, 30% SpMM with 2..kmax columns, 10% power iteration (20 steps and the quotient)
        for share, k, units in ((0.6, 1, 1), (0.3, (2 + case["kmax"]) / 2, 1), (0.1, 1, POWER_STEPS + 1)):
            for dtype in ("f32", "bf16"):
                per = [_product(r, 27.5 * r, dtype, k) for r in rows]
                b += case["requests"] * share * units * 0.5 * float(np.mean([p[0] for p in per]))
                f += case["requests"] * share * units * 0.5 * float(np.mean([p[1] for p in per]))
    elif kind == "power":
        rows, nnz = _size(case)
        b, f = (q * (POWER_STEPS + 1) for q in _product(rows, nnz, case["dtype"]))
    elif kind == "prep":
        rows, nnz = _size(case)
        # the matrix in and out, the permutations out
        b, f = 2 * (nnz * (4 + VALUE_BYTES[case["dtype"]]) + 4 * (rows + 1)) + 4 * rows * (2 if case["cols"] else 1), 0
    else:
        rows, nnz = _size(case)
        b, f = 4 * nnz + 4 * (rows + 1) + 8 * case["grid"] ** 2, 0
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64-bit values, plain torch

def _shr(z, n):
    """Logical right shift of int64 bit patterns."""
    return (z >> n) & ((1 << (64 - n)) - 1)


def _i64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >= 1 << 63 else v


def _perm64(seed, n, tag):
    """0..n-1 in the order of SplitMix64's outputs 2i + tag + 1 for this seed, ties by index."""
    m = 2 * torch.arange(n, device="cuda", dtype=torch.int64) + (tag + 1)
    z = m * _i64(0x9E3779B97F4A7C15) + _i64(seed)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    return torch.sort(z ^ _i64(1 << 63), stable=True).indices


def _rows_of(A):
    rp = A.rowptr.long()
    return torch.repeat_interleave(torch.arange(A.rows, device="cuda"), rp[1:] - rp[:-1])


def _mul64(A, X, rows=None):
    """A X in FP64 for X of one or two dimensions."""
    rows = _rows_of(A) if rows is None else rows
    two = X.dim() == 2
    X = X.double() if two else X.double().unsqueeze(1)
    Y = torch.zeros(A.rows, X.shape[1], dtype=torch.float64, device="cuda")
    val, col = A.val.double(), A.col.long()
    for c in range(0, X.shape[1], 4):  # a few columns at a time bounds the products held
        Y[:, c:c + 4].index_add_(0, rows, val.unsqueeze(1) * X[:, c:c + 4][col])
    return Y if two else Y[:, 0]


def _mul64_permuted(A, X, r, c):
    """A' X' in FP64 for X' in the permuted space (perm[new] = old)."""
    Xo = torch.empty_like(X, dtype=torch.float64)
    Xo[c] = X.double()
    return _mul64(A, Xo)[r]


def _power64(A, v, steps):
    rows, hist = _rows_of(A), []
    v = v.double()
    w = _mul64(A, v, rows)
    for _ in range(steps):
        v = w / torch.linalg.vector_norm(w)
        w = _mul64(A, v, rows)
        hist.append(float(torch.dot(v, w)))
    return hist[-1], v, np.array(hist)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("spmv", "spmm"):
        A = _matrix(case, seed)
        X = _rand(seed + 17, A.cols, VECTOR[case["dtype"]]) if kind == "spmv" else _rhs(case, A, seed)
        if case["order"] == "rc" and case["space"] == "permuted":
            return _mul64_permuted(A, X, _perm64(seed, A.rows, 0), _perm64(seed, A.cols, 1))
        return _mul64(A, X)
    if kind == "batch":
        mats, ks = _batch_set(case, seed)
        align = 4 if case["dtype"] != "f64" else 2
        parts = []
        for i, (A, k) in enumerate(zip(mats, ks)):
            X = _batch_rhs(case, A, k, seed, i)
            ld = _batch_ld(case, k)
            n = (A.rows * ld + align - 1) // align * align
            part = torch.zeros(n, dtype=torch.float64, device="cuda")
            part[:A.rows * ld].view(A.rows, ld)[:, :k] = _mul64_permuted(A, X, _perm64(seed + i, A.rows, 0),
                                                                         _perm64(seed + i, A.cols, 1))
            parts.append(part)
        return torch.cat(parts)
    if kind == "serve":
        mats, out = _serve_set(case, seed), []
        g = torch.Generator(device="cuda")
        for q in _trace(case, seed):
            A = mats[q.mat]
            r, c = _perm64(seed + q.mat, A.rows, 0), _perm64(seed + q.mat, A.cols, 1)
            g.manual_seed(q.seed)
            if q.kind == "power":
                v0 = torch.empty(A.cols, dtype=torch.float64, device="cuda")
                v0[c] = (torch.rand(A.cols, generator=g, device="cuda") * 2 - 1).double()
                lam, v, _ = _power64(A, v0, q.steps)
                out.append([lam, v[c]])
            else:
                X = torch.rand(A.cols, q.k, generator=g, device="cuda") * 2 - 1
                out.append(_mul64_permuted(A, X, r, c))
        return out
    if kind == "power":
        A = W.poisson_uniform(seed, case["n"], case["lam"], case["dtype"], "cuda")
        lam, v, hist = _power64(A, _rand(seed + 17, A.rows, VECTOR[case["dtype"]]), POWER_STEPS)
        return {"lambda": lam, "v": v, "history": hist}
    A = _prep_matrix(case, seed) if kind == "prep" else _matrix(case, seed)
    if kind == "prep":
        r, c = _perm64(seed, A.rows, 0), _perm64(seed, A.cols, 1) if case["cols"] else None
        new_row, new_col = torch.empty_like(r), A.col.long()
        new_row[r] = torch.arange(A.rows, device="cuda")
        if c is not None:
            cinv = torch.empty_like(c)
            cinv[c] = torch.arange(A.cols, device="cuda")
            new_col = cinv[new_col]
        rows = new_row[_rows_of(A)]
        order = torch.sort(rows * A.cols + new_col, stable=True).indices
        rowptr = torch.zeros(A.rows + 1, dtype=torch.int64, device="cuda")
        rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=A.rows), 0)
        return {"rowptr": rowptr, "col": new_col[order], "val": A.val.double()[order], "rperm": r, "cperm": c}
    rows, cols, g = _rows_of(A), A.col.long(), min(case["grid"], A.rows)
    if case["order"] == "rc":
        for what, n, tag in (("r", A.rows, 0), ("c", A.cols, 1)):
            inv = torch.empty(n, dtype=torch.int64, device="cuda")
            inv[_perm64(seed, n, tag)] = torch.arange(n, device="cuda")
            if what == "r":
                rows = inv[rows]
            else:
                cols = inv[cols]
    counts = torch.bincount((rows * g // A.rows) * g + cols * g // A.cols, minlength=g * g).view(g, g)

    def entropy(t):
        p = t[t > 0].double() / max(1, int(t.sum()))
        return float(-(p * torch.log2(p)).sum())

    L = case["levels"]
    edge = [-(-a * g // L) for a in range(L + 1)]
    m = [[entropy(counts[edge[a]:edge[a + 1], edge[b]:edge[b + 1]]) for b in range(L)] for a in range(L)]
    return {"H": entropy(counts), "counts": counts, "map": torch.tensor(m, dtype=torch.float64, device="cuda")}
