"""What the performance of this package is measured on: the SpMM calls a program makes, from the
smallest to the largest, each through the public entry points.

A case names a family (one kind of matrix and one way of calling the package) and its sizes:

  uniform    a square matrix with the same number of random columns in every row; one
             ``Plan.spmm`` with the plan's default split threshold
  laplacian  the 5-point Laplacian with dense 8 x 8 diagonal blocks in FP64, the hybrid split;
             one ``Plan.spmm``
  features   a power-law graph in FP16 / BF16: FP32 features are scaled per column and cast
             (``cast_scaled``), then multiplied (``Plan.spmm`` with the column scales)
  layer      a power-law graph with any N (class logits, odd widths); one ``Plan.spmm``
  train      a GCN-style layer: ``spmm`` under autograd and its gradients for A's values and B
  mix        half the 16-row blocks hold two dense 16 x 16 blocks, the other rows scattered
             entries: both parts of the hybrid split at work; one ``Plan.spmm``
  batch      many matrices of uneven size, structure and N behind one ``BatchedPlan.spmm``
  replan     a pattern that changes from call to call: ``Plan(build_on_device=True)``, then one
             ``Plan.spmm``
  noalloc    ``csr_spmm_noalloc`` on the caller's own CSR arrays

Inputs are made on the GPU from the seed. Plans use fixed thresholds, so that one case is one
split: the default (2.0) where a hybrid split is wanted, and no BCSR part for graphs, which is
what the autotuner keeps for them.
"""
from __future__ import annotations

import math

import torch

import paper_2511_08158_gb300 as lp

_TORCH = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: a 2,000-row matrix, bound by launches and the host
        {"name": "uniform_2k_f32_n32", "family": "uniform", "n": 2000, "per_row": 10, "N": 32, "dtype": "f32"},
        # a discretised operator with locally dense couplings in FP64, several right-hand sides
        {"name": "laplacian_512_f64_n64", "family": "laplacian", "grid": 512, "N": 64, "dtype": "f64"},
        # inference over a graph of a million nodes with 16-bit features
        {"name": "features_1m_f16_n128", "family": "features", "n": 1 << 20, "degree": 16, "N": 128,
         "dtype": "f16"},
        # the last layer of a graph network: one column per class, an odd number of them
        {"name": "layer_200k_f32_n47", "family": "layer", "n": 200003, "degree": 24, "N": 47, "dtype": "f32"},
        # one training step of a GCN layer, FP32: forward, gradients of the values and of B
        {"name": "train_256k_f32_n256", "family": "train", "n": 1 << 18, "degree": 32, "N": 256, "dtype": "f32"},
        # the same step on 16-bit operands, with the per-column scaled gradients
        {"name": "train_256k_bf16_n128", "family": "train", "n": 1 << 18, "degree": 32, "N": 128, "dtype": "bf16"},
        # the matrix the hybrid split is made for, BF16: tensor-core blocks beside scattered rows
        {"name": "mix_1m_bf16_n64", "family": "mix", "n": 1 << 20, "N": 64, "dtype": "bf16"},
        # the same structure in FP32 (CUDA-core blocks), the width the paper measures at
        {"name": "mix_256k_f32_n32", "family": "mix", "n": 1 << 18, "N": 32, "dtype": "f32"},
        # many small and middling matrices in one call, FP32 and BF16
        {"name": "batch_128_f32", "family": "batch", "count": 128, "max_rows": 65536, "dtype": "f32"},
        {"name": "batch_96_bf16", "family": "batch", "count": 96, "max_rows": 65536, "dtype": "bf16"},
        # a dynamic graph: the matrix is converted on the GPU for every product
        {"name": "replan_256k_f16_n128", "family": "replan", "n": 1 << 18, "degree": 16, "N": 128, "dtype": "f16"},
        # a caller that may not allocate: its own CSR arrays, no plan
        {"name": "noalloc_64k_f32_n64", "family": "noalloc", "n": 65536, "per_row": 32, "N": 64, "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _any_n(rng, hi):
    """Columns of B: the widths the package is tuned for, or any number."""
    if rng.random() < 0.5:
        return rng.choice([w for w in (8, 16, 32, 64, 128, 256) if w <= hi])
    return rng.randint(1, hi)


def draw(rng):
    family = rng.choice(["uniform", "laplacian", "features", "layer", "train", "mix", "batch", "replan", "noalloc"])
    if family == "uniform":
        per_row = rng.randint(4, 64)
        return {"family": family, "n": _log_int(rng, 500, 4_000_000 // per_row), "per_row": per_row,
                "N": _any_n(rng, 128), "dtype": rng.choice(["f64", "f32", "f16", "bf16"])}
    if family == "laplacian":
        return {"family": family, "grid": _log_int(rng, 40, 512), "N": _any_n(rng, 96), "dtype": "f64"}
    if family == "features":
        return {"family": family, "n": _log_int(rng, 4000, 1 << 20), "degree": rng.randint(6, 16),
                "N": rng.choice([16, 32, 64, 96, 128, rng.randint(9, 120)]), "dtype": rng.choice(["f16", "bf16"])}
    if family == "layer":
        return {"family": family, "n": _log_int(rng, 4000, 250_000), "degree": rng.randint(8, 32),
                "N": rng.randint(2, 130), "dtype": rng.choice(["f32", "f16", "bf16"])}
    if family == "train":
        return {"family": family, "n": _log_int(rng, 2000, 1 << 18), "degree": rng.randint(8, 32),
                "N": rng.choice([16, 32, 64, 128, 256, rng.randint(5, 200)]),
                "dtype": rng.choice(["f32", "f32", "f16", "bf16"])}
    if family == "mix":
        return {"family": family, "n": _log_int(rng, 8000, 1 << 19), "N": _any_n(rng, 128),
                "dtype": rng.choice(["f64", "f32", "f16", "bf16"])}
    if family == "batch":
        return {"family": family, "count": _log_int(rng, 8, 96), "max_rows": _log_int(rng, 4000, 65536),
                "dtype": rng.choice(["f32", "f16", "bf16"])}
    if family == "replan":
        return {"family": family, "n": _log_int(rng, 4000, 1 << 18), "degree": rng.randint(4, 16),
                "N": _any_n(rng, 128), "dtype": rng.choice(["f64", "f32", "f16", "bf16"])}
    per_row = rng.randint(4, 48)
    return {"family": family, "n": _log_int(rng, 500, 2_000_000 // per_row), "per_row": per_row,
            "N": _any_n(rng, 64), "dtype": rng.choice(["f64", "f32", "f16", "bf16"])}


# ------------------------------------------------------------------ inputs
class _Matrix:
    """A CSR matrix in device memory, as ``Plan(build_on_device=True)`` takes it."""

    def __init__(self, n_rows, n_cols, row_ptr, col_idx, vals):
        self.n_rows, self.n_cols = n_rows, n_cols
        self.row_ptr, self.col_idx, self.vals = row_ptr, col_idx, vals

    @property
    def nnz(self):
        return int(self.col_idx.numel())

    def rows(self):
        n = torch.arange(self.n_rows, device="cuda")
        return torch.repeat_interleave(n, self.row_ptr[1:] - self.row_ptr[:-1])


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _row_ptr(counts):
    rp = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=rp[1:])
    return rp


def _spread(g, rows_k, place, n_cols):
    """Random columns, distinct and ascending within a row: entry ``place`` of a row of
    ``rows_k`` entries lies anywhere in its own share of the columns."""
    lo = place * n_cols // rows_k
    hi = (place + 1) * n_cols // rows_k
    u = torch.rand(place.numel(), generator=g, device="cuda", dtype=torch.float64)
    return torch.minimum(lo + (u * (hi - lo)).long(), hi - 1)


def _scattered(g, n, counts, vals_dtype):
    """n x n matrix with counts[i] random columns in row i and N(0, 1) values."""
    counts = counts.clamp(max=n)
    rp = _row_ptr(counts)
    k = torch.repeat_interleave(counts, counts)
    place = torch.arange(k.numel(), device="cuda") - torch.repeat_interleave(rp[:-1], counts)
    cols = _spread(g, k, place, n)
    return _Matrix(n, n, rp, cols.int(), _normal(g, k.numel(), dtype=vals_dtype))


def _uniform(g, n, per_row, vals_dtype):
    return _scattered(g, n, torch.full((n,), per_row, dtype=torch.int64, device="cuda"), vals_dtype)


def _from_keys(n, keys, vals):
    rows, cols = keys // n, keys % n
    return _Matrix(n, n, _row_ptr(torch.bincount(rows, minlength=n)), cols.int(), vals)


def _graph_entries(n, degree):
    """Entries off the diagonal: about what R-MAT's n * degree samples leave without duplicates."""
    return min(int(0.85 * n * degree), n * (n - 1) // 2)


def _graph(g, n, degree, loops):
    """R-MAT(0.57, 0.19, 0.19, 0.05) graph of n nodes, both directions of every sampled edge,
    without duplicates, then cut (or filled with random edges) to a fixed number of entries; with
    ``loops`` the diagonal too. Values 1 / sqrt(d_i d_j) in FP32."""
    want = _graph_entries(n, degree)
    scale = max(1, (n - 1).bit_length())
    m = n * degree // 2
    src = torch.zeros(m, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device="cuda")
        src = (src << 1) | (r >= 0.76).long()
        dst = (dst << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long()
    src, dst = src % n, dst % n
    keys = torch.cat([src * n + dst, dst * n + src])
    keys = torch.unique(keys[keys // n != keys % n])
    while keys.numel() < want:
        more = torch.randint(0, n * n, (want,), generator=g, device="cuda")
        keys = torch.unique(torch.cat([keys, more[more // n != more % n]]))
    if keys.numel() > want:
        keep = torch.randperm(keys.numel(), generator=g, device="cuda")[:want]
        keys = keys[torch.sort(keep).values]
    if loops:
        i = torch.arange(n, device="cuda")
        keys = torch.sort(torch.cat([keys, i * n + i])).values
    rows, cols = keys // n, keys % n
    d_out = torch.bincount(rows, minlength=n).double().clamp(min=1)
    d_in = torch.bincount(cols, minlength=n).double().clamp(min=1)
    return _from_keys(n, keys, (1 / torch.sqrt(d_out[rows] * d_in[cols])).float())


def _laplacian(g, grid):
    """5-point Laplacian on a grid x grid mesh, one in eight of the aligned 8 x 8 diagonal
    blocks filled with N(0, 1) on top."""
    n = grid * grid
    i = torch.arange(n, device="cuda")
    x, y = i % grid, i // grid
    keys, vals = [i * n + i], [torch.full((n,), 4.0, dtype=torch.float64, device="cuda")]
    for dx, dy in ((-1, 0), (1, 0), (0, -1), (0, 1)):
        ok = (x + dx >= 0) & (x + dx < grid) & (y + dy >= 0) & (y + dy < grid)
        k = i[ok] * n + i[ok] + dx + dy * grid
        keys.append(k)
        vals.append(torch.full((k.numel(),), -1.0, dtype=torch.float64, device="cuda"))
    n_diag = n // 8
    at = torch.randperm(n_diag, generator=g, device="cuda")[: max(1, n_diag // 8)] * 8
    e = torch.arange(8, device="cuda")
    k = ((at[:, None, None] + e[None, :, None]) * n + at[:, None, None] + e[None, None, :]).reshape(-1)
    keys.append(k)
    vals.append(_normal(g, k.numel(), dtype=torch.float64))
    keys, where = torch.unique(torch.cat(keys), return_inverse=True)
    v = torch.zeros(keys.numel(), dtype=torch.float64, device="cuda")
    order = torch.argsort(where, stable=True)      # coincident entries added in one fixed order
    all_v, where = torch.cat(vals)[order], where[order]
    first = torch.ones_like(where, dtype=torch.bool)
    first[1:] = where[1:] != where[:-1]
    v[where[first]] = all_v[first]
    v[where[~first]] += all_v[~first]
    return _from_keys(n, keys, v)


def _mix(g, n, vals_dtype, dense_fraction=0.5):
    """A random half of the 16-row blocks hold two dense 16 x 16 blocks, the other rows 16
    scattered entries each; values N(0, 1)."""
    n_rb, n_cb = (n + 15) // 16, n // 16
    dense_rb = torch.rand(n_rb, generator=g, device="cuda") < dense_fraction
    i = torch.arange(n, device="cuda")
    dense = dense_rb[i // 16]
    counts = torch.where(dense, 32, 16)
    rp = _row_ptr(counts)
    cols = torch.empty(int(rp[-1]), dtype=torch.int32, device="cuda")
    c0 = torch.randint(0, n_cb, (n_rb,), generator=g, device="cuda")
    c1 = (c0 + 1 + torch.randint(0, n_cb - 1, (n_rb,), generator=g, device="cuda")) % n_cb
    e = torch.arange(16, device="cuda")
    pair = torch.cat([torch.minimum(c0, c1)[:, None] * 16 + e, torch.maximum(c0, c1)[:, None] * 16 + e], 1)
    rows = i[dense]
    cols[(rp[rows][:, None] + torch.arange(32, device="cuda")).reshape(-1)] = pair[rows // 16].reshape(-1).int()
    rows = i[~dense]
    place = e.repeat(rows.numel())
    cols[(rp[rows][:, None] + e).reshape(-1)] = _spread(g, torch.full_like(place, 16), place, n).int()
    return _Matrix(n, n, rp, cols, _normal(g, cols.numel(), dtype=vals_dtype))


def _banded(g, n, half):
    i = torch.arange(n, device="cuda")
    j = i[:, None] + torch.arange(-half, half + 1, device="cuda")
    ok = (j >= 0) & (j < n)
    cols = j[ok].int()
    return _Matrix(n, n, _row_ptr(ok.sum(1)), cols, _normal(g, cols.numel()))


def _batch_shapes(case):
    """(rows, N, structure) of every matrix: fixed by the case, spread evenly over the range."""
    out = []
    for m in range(case["count"]):
        f = (m * 0.6180339887498949) % 1.0         # low-discrepancy points of [0, 1)
        rows = int(1000 * (case["max_rows"] / 1000) ** f)
        out.append((rows, (16, 32, 64, 128)[(m // 3) % 4], m % 3))
    return out


def _batch(g, case):
    mats = []
    for rows, _, kind in _batch_shapes(case):
        if kind == 0:
            mats.append(_scattered(g, rows, torch.randint(8, 65, (rows,), generator=g, device="cuda"), torch.float32))
        elif kind == 1:
            mats.append(_banded(g, rows, 16))
        else:
            mats.append(_mix(g, rows, torch.float32, dense_fraction=2.0))
    return mats


def _matrix(g, case):
    f = case["family"]
    vals_dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    if f == "laplacian":
        return _laplacian(g, case["grid"])
    if f == "mix":
        return _mix(g, case["n"], vals_dtype)
    if f in ("uniform", "noalloc"):
        A = _uniform(g, case["n"], case["per_row"], vals_dtype)
        if f == "noalloc":                          # the values as the kernel multiplies them
            A.vals = A.vals.to(_TORCH[case["dtype"]])
        return A
    return _graph(g, case["n"], case["degree"], loops=f == "train")


def _inputs(case, seed):
    """Everything random of a case, from the seed alone."""
    g = _gen(seed)
    if case["family"] == "batch":
        mats = _batch(g, case)
        Bs = [_normal(g, A.n_cols, N).to(_TORCH[case["dtype"]]) for A, (_, N, _) in zip(mats, _batch_shapes(case))]
        return mats, Bs
    A = _matrix(g, case)
    f, N, dt = case["family"], case["N"], _TORCH[case["dtype"]]
    if f == "features":
        # features of very different magnitudes per column: what the column scales are for
        B = _normal(g, A.n_cols, N) * torch.exp2(torch.randint(-12, 13, (N,), generator=g, device="cuda").float())
    else:
        B = _normal(g, A.n_cols, N, dtype=torch.float64 if dt == torch.float64 else torch.float32).to(dt)
    dC = _normal(g, A.n_rows, N) if f == "train" else None
    return A, B, dC


def _graph_tau(case):
    return math.inf if case["family"] in ("features", "layer", "train", "replan") else 2.0


def prepare(case, seed):
    s = dict(case=case)
    if case["family"] == "batch":
        mats, s["B"] = _inputs(case, seed)
        Ns = [N for _, N, _ in _batch_shapes(case)]
        s["plan"] = lp.BatchedPlan(mats, Ns, case["dtype"], tau=2.0, block_rows=8 if case["dtype"] == "f32" else 0,
                                   build_on_device=True)
        # every C back to back in one array, as a program with one output arena lays them out
        s["arena"] = torch.empty(sum(A.n_rows * N for A, N in zip(mats, Ns)), device="cuda")
        s["C"], at = [], 0
        for A, N in zip(mats, Ns):
            s["C"].append(s["arena"][at:at + A.n_rows * N].view(A.n_rows, N))
            at += A.n_rows * N
        return s
    s["A"], s["B"], s["dC"] = _inputs(case, seed)
    f = case["family"]
    if f == "noalloc":
        s["C"] = torch.empty(s["A"].n_rows, case["N"], device="cuda",
                             dtype=torch.float64 if case["dtype"] == "f64" else torch.float32)
    elif f != "replan":
        s["plan"] = lp.Plan(s["A"], case["N"], case["dtype"], tau=_graph_tau(case), want_backward=f == "train",
                            build_on_device=True)
    if f == "train":
        s["vals"] = s["A"].vals.clone().requires_grad_()
        s["B"].requires_grad_()
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    f = case["family"]
    if f == "batch":
        s["plan"].spmm(s["B"], s["C"])
        return s["arena"]
    if f == "features":
        Y, scale = lp.cast_scaled(s["B"], case["dtype"])
        return [s["plan"].spmm(Y, col_scale=scale), Y, scale]
    if f == "train":
        C = lp.spmm(s["plan"], s["vals"], s["B"])
        dvals, dB = torch.autograd.grad(C, [s["vals"], s["B"]], s["dC"])
        return [C.detach(), dvals, dB]
    if f == "replan":
        plan = lp.Plan(s["A"], case["N"], case["dtype"], tau=_graph_tau(case), build_on_device=True)
        return plan.spmm(s["B"])
    if f == "noalloc":
        A = s["A"]
        return lp.csr_spmm_noalloc(A.row_ptr, A.col_idx, A.vals, A.n_cols, s["B"], s["C"])
    return s["plan"].spmm(s["B"])


# ------------------------------------------------------------------ what a pass cannot do without
def _nnz(case):
    f = case["family"]
    if f in ("uniform", "noalloc"):
        return case["n"] * min(case["per_row"], case["n"])
    if f == "laplacian":
        n = case["grid"] ** 2
        return 5 * n - 4 * case["grid"] + 42 * max(1, n // 64)
    if f == "mix":
        return 24 * case["n"]
    return _graph_entries(case["n"], case["degree"]) + (case["n"] if f == "train" else 0)


def work(case):
    f, e = case["family"], _BYTES[case["dtype"]]
    c = 8 if case["dtype"] == "f64" else 4
    if f == "batch":
        total, flops = 0, 0
        for rows, N, kind in _batch_shapes(case):
            nnz = rows * (36, 33, 32)[kind]
            total += 8 * (rows + 1) + nnz * (4 + e) + rows * N * (e + c)
            flops += 2 * nnz * N
        return {"bytes": total, "flops": flops}
    n = case["grid"] ** 2 if f == "laplacian" else case["n"]
    nnz, N = _nnz(case), case["N"]
    a = 8 * (n + 1) + nnz * (4 + e)                 # the pattern and the values, once
    if f == "features":                             # FP32 features in, their cast and C out
        return {"bytes": a + n * N * (4 + e + c), "flops": 2 * nnz * N}
    if f == "train":                                # values, B and dC in; C, dvals and dB out
        return {"bytes": 8 * (n + 1) + nnz * (4 + 4 + 4) + n * N * (e + 4 + c + e), "flops": 6 * nnz * N}
    return {"bytes": a + n * N * (e + c), "flops": 2 * nnz * N}


# ------------------------------------------------------------------ the same results in 64 bits
def _spmm64(row_ptr, col_idx, vals, n_rows, n_cols, B):
    A = torch.sparse_csr_tensor(row_ptr, col_idx.long(), vals.double(), size=(n_rows, n_cols))
    return A @ B.double()


def exact(case, seed):
    with torch.no_grad():
        if case["family"] == "batch":
            mats, Bs = _inputs(case, seed)
            return torch.cat([_spmm64(A.row_ptr, A.col_idx, A.vals, A.n_rows, A.n_cols, B).reshape(-1)
                              for A, B in zip(mats, Bs)])
        A, B, dC = _inputs(case, seed)
        f = case["family"]
        C = _spmm64(A.row_ptr, A.col_idx, A.vals, A.n_rows, A.n_cols, B)
        if f == "features":
            top = B.abs().amax(0).double()
            scale = torch.where(top > 0, torch.exp2(torch.ceil(torch.log2(top))), torch.ones_like(top))
            return [C, B.double() / scale, scale]
        if f == "train":
            rows, cols = A.rows(), A.col_idx.long()
            order = torch.argsort(cols, stable=True)
            t_rp = _row_ptr(torch.bincount(cols, minlength=A.n_cols))
            dB = _spmm64(t_rp, rows[order], A.vals[order], A.n_cols, A.n_rows, dC)
            dv = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
            for at in range(0, A.nnz, 1 << 20):
                r, c = rows[at:at + (1 << 20)], cols[at:at + (1 << 20)]
                dv[at:at + (1 << 20)] = (dC[r].double() * B[c].double()).sum(1)
            return [C, dv, dB]
        return C
