"""The allocation-free SpMM over its column layouts (vectors, single columns, several per lane) and row
shapes: rows inside a chunk of 128 entries, on its boundary, over many chunks, empty runs at the
start, in the middle and at the end, and entries whose column lies outside B."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, to_device, torch_dtype

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _counts(shape):
    if shape == "short":
        return np.arange(700) % 9
    if shape == "aligned":      # every row ends on a chunk boundary
        return np.full(20, 128)
    if shape == "long":
        return np.array([0, 0, 3, 5000, 0, 127, 1, 128, 0, 129, 2000, 0])
    if shape == "empty":
        return np.zeros(100, dtype=np.int64)
    return np.concatenate([np.zeros(400), [1], np.zeros(2000), [300], np.zeros(300)]).astype(np.int64)   # sparse


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [1, 2, 7, 8, 16, 17, 32, 33, 48, 64, 65, 100, 128, 264])
@pytest.mark.parametrize("shape", ["short", "aligned", "long", "empty", "sparse"])
def test_noalloc_shapes(loops_lib, fmt, N, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(N)
    counts, n_cols = _counts(shape), 90
    rows = np.repeat(np.arange(counts.size), counts)
    A = W.csr_from_coo(counts.size, n_cols, rows, rng.integers(0, n_cols, rows.size),
                       oracle.round_to(rng.standard_normal(rows.size), fmt), sort_cols=False)
    ci = A.col_idx.copy()
    out = rng.random(ci.size) < 0.05                  # skipped entries: below 0 and past the last column
    ci[out] = np.where(rng.random(int(out.sum())) < 0.5, -3, n_cols + 2)
    A.vals[out] = 0.0
    Bq = oracle.round_to(W.dense_normal(n_cols, N, 5), fmt)
    dt = torch_dtype(torch, fmt)
    va = torch.as_tensor(np.where(out, 1.0, A.vals)).to(dt).cuda()
    for pad in (0, 8):
        C = torch.full((counts.size, N + pad), float("nan"), device="cuda",
                       dtype=torch.float64 if fmt == "f64" else torch.float32)[:, :N]
        loops_lib.csr_spmm_noalloc(torch.as_tensor(A.row_ptr).cuda(), torch.as_tensor(ci).cuda(), va, n_cols,
                                   to_device(torch, Bq, fmt, ld=N + pad), C)
        assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A, Bq)) <= TOL[fmt]
