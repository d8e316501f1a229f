"""FP32 batched units for either tile height: column groups that cover N exactly and not, odd and even
tile counts around the tiles in flight, a last row block that is not full, host and device builds."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def blocks_of(n_rows, n_cols, tiles, seed):
    """Row block i (8 rows) holds entries of tiles[i % len(tiles)] columns, every column in some row."""
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for b in range(-(-n_rows // 8)):
        t = tiles[b % len(tiles)]
        c = rng.choice(n_cols, t, replace=False)
        r = np.arange(b * 8, min(b * 8 + 8, n_rows))
        keep = rng.random((r.size, t)) < 0.6
        keep[rng.integers(0, r.size, t), np.arange(t)] = True
        i, j = np.nonzero(keep)
        rows.append(r[i])
        cols.append(c[j])
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    return W.csr_from_coo(n_rows, n_cols, rows, cols, rng.standard_normal(rows.size))


@pytest.mark.parametrize("block_rows", [8, 16])
@pytest.mark.parametrize("tau", [0.0, 2.0])
@pytest.mark.parametrize("on_device", [False, True])
def test_batched_f32_units(loops_lib, block_rows, tau, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tiles = [1, 2, 3, 4, 5, 6, 7, 300]             # 300: more tiles than a unit takes
    mats = [(blocks_of(8 * 9 + m % 8, 400, tiles, m), N)
            for m, N in enumerate((4, 8, 12, 16, 24, 32, 40, 48, 64, 68, 96, 124, 128))]
    plan = loops_lib.BatchedPlan([A for A, _ in mats], [N for _, N in mats], "f32", tau=tau, block_rows=block_rows,
                                 build_on_device=on_device)
    assert plan.info()["block_rows"] == block_rows and plan.stats()["nnz_bcsr"] > 0
    Bs = [oracle.round_to(W.dense_normal(A.n_cols, N, N), "f32") for A, N in mats]
    Cs = plan.spmm([torch.as_tensor(B, dtype=torch.float32).cuda() for B in Bs])
    for (A, _), B, C in zip(mats, Bs, Cs):
        A_r = W.CSR(A.n_rows, A.n_cols, A.row_ptr, A.col_idx, oracle.round_to(A.vals, "f32"))
        assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A_r, B)) <= TOL["f32"]
