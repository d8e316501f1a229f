"""The FP64 BCSR kernel on groups of tiles whose rows hold none to all of the group's four entries,
with ragged rows and columns, unaligned leading dimensions and blocks cut into units."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [1, 2, 15, 16, 17, 32, 33, 64, 100])
@pytest.mark.parametrize("pad", [0, 1, 2])
@pytest.mark.parametrize("per_row", [1, 3, 40, 300])   # 300: more tiles than a unit takes
def test_bcsr_f64_entry_patterns(loops_lib, N, pad, per_row):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_rows, n_cols = 61, 500
    rng = np.random.default_rng(per_row)
    counts = rng.integers(0, per_row + 1, n_rows)
    counts[8:16] = per_row          # one block of full rows, one empty block
    counts[24:32] = 0
    rows = np.repeat(np.arange(n_rows), counts)
    cols = rng.integers(0, min(n_cols, 2 * per_row), rows.size)   # clustered: full and sparse groups
    A = W.csr_from_coo(n_rows, n_cols, rows, cols, rng.standard_normal(rows.size), sort_cols=False)
    plan = loops_lib.Plan(A, N, "f64", tau=0.0)
    assert plan.info()["n_row_blocks"] > 0
    B = W.dense_normal(n_cols, N, N)
    C = plan.spmm(to_device(torch, B, "f64", ld=N + pad))
    assert rel_l2(C.cpu().numpy(), oracle.spmm(A, B)) <= TOL["f64"]
