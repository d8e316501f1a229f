"""The 16-bit BCSR kernel over its column tiles and unit lengths: units of one to many K-groups (more
than the ring holds, and blocks cut into units), padded tiles, ragged rows and columns, rows of B
that the bulk copies can and cannot take."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, rounded_inputs, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("N", [1, 8, 16, 20, 32, 40, 64, 72, 128, 136, 256])
@pytest.mark.parametrize("tiles", [3, 16, 17, 33, 90, 400])
def test_bcsr_hmma_shapes(loops_lib, fmt, N, tiles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_rows, n_cols = 16 * 5 + 3, 600
    rng = np.random.default_rng(tiles)
    # every 16-row block holds entries of up to `tiles` distinct columns, the third block none
    rows, cols = [], []
    for i in range(n_rows):
        if i // 16 == 2:
            continue
        pool = np.random.default_rng(100 + i // 16).choice(n_cols, tiles, replace=False)
        take = rng.choice(pool, max(1, tiles // 2), replace=False)
        rows.append(np.full(take.size, i))
        cols.append(take)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    A = W.csr_from_coo(n_rows, n_cols, rows, cols, rng.standard_normal(rows.size))
    A_r, Bg, s, B_eff = rounded_inputs(A, W.dense_normal(n_cols, N, N), fmt)
    plan = loops_lib.Plan(A, N, fmt, tau=0.0)
    assert plan.info()["n_row_blocks"] == 5
    for pad in (0, 1, 8):
        C = plan.spmm(to_device(torch, Bg, fmt, ld=N + pad),
                      col_scale=torch.as_tensor(s, dtype=torch.float32).cuda())
        plan.check()
        assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A_r, B_eff)) <= TOL[fmt]
