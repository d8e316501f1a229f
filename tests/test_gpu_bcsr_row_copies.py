"""The 16-bit BCSR kernel where rows of B are copied by its lanes: pairs of elements and single ones, by
the parity of N, of the leading dimension and of B's address; one to many 32-column tiles, units of
one to many K-groups and blocks cut into units, rows that end with B's memory."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, rounded_inputs, torch_dtype

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("N", [2, 9, 18, 31, 33, 62, 99, 130])
@pytest.mark.parametrize("tiles", [5, 17, 40, 300])
def test_bcsr_row_copies(loops_lib, fmt, N, tiles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_rows, n_cols = 16 * 3 + 5, 400
    rng = np.random.default_rng(tiles)
    rows, cols = [], []
    for i in range(n_rows):
        pool = np.random.default_rng(7 + i // 16).choice(n_cols, tiles, replace=False)
        if i // 16 == 0:
            pool[0] = n_cols - 1                    # the last row of B
        take = np.unique(pool[rng.random(tiles) < 0.6])
        rows.append(np.full(take.size, i))
        cols.append(take)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    A = W.csr_from_coo(n_rows, n_cols, rows, cols, rng.standard_normal(rows.size))
    A_r, Bg, s, B_eff = rounded_inputs(A, W.dense_normal(n_cols, N, N), fmt)
    ref = oracle.spmm(A_r, B_eff)
    plan = loops_lib.Plan(A, N, fmt, tau=0.0)
    scale = torch.as_tensor(s, dtype=torch.float32).cuda()
    for pad in (0, 1, 2):
        for offset in (0, 1):                       # elements from an aligned address
            ld = N + pad
            flat = torch.full((offset + (n_cols - 1) * ld + N,), float("nan"), dtype=torch_dtype(torch, fmt),
                              device="cuda")
            B = torch.as_strided(flat, (n_cols, N), (ld, 1), offset)
            B.copy_(torch.as_tensor(Bg))
            C = plan.spmm(B, col_scale=scale)
            plan.check()
            assert rel_l2(C.double().cpu().numpy(), ref) <= TOL[fmt], (pad, offset)
