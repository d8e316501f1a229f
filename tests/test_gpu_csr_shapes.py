"""The CSR kernel at the edges of its shapes: every lane-group width, one and two vectors per lane,
groups that cover the columns exactly or not, rows shorter and longer than a chunk of entries,
rows cut into segments, padded leading dimensions -- against the oracle."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, rounded_inputs, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def staircase(n_rows, n_cols, seed):
    """Row i holds i % 75 entries at random columns (repeats allowed)."""
    rng = np.random.default_rng(seed)
    counts = np.arange(n_rows) % 75
    rows = np.repeat(np.arange(n_rows), counts)
    return W.csr_from_coo(n_rows, n_cols, rows, rng.integers(0, n_cols, rows.size), rng.standard_normal(rows.size),
                          sort_cols=False)


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [8, 16, 24, 48, 64, 88, 128, 136, 256, 264, 520])
@pytest.mark.parametrize("split_len", [0, 33])
def test_csr_shapes(loops_lib, fmt, N, split_len):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = staircase(150, 90, N)
    A_r, Bg, s, B_eff = rounded_inputs(A, W.dense_normal(90, N, N + 1), fmt)
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, split_len=split_len)
    cs = torch.as_tensor(s, dtype=torch.float32).cuda() if s is not None else None
    C = plan.spmm(to_device(torch, Bg, fmt, ld=N + 8), col_scale=cs)
    assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A_r, B_eff)) <= TOL[fmt]


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [1, 2, 7, 9, 17, 23, 26, 33, 47, 50, 63, 65, 97, 98, 127, 130, 193, 260, 387])
@pytest.mark.parametrize("pad", [0, 1])
def test_csr_any_columns(loops_lib, fmt, N, pad):
    # any N and alignment: single columns and pairs per load, every count of pieces per lane
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = staircase(150, 90, N)
    A_r, Bg, s, B_eff = rounded_inputs(A, W.dense_normal(90, N, N + 1), fmt)
    cs = torch.as_tensor(s, dtype=torch.float32).cuda() if s is not None else None
    for split_len in (0, 33):
        plan = loops_lib.Plan(A, N, fmt, tau=math.inf, split_len=split_len)
        C = plan.spmm(to_device(torch, Bg, fmt, ld=N + pad), col_scale=cs)
        assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A_r, B_eff)) <= TOL[fmt]


@pytest.mark.parametrize("n,N,fmt", [(40, 64, "f32"), (40, 256, "f32"), (700, 16, "f16"), (700, 64, "f64")])
@pytest.mark.parametrize("on_device", [False, True])
def test_default_split_length_follows_the_size(loops_lib, n, N, fmt, on_device):
    # one dense row among short ones: cut by the default rule as by the same length given
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m = 3000
    rows = np.concatenate([np.full(m, 3), np.arange(n)])
    cols = np.concatenate([np.arange(m), np.arange(n)])
    A = W.csr_from_coo(n, m, rows, cols, np.random.default_rng(1).standard_normal(rows.size))
    B = torch.randn(m, N, device="cuda", dtype=torch.float64).to(
        {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}[fmt])
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, build_on_device=on_device)
    assert plan.info()["n_segments"] == -(-(m + 1) // 64)      # small problems: 64 entries
    same = loops_lib.Plan(A, N, fmt, tau=math.inf, split_len=64, build_on_device=on_device)
    assert torch.equal(plan.spmm(B), same.spmm(B))
