"""dB and dvals of one backward call (one pass over A^T where the transposed plan is all CSR) against
the two separate kernels, which calls for one of them alone take: dB bit for bit (the same sums in
the same order), dvals within the bound of two summation orders."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import to_device
from test_gpu_csr_shapes import staircase

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = {"f64": 2.0 ** -53, "f32": 2.0 ** -24, "f16": 2.0 ** -24, "bf16": 2.0 ** -24}


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [2, 4, 8, 16, 24, 40, 64, 88, 128, 136, 256, 264, 512, 520, 37])
@pytest.mark.parametrize("split_len,on_device", [(0, True), (9, False), (9, True)])
def test_backward_in_one_pass_equals_two(loops_lib, fmt, N, split_len, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = staircase(160, 110, N)                       # repeated entries, empty rows and columns
    A.col_idx[A.col_idx == 7] = 8
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, want_backward=True, split_len=split_len,
                          build_on_device=on_device)
    dC = oracle.round_to(W.dense_normal(160, N, 2), fmt)
    B = oracle.round_to(W.dense_normal(110, N, 3), fmt)
    scales = {}
    w = np.ones(N)
    if fmt in ("f16", "bf16"):
        ds, bs = np.exp2(np.arange(N) % 9 - 4.0), np.exp2(3.0 - np.arange(N) % 7)
        scales = dict(dc_scale=torch.as_tensor(ds, dtype=torch.float32).cuda(),
                      b_scale=torch.as_tensor(bs, dtype=torch.float32).cuda())
        w = ds * bs
    # leading dimensions that keep rows on 16 bytes, except for an odd N
    dCd, Bd = to_device(torch, dC, fmt, ld=N + 8), to_device(torch, B, fmt, ld=N + 16)
    dB, dv = plan.backward(dCd, Bd, **scales)
    dB1, _ = plan.backward(dCd, Bd, need_dvals=False, **scales)
    _, dv1 = plan.backward(dCd, Bd, need_dB=False, **scales)
    assert torch.equal(dB, dB1)
    # any order of a sum of N rounded products is within N * eps * sum |terms| of the exact one
    terms = oracle.sddmm(A, np.abs(dC) * w, np.abs(B))
    diff = np.abs(dv.double().cpu().numpy() - dv1.double().cpu().numpy())
    assert np.all(diff <= 2 * (N + 1) * EPS[fmt] * terms)
