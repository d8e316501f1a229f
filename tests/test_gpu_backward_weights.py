"""dvals of the 16-bit backward where the column weights times B leave binary32's normal range (above
and below it) while the weights times dC, and the results, do not."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import to_device
from test_gpu_csr_shapes import staircase

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("N", [8, 16, 40, 64, 128, 136, 256])
@pytest.mark.parametrize("split_len,on_device", [(0, False), (9, True)])
def test_dvals_with_weights_out_of_range_on_B(loops_lib, fmt, N, split_len, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, m = 150, 90
    A = staircase(n, m, N)
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, want_backward=True, split_len=split_len, build_on_device=on_device)
    row, big, small = np.arange(n), 0, N - 1
    dC = W.dense_normal(n, N, 2)
    # column `big`: weight 2^120, dC zero or near 2^-20; column `small`: weight 2^-118, dC near 2^10
    dC[:, [big, small]] = 0.0
    dC[row % 3 == 0] = 0.0
    dC[row % 3 == 0, big] = W.dense_normal(n, 1, 4)[row % 3 == 0, 0] * 2.0 ** -20
    dC[row % 3 == 1] = 0.0
    dC[row % 3 == 1, small] = W.dense_normal(n, 1, 5)[row % 3 == 1, 0] * 2.0 ** 10
    B = W.dense_normal(m, N, 3)
    B[:, big] *= 2.0 ** 10
    B[:, small] *= 2.0 ** -10
    B[::7, big] = 0.0                                        # rows whose weighted elements stay in range
    B[::7, small] = 0.0
    dC, B = oracle.round_to(dC, fmt), oracle.round_to(B, fmt)
    ds, bs = np.ones(N), np.ones(N)
    ds[big], bs[big], ds[small], bs[small] = 2.0 ** 100, 2.0 ** 20, 2.0 ** -98, 2.0 ** -20
    f32 = dict(dtype=torch.float32, device="cuda")
    scales = dict(dc_scale=torch.as_tensor(ds, **f32), b_scale=torch.as_tensor(bs, **f32))
    dCd, Bd = to_device(torch, dC, fmt, ld=N + 8), to_device(torch, B, fmt)
    dB, dv = plan.backward(dCd, Bd, **scales)
    dB1, _ = plan.backward(dCd, Bd, need_dvals=False, **scales)
    assert torch.equal(dB, dB1)
    got, ref = dv.double().cpu().numpy(), oracle.sddmm(A, dC * (ds * bs), B)
    # N rounded products in any order of summation; the weights are powers of two
    assert np.all(np.abs(got - ref) <= (N + 1) * 2.0 ** -24 * oracle.sddmm(A, np.abs(dC) * (ds * bs), np.abs(B)))
