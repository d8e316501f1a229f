"""Paths that only very large operands take: 64-bit value maps, and rows of B or dC 2^32 bytes apart."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, to_device, torch_dtype

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("tau", [math.inf, 2.0, 0.0])
@pytest.mark.parametrize("on_device", [False, True])
def test_wide_value_maps(loops_lib, monkeypatch, fmt, tau, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lp = loops_lib
    A = W.random_csr(90, 70, 0.1, 3, unsorted=True)
    plain = lp._opts

    def wide(*a, **k):
        o = plain(*a, **k)
        o.test_wide_maps = 1
        return o

    plans = [lp.Plan(A, 16, fmt, tau=tau, want_backward=True, build_on_device=on_device)]
    monkeypatch.setattr(lp, "_opts", wide)
    plans.append(lp.Plan(A, 16, fmt, tau=tau, want_backward=True, build_on_device=on_device))
    # the map of every stored entry, in A's part and its transpose's, has twice the bytes
    assert plans[1].info()["device_bytes"] >= plans[0].info()["device_bytes"] + 2 * 4 * A.nnz - 2 * 256
    rng = np.random.default_rng(4)
    dC, B = (to_device(torch, oracle.round_to(W.dense_normal(n, 16, n), fmt), fmt) for n in (90, 70))
    for dt in (torch.float32, torch.float64):
        v = torch.as_tensor(rng.standard_normal(A.nnz), dtype=dt)
        got = []
        for plan in plans:
            plan.set_values(v.cuda())
            got.append((plan.export(), plan.spmm(B), *plan.backward(dC, B)))
        for key in got[0][0]:
            assert np.array_equal(np.asarray(got[0][0][key]), np.asarray(got[1][0][key]))
        assert torch.equal(got[0][1], got[1][1]) and torch.equal(got[0][2], got[1][2])
        assert rel_l2(got[1][3].double().cpu().numpy(), got[0][3].double().cpu().numpy()) <= TOL["f32"]
    v = rng.standard_normal(A.nnz)
    for plan in plans:
        plan.update_values(v)
    e0, e1 = plans[0].export(), plans[1].export()
    assert all(np.array_equal(np.asarray(e0[k]), np.asarray(e1[k])) for k in e0)


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [16, 47])
def test_rows_more_than_32_bits_apart(loops_lib, fmt, N):
    # two rows of B, then of dC, 2^32 + 64 bytes apart
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    eb = {"f64": 8, "f32": 4}.get(fmt, 2)
    ld = (2 ** 32 + 64) // eb
    buf = torch.zeros(ld + N, dtype=torch_dtype(torch, fmt), device="cuda")
    far = buf.as_strided((2, N), (ld, 1))
    A = W.random_csr(80, 2, 0.7, 5, unsorted=True)
    T = W.random_csr(2, 80, 0.7, 6, unsorted=True)
    for M, rows_of_B in ((A, 2), (T, 80)):
        s_a = oracle.plan_scale(M.vals, fmt)
        M_r = W.CSR(M.n_rows, M.n_cols, M.row_ptr, M.col_idx, oracle.round_to(M.vals * s_a, fmt) / s_a)
        B, dC = (oracle.round_to(W.dense_normal(n, N, n), fmt) for n in (M.n_cols, M.n_rows))
        Bd, dCd = to_device(torch, B, fmt), to_device(torch, dC, fmt)
        if M is A:
            Bd = far.copy_(Bd)
        else:
            dCd = far.copy_(dCd)
        plan = loops_lib.Plan(M, N, fmt, tau=math.inf, want_backward=True)
        assert rel_l2(plan.spmm(Bd).double().cpu().numpy(), oracle.spmm(M_r, B)) <= TOL[fmt]
        dB, dv = plan.backward(dCd, Bd)
        assert rel_l2(dB.double().cpu().numpy(), oracle.spmm_t(M_r, dC)) <= TOL[fmt]
        assert rel_l2(dv.double().cpu().numpy(), oracle.sddmm(M_r, dC, B)) <= TOL[fmt]
