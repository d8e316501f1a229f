"""Which backward calls take the one pass over A^T, told by the kernels that a captured call holds (one, or
the SpMM and the SDDMM), and their gradients against the oracle."""
import ctypes
import math
import os

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, to_device
from test_gpu_csr_shapes import staircase

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def kernels_in(call):
    """Nodes of the CUDA graph that `call` (on the current stream) records."""
    from paper_2511_08158_gb300 import builder
    rt = ctypes.CDLL(os.path.join(os.path.dirname(os.path.dirname(builder.nvcc())), "lib64", "libcudart.so"))
    st = torch.cuda.Stream()
    h, graph, n = ctypes.c_void_p(st.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        assert rt.cudaStreamBeginCapture(h, 2) == 0        # relaxed: the caller may allocate its outputs
        try:
            call()
        finally:
            ended = rt.cudaStreamEndCapture(h, ctypes.byref(graph))
    assert ended == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [2, 4, 8, 16, 37, 40, 64, 128, 136, 256, 264, 512, 520])
@pytest.mark.parametrize("on_device", [False, True])
def test_backward_route_and_gradients(loops_lib, fmt, N, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = staircase(160, 110, N)
    s_a = oracle.plan_scale(A.vals, fmt)
    A_r = W.CSR(A.n_rows, A.n_cols, A.row_ptr, A.col_idx, oracle.round_to(A.vals * s_a, fmt) / s_a)
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, want_backward=True, build_on_device=on_device)
    dC, B = (oracle.round_to(W.dense_normal(n, N, n), fmt) for n in (160, 110))
    ve = {"f64": 2, "f32": 4}.get(fmt, 8)
    for pad in (0, 1):                                     # 1: rows off 16 bytes
        dCd, Bd = to_device(torch, dC, fmt, ld=N + pad), to_device(torch, B, fmt)
        one_pass = N % ve == 0 and N // ve <= 64 and pad == 0
        assert kernels_in(lambda: plan.backward(dCd, Bd)) == (1 if one_pass else 2)
        dB, dv = plan.backward(dCd, Bd)
        assert rel_l2(dB.double().cpu().numpy(), oracle.spmm_t(A_r, dC)) <= TOL[fmt]
        assert rel_l2(dv.double().cpu().numpy(), oracle.sddmm(A_r, dC, B)) <= TOL[fmt]
    hybrid = loops_lib.Plan(A, N, fmt, tau=0.0, want_backward=True, build_on_device=on_device)
    assert kernels_in(lambda: hybrid.backward(dCd, Bd)) > 1
