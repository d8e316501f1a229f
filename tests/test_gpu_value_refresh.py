"""The binary32 value refresh against the binary64 one, which rounds scale * v once: stored values
equal bit for bit, also where the binary32 product would be subnormal, overflow or be special."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("tau", [math.inf, 0.0])
@pytest.mark.parametrize("magnitude", [1.0, 2.0 ** -120, 2.0 ** -300])   # of A: sets the plan scale
@pytest.mark.parametrize("on_device", [False, True])
def test_binary32_refresh_equals_binary64(loops_lib, fmt, tau, magnitude, on_device):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = W.random_csr(90, 70, 0.1, 3, unsorted=True)
    A.vals = A.vals * magnitude
    rng = np.random.default_rng(4)
    v = (rng.standard_normal(A.nnz) * np.exp2(rng.integers(-150, 127, A.nnz))).astype(np.float32)
    v[:4] = [0.0, -0.0, np.inf, -np.inf]
    plan = loops_lib.Plan(A, 16, fmt, tau=tau, want_backward=True, build_on_device=on_device)
    got = []
    for dt in (torch.float32, torch.float64):
        plan.set_values(torch.as_tensor(v, dtype=dt).cuda())
        got.append(plan.export())
    for key in ("csr_val", "tile_val"):
        assert np.array_equal(np.asarray(got[0][key]).view(np.int64), np.asarray(got[1][key]).view(np.int64)), key
