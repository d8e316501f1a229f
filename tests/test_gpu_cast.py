"""The per-column scaled cast at the edges of its thread layout, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("rows,cols,pad,shift", [
    (1, 1, 0, 0), (3, 4, 0, 0), (1000, 47, 0, 0), (257, 300, 0, 0), (5, 1028, 0, 0), (20011, 128, 0, 0),
    (300, 64, 3, 0),   # rows of X not 16-byte aligned: one column per thread
    (300, 64, 4, 1),   # nor its first element
    (9000, 3, 0, 0),
])
def test_cast_scaled_shapes(loops_lib, fmt, rows, cols, pad, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = W.dense_normal(rows, cols, rows + cols) * np.exp2(np.arange(cols) % 25 - 12.0)[None, :]
    X[:, 0] *= 2.0 ** -140   # a subnormal column maximum: its scale has no binary32 reciprocal
    if cols > 2:
        X[:, 2] = 0.0
    X = X.astype(np.float32).astype(np.float64)
    buf = torch.zeros(rows * (cols + pad) + shift, dtype=torch.float32, device="cuda")
    Xd = buf[shift:].view(rows, cols + pad)[:, :cols]
    Xd.copy_(torch.as_tensor(X, dtype=torch.float32))
    Y, s = loops_lib.cast_scaled(Xd, fmt)
    ref_y, ref_s = oracle.scale_round_columns(X, fmt)
    assert np.array_equal(s.double().cpu().numpy(), ref_s)
    assert np.array_equal(Y.double().cpu().numpy(), ref_y)
