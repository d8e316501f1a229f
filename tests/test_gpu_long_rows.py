"""Rows of up to 512 entries under the default split length: taken by a whole block where few of them
would leave the chip idle, and without partial sums in the plan's memory, so that calls of one plan
may overlap on two streams. With a longer row all are cut into segments."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import TOL, rel_l2, rounded_inputs, to_device, torch_dtype

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rows_of(counts, n_cols, seed):
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(len(counts)), counts)
    return W.csr_from_coo(len(counts), n_cols, rows, rng.integers(0, n_cols, rows.size),
                          rng.standard_normal(rows.size), sort_cols=False)


def skewed(seed, longest):
    """Short rows around rows at the edges of the length classes and the longest team rows."""
    counts = np.arange(130) % 11
    counts[3:120:9] = [62, 63, 64, 65, 126, 127, 128, 300, 511, 512, longest, 400, 100]
    return rows_of(counts, 140, seed)


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("longest,cut_rows", [(512, 0), (513, 10)])      # segments of 64
@pytest.mark.parametrize("N", [1, 2, 4, 8, 13, 16, 26, 32, 47, 64, 66, 97, 128, 136, 194, 256, 520])
def test_long_rows(loops_lib, fmt, N, longest, cut_rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = skewed(N, longest)
    A_r, Bg, s, B_eff = rounded_inputs(A, W.dense_normal(140, N, N + 1), fmt)
    cs = torch.as_tensor(s, dtype=torch.float32).cuda() if s is not None else None
    dCq = oracle.round_to(W.dense_normal(A.n_rows, N, 2), fmt)
    Bq = oracle.round_to(W.dense_normal(140, N, 3), fmt)
    out = []
    for on_device in (False, True):
        plan = loops_lib.Plan(A, N, fmt, tau=math.inf, want_backward=True, build_on_device=on_device)
        assert plan.info()["n_split_rows"] == cut_rows
        C = plan.spmm(to_device(torch, Bg, fmt, ld=N + 8), col_scale=cs)
        dB, dv = plan.backward(to_device(torch, dCq, fmt), to_device(torch, Bq, fmt))
        assert rel_l2(C.double().cpu().numpy(), oracle.spmm(A_r, B_eff)) <= TOL[fmt]
        assert rel_l2(dB.double().cpu().numpy(), oracle.spmm_t(A_r, dCq)) <= TOL[fmt]
        assert rel_l2(dv.double().cpu().numpy(), oracle.sddmm(A_r, dCq, Bq)) <= TOL[fmt]
        out.append((C, dB, dv))
    assert all(torch.equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("fmt", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("N", [47, 64])
def test_long_rows_added_to_the_bcsr_part(loops_lib, fmt, N):
    # tile-level split: the moved entries of a block's rows are added to what the BCSR part wrote
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    counts = np.full(64, 3)
    counts[[1, 20, 40]] = [150, 400, 512]
    A = rows_of(counts, 900, N)
    A_r, Bg, _, B_eff = rounded_inputs(A, W.dense_normal(900, N, 1), fmt, scale_columns=False)
    for on_device in (False, True):
        plan = loops_lib.Plan(A, N, fmt, tau=0.0, tile_min=2, build_on_device=on_device)
        assert plan.info()["nnz_bcsr"] > 0 and plan.info()["nnz_csr"] > 500
        assert rel_l2(plan.spmm(to_device(torch, Bg, fmt)).double().cpu().numpy(), oracle.spmm(A_r, B_eff)) <= TOL[fmt]


@pytest.mark.parametrize("fmt,N", [("f32", 64), ("f32", 47), ("bf16", 128), ("f64", 32)])
def test_calls_of_one_plan_on_two_streams(loops_lib, fmt, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 1500
    A = rows_of(np.random.default_rng(1).integers(100, 400, n), n, 2)    # columns hold about 250 entries
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, want_backward=True, build_on_device=True)
    assert plan.info()["n_segments"] == 0
    dt = torch_dtype(torch, fmt)
    g = torch.Generator(device="cuda").manual_seed(3)
    X = [torch.randn(n, N, generator=g, device="cuda", dtype=torch.float64).to(dt) for _ in range(2)]
    ref = [(plan.spmm(x), plan.backward(x, x)) for x in X]
    streams = [torch.cuda.Stream() for _ in X]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(20):
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                got[i].append((plan.spmm(X[i]), plan.backward(X[i], X[i])))
    torch.cuda.synchronize()
    for i in range(2):
        for C, (dB, dv) in got[i]:
            assert torch.equal(C, ref[i][0]) and torch.equal(dB, ref[i][1][0]) and torch.equal(dv, ref[i][1][1])


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("fmt,N,segment", [("f32", 64, 64), ("f32", 512, 128), ("bf16", 2048, 128), ("f64", 1024, 128),
                                           ("f32", 4096, 256), ("f32", 1 << 16, 512)])
def test_default_segments_of_wide_rows(loops_lib, fmt, N, segment, on_device):
    # one row of 10^6 entries: the segments' partial sums (n_segments x N) stay small for any N
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nnz = 1_000_000
    A = rows_of(np.array([5, nnz, 0]), 700, 1)
    info = loops_lib.Plan(A, N, fmt, tau=math.inf, build_on_device=on_device).info()
    assert info["n_segments"] == -(-nnz // segment)
    plan = loops_lib.Plan(A, N, fmt, tau=math.inf, split_len=512, build_on_device=on_device)
    assert info["device_bytes"] <= plan.info()["device_bytes"] + (65 << 20)
