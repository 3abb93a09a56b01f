"""Streams of few rows, which are cut into runs that warps share: every storage type of Z, aligned and odd rows, rows that end
inside a run and inside a sub-token, and the time of a few rows against that of many."""
import numpy as np
import pytest
import torch

import oracle
import velora_inputs as vi
from _util import TOL_GEMM, TOL_Z, Guard, assert_matches, to_f64

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
F8 = torch.float8_e4m3fn


@pytest.fixture(scope="module")
def vl():
    import paper_2405_17991_b200 as pkg
    pkg.lib()
    return pkg


@pytest.fixture
def guard():
    g = Guard(DEV)
    yield g
    g.check()


# One row, a few, and as many as leave each one run; runs of one round and of several; one, two and many sub-tokens.
@pytest.mark.parametrize("N,D,Dsub", [(1, 11005, 64), (3, 11008, 8), (40, 11005, 256), (16, 5461, 1024), (7, 8200, 512), (1, 4099, 16), (2, 2304, 128),
                                      (5000, 264, 256), (4800, 515, 32), (600, 4100, 8)])
@pytest.mark.parametrize("dtype,pad", [("bf16", 0), ("bf16", 3), ("f32", 0), ("f32", 1)])
def test_streams(vl, guard, N, D, Dsub, dtype, pad):
    case = vi.small_case(N + D + Dsub, N, D, 8, dtype=dtype, mean_offset=0.1)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    ld = (D + pad) if pad else -(-D // 8) * 8
    buf = torch.full((N * ld,), float("nan"), dtype=dt, device=DEV)
    X = buf.as_strided((N, D), (ld, 1))
    X.copy_(case["X"].torch(DEV))
    X64 = case["X"].f64()
    s = vl.velora_subtoken_sum(X, Dsub, s=guard.vec(Dsub))
    M = vl.num_subtokens(D, Dsub)
    padded = np.zeros((N, M * Dsub))
    padded[:, :D] = X64
    assert_matches(s, padded.reshape(N * M, Dsub).sum(0), TOL_Z, "s")
    v = vl.velora_init_v(X, Dsub)
    v64 = to_f64(v)
    ref = oracle.compress(X64, v64)
    Z = vl.velora_compress(X, v, Z=guard.mat(N, M, torch.float32, ld=M + pad))
    assert_matches(Z, ref, TOL_Z, "Z")
    Zh = vl.velora_compress(X, v, Z=guard.mat(N, M, torch.bfloat16, ld=M + pad))
    assert_matches(Zh, ref, TOL_Z, "Z in bf16")
    Z8 = vl.velora_compress(X, v, Z=guard.mat(N, M, torch.uint8, ld=M + pad))
    # one code either way of the rounded reference: an eighth of the value, or the subnormals' step
    assert bool(((Z8.view(F8).double() - Z.to(F8).double()).abs() <= torch.clamp(Z.double().abs() / 8, min=2.0 ** -9)).all())
    assert float((Z8 != Z.to(F8).view(torch.uint8)).double().mean()) < 1e-3
    for z, what in ((Z, "fp32"), (Zh, "bf16"), (Z8, "E4M3")):
        if dtype == "f32" and z is not Z:
            continue
        z64 = to_f64(z.view(F8).float() if z is Z8 else z)
        Xhat = vl.velora_reconstruct(z, v, D, Xhat=guard.mat(N, D, dt, ld=ld))
        assert_matches(Xhat, oracle.reconstruct(z64, v64, D), TOL_Z, "Xhat from " + what)
    W0 = torch.randn((N, D), device=DEV).to(dt)
    for beta in (0, 1):
        W = vl.velora_expand_p(Z, v, D, dW=guard.mat(N, D, dt, ld=ld, init=W0), beta=beta)
        assert_matches(W, oracle.reconstruct(to_f64(Z), v64, D) + beta * to_f64(W0), TOL_Z, "W + P v", c=2e-3)


def _replayed_us(call):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(10):
                call()
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(5):
            start.record()
            graph.replay()
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 100)
    return best


# 16 rows are 1/512 of 8192 and bound by latency.  With a warp per row they took 0.9 of the time of 8192 (expansion), 0.23 (compress)
# and 0.26 (reconstruct); cut into runs, 0.02 to 0.06.
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_a_few_long_rows_take_a_fraction_of_the_time_of_many(vl, dtype):
    D, Dsub = 11005, 64
    M = vl.num_subtokens(D, Dsub)
    v = torch.full((Dsub,), Dsub ** -0.5, device=DEV)
    us = {}
    for N in (16, 8192):
        X, Xhat = torch.randn((N, D), device=DEV).to(dtype), torch.zeros((N, D), dtype=dtype, device=DEV)
        Z = torch.randn((N, M), device=DEV)
        us[N] = [_replayed_us(lambda: vl.velora_compress(X, v, Z=Z)), _replayed_us(lambda: vl.velora_reconstruct(Z, v, D, Xhat=Xhat)),
                 _replayed_us(lambda: vl.velora_expand_p(Z, v, D, dW=Xhat, beta=1))]
    for name, few, many in zip(("compress", "reconstruct", "expansion"), us[16], us[8192]):
        assert few < many / 8, "%s: %.1f us for 16 rows, %.1f for 8192" % (name, few, many)
