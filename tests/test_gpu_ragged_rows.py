"""Rows on odd boundaries (no padding, odd pitch, offset views): the tensor-core path through packed copies, the staged
output stores, and the same calls with a workspace that has no room for the copies.

Outputs are guard-banded with the pitch under test, so a store next to a row is seen; bounds are those of ``_util``.
"""
import pytest
import torch

import oracle
import velora_inputs as vi
from _util import C_ROUNDED, TOL_GEMM, TOL_Z, Guard, assert_matches, to_f64

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


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


def _view(t, ld, offset):
    """The same values with row pitch ``ld``, starting ``offset`` elements into a buffer that ends with the last one."""
    n, d = t.shape
    buf = torch.full((offset + (n - 1) * ld + d,), float("nan"), dtype=t.dtype, device=t.device)
    out = buf.as_strided((n, d), (ld, 1), offset)
    out.copy_(t)
    return out


# N, D, O, Dsub: one tile and less, tile edges, several tiles of the CTA-pair kernel, adapter width, whole rows of
# 8-element chunks beside ragged ones, sub-tokens that are no power of two.
CASES = [(37, 257, 131, 16), (300, 321, 520, 64), (129, 200, 77, 24), (1100, 2049, 1801, 128), (2500, 640, 2731, 64), (513, 1023, 16, 32),
         (200, 130, 1031, 130)]


@pytest.mark.parametrize("N,D,O,Dsub", CASES)
@pytest.mark.parametrize("pad,offset", [(0, 0), (3, 1), (8, 4)])
@pytest.mark.parametrize("room", [True, False])
def test_layer_on_rows_that_start_anywhere(vl, guard, N, D, O, Dsub, pad, offset, room):
    if not room and N * D * O > 1 << 27:
        pytest.skip("the CUDA-core route at this size adds nothing")
    case = vi.small_case(11 * N + D, N, D, O, dtype="bf16", mean_offset=0.1)
    X, W, dY = (_view(case[k].torch(DEV), case[k].torch(DEV).shape[1] + pad, offset) for k in ("X", "W", "dY"))
    X64, W64, dY64 = (case[k].f64() for k in ("X", "W", "dY"))
    v = vl.velora_init_v(X, Dsub)
    v64 = to_f64(v)
    assert_matches(v, oracle.init_v(X64, Dsub), TOL_Z, "v")
    M = vl.num_subtokens(D, Dsub)

    def ws(op):
        nbytes = vl.velora_workspace_bytes(op, N, D, O, Dsub)
        if not room:                                     # what the same widths need with padded rows
            nbytes = 256 if op == vl.OP_LINEAR_FORWARD else vl.velora_workspace_bytes(op, N, D, -(-O // 8) * 8, Dsub)
        return guard.workspace(vl, nbytes)

    Y, Z = vl.velora_linear_forward(X, W, v, Y=guard.mat(N, O, ld=O + pad), Z=guard.mat(N, M, torch.float32), ws=ws(vl.OP_LINEAR_FORWARD))
    assert_matches(Z, oracle.compress(X64, v64), TOL_Z, "Z")
    assert_matches(Y, oracle.linear_forward(X64, W64), TOL_GEMM, "Y")
    dX, dW = vl.velora_linear_backward(dY, W, Z, v, dX=guard.mat(N, D, ld=D + pad), dW=guard.mat(O, D, ld=D + pad),
                                       ws=ws(vl.OP_LINEAR_BACKWARD_FACTORED))
    dW_ref = oracle.weight_grad(dY64, to_f64(Z), v64, D)
    assert_matches(dX, oracle.input_grad(dY64, W64), TOL_GEMM, "dX")
    assert_matches(dW, dW_ref, TOL_GEMM, "dW", c=C_ROUNDED)
    for mode, op in ((vl.WG_FACTORED, vl.OP_WEIGHT_GRAD_FACTORED), (vl.WG_EXPLICIT, vl.OP_WEIGHT_GRAD_EXPLICIT)):
        got = vl.velora_weight_grad(dY, Z, v, D, dW=guard.mat(O, D, torch.float32, ld=D + pad), mode=mode, ws=ws(op))
        assert_matches(got, dW_ref, TOL_GEMM, "dW mode %d" % mode, c=C_ROUNDED)
    P = vl.velora_weight_grad_p(dY, Z, D, Dsub, P=guard.mat(O, M, torch.float32), ws=ws(vl.OP_WEIGHT_GRAD_FACTORED))
    assert_matches(P, oracle.linear_forward(dY64.T, to_f64(Z).T), TOL_GEMM, "P", c=C_ROUNDED)


# The factored gradient of rows on odd boundaries is an fp32 sum of products with Z as stored, whatever the workspace holds:
# a Z rounded to bf16 on the way would show as 2e-3.  One slice, several, blocks of 1 .. 8 times 32 sub-tokens, more than 256
# sub-tokens (the general fp32 product), adapter width.  Bound as in the fp32 tests: 3.84 * N * 2^-24 of the column's rms.
@pytest.mark.parametrize("N,D,O,Dsub", [(37, 257, 131, 16), (1100, 2049, 1801, 128), (2500, 640, 2731, 64), (777, 1025, 97, 8), (700, 1031, 203, 4),
                                        (513, 1023, 13, 32)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("room", [True, False])
def test_factored_gradient_keeps_every_bit_of_z(vl, guard, N, D, O, Dsub, z_dtype, room):
    case = vi.small_case(13 * N + D, N, D, O, dtype="bf16", mean_offset=0.1)
    X, W, dY = (_view(case[k].torch(DEV), case[k].torch(DEV).shape[1], 1) for k in ("X", "W", "dY"))
    v = vl.velora_init_v(X, Dsub)
    M = vl.num_subtokens(D, Dsub)
    Z = vl.velora_compress(X, v, z_dtype=z_dtype)
    c = 3.84 * 2500 * 2.0 ** -24

    def ws(op):
        return guard.workspace(vl, vl.velora_workspace_bytes(op, N, D, O if room else -(-O // 8) * 8, Dsub))

    P = vl.velora_weight_grad_p(dY, Z, D, Dsub, P=guard.mat(O, M, torch.float32), ws=ws(vl.OP_WEIGHT_GRAD_FACTORED))
    assert_matches(P, case["dY"].f64().T @ to_f64(Z), 1e-5, "P", c=c)
    ref = oracle.weight_grad(case["dY"].f64(), to_f64(Z), to_f64(v), D)
    dW = vl.velora_weight_grad(dY, Z, v, D, dW=guard.mat(O, D, torch.float32, ld=D), ws=ws(vl.OP_WEIGHT_GRAD_FACTORED))
    assert_matches(dW, ref, 1e-5, "dW", c=c)
    for need_dX in (True, False):
        _, dW = vl.velora_linear_backward(dY, W, Z, v, dX=guard.mat(N, D, ld=D), dW=guard.mat(O, D, torch.float32, ld=D), need_dX=need_dX,
                                          ws=ws(vl.OP_LINEAR_BACKWARD_FACTORED))
        assert_matches(dW, ref, 1e-5, "dW of the backward", c=c)


@pytest.mark.parametrize("c_dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("Mdim,Ndim,Kdim", [(130, 259, 64), (40, 31, 264), (2600, 2051, 128)])
def test_products_add_to_an_output_with_odd_rows(vl, guard, c_dtype, Mdim, Ndim, Kdim):
    g = torch.Generator(device=DEV)
    g.manual_seed(Mdim)
    A = torch.randn((Mdim, Kdim), generator=g, device=DEV).to(torch.bfloat16)
    B = torch.randn((Ndim, Kdim), generator=g, device=DEV).to(torch.bfloat16)
    C0 = torch.randn((Mdim, Ndim), generator=g, device=DEV).to(c_dtype)
    C = guard.mat(Mdim, Ndim, c_dtype, ld=Ndim, init=C0)
    vl.velora_dense_product(vl.PRODUCT_A_BT, A, B, C=C, beta=1)
    assert_matches(C, to_f64(A) @ to_f64(B).T + to_f64(C0), TOL_GEMM, "C")


# Sub-tokens of every length class of the one-element walk (8 .. 1024), fp32 and bf16, last sub-token ragged or whole.
@pytest.mark.parametrize("N,D,Dsub", [(1, 9, 8), (37, 257, 8), (300, 1041, 16), (129, 1375, 32), (70, 2049, 64), (33, 2051, 256), (20, 3071, 1024)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("pad", [0, 3])
def test_streams_on_odd_rows(vl, guard, N, D, Dsub, dtype, pad):
    case = vi.small_case(3 * N + D, N, D, 8, dtype=dtype, mean_offset=0.1)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    X = _view(case["X"].torch(DEV), D + pad, 1)
    v = vl.velora_init_v(X, Dsub)
    assert_matches(v, oracle.init_v(case["X"].f64(), Dsub), TOL_Z, "v")
    M, v64 = vl.num_subtokens(D, Dsub), to_f64(v)
    Z = vl.velora_compress(X, v, Z=guard.mat(N, M, torch.float32))
    assert_matches(Z, oracle.compress(case["X"].f64(), v64), TOL_Z, "Z")
    Xhat = vl.velora_reconstruct(Z, v, D, Xhat=guard.mat(N, D, dt, ld=D + pad))
    assert_matches(Xhat, oracle.reconstruct(to_f64(Z), v64, D), TOL_Z, "Xhat")
    W0 = torch.randn((N, D), device=DEV).to(dt)
    W = guard.mat(N, D, dt, ld=D + pad, init=W0)
    vl.velora_expand_p(Z, v, D, dW=W, beta=1)
    assert_matches(W, oracle.reconstruct(to_f64(Z), v64, D) + to_f64(W0), TOL_Z, "W + P v", c=2e-3)


# fp32 results on odd rows are sums rounded at every step.  Positive terms: a chain of K additions, each off by 2^-24 / sqrt(3) of
# the running sum at most (rms), ends up off by 2^-24 / sqrt(3) * sqrt(K / 3) = 1.8e-6 of the result at K = 8192 and less in
# shares; twice that is allowed.  Sums that are truncated, as the tensor cores', are 3.5e-5 off.
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("Mdim,Ndim", [(130, 259), (2600, 2051)])
def test_fp32_results_on_odd_rows_are_rounded_sums(vl, guard, kind, Mdim, Ndim):
    K = 8192
    g = torch.Generator(device=DEV)
    g.manual_seed(Mdim + kind)
    mat = lambda r, c: torch.rand((r, -(-c // 8) * 8), generator=g, device=DEV).to(torch.bfloat16)[:, :c]
    A = mat(K, Mdim) if kind == vl.PRODUCT_AT_B else mat(Mdim, K)
    B = mat(Ndim, K) if kind == vl.PRODUCT_A_BT else mat(K, Ndim)
    C = vl.velora_dense_product(kind, A, B, C=guard.mat(Mdim, Ndim, torch.float32, ld=Ndim))
    a = (A.T if kind == vl.PRODUCT_AT_B else A).double()
    b = (B.T if kind == vl.PRODUCT_A_BT else B).double()
    ref = a @ b
    assert float((C.double() - ref).norm() / ref.norm()) < 3.6e-6


@pytest.mark.parametrize("dy_pad,dw_pad", [(0, 1), (1, 0), (1, 1)])
def test_explicit_fp32_gradient_on_odd_rows_is_a_rounded_sum(vl, guard, dy_pad, dw_pad):
    N, D, O, Dsub = 8192, 520, 264, 8
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    dY = _view(torch.rand((N, O), generator=g, device=DEV).to(torch.bfloat16), O + dy_pad, 0)
    Z = torch.rand((N, vl.num_subtokens(D, Dsub)), generator=g, device=DEV)
    v = torch.rand(Dsub, generator=g, device=DEV)
    dW = vl.velora_weight_grad(dY, Z, v, D, dW=guard.mat(O, D, torch.float32, ld=D + dw_pad), mode=vl.WG_EXPLICIT)
    ref = dY.double().T @ vl.velora_reconstruct(Z, v, D, x_dtype=torch.bfloat16).double()
    assert float((dW.double() - ref).norm() / ref.norm()) < 3.6e-6


# A call without a workspace allocates room for copies only where it makes them.
@pytest.mark.parametrize("dtype,pad,copies", [(torch.bfloat16, 0, True), (torch.bfloat16, 3, False), (torch.float32, 0, False)])
def test_own_workspace_of_a_call(vl, monkeypatch, dtype, pad, copies):
    from paper_2405_17991_b200 import binding
    N, D, O, Dsub = 64, 1021, 509, 16
    asked = []
    alloc = binding.velora_workspace_alloc
    monkeypatch.setattr(binding, "velora_workspace_alloc", lambda n, device: asked.append(n) or alloc(n, device))
    X, W, dY = (torch.randn((r, c + pad), device=DEV).to(dtype)[:, :c] for r, c in ((N, D), (O, D), (N, O)))
    v = torch.full((Dsub,), 0.25, device=DEV)
    _, Z = vl.velora_linear_forward(X, W, v)
    vl.velora_linear_backward(dY, W, Z, v)
    need = [vl.velora_workspace_bytes(op, N, D, O, Dsub, any_rows=copies) for op in (vl.OP_LINEAR_FORWARD, vl.OP_LINEAR_BACKWARD_FACTORED)]
    assert asked == need
