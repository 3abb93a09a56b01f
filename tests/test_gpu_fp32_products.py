"""fp32 products at the edges of their tiles, slices and splits, and the fp32 weight gradient of wide layers.
Bounds: an fp32 sum of K terms, ``_util``'s 3.84 * K * 2^-24 of the column's rms with K <= 1400 for the products."""
import pytest
import torch

import oracle
import velora_inputs as vi
from _util import TOL_GEMM, Guard, assert_matches, to_f64

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
C_K1400 = 3.84 * 1400 * 2.0 ** -24


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


# One element; tile edges; two shares of unequal length (9 slices of 32); eight of five slices, the last one empty; eight even ones; the
# 128-wide tile (at least 148 of them) with ragged edges in all three directions; 304 of those, which run as half tiles.
SIZES = [(1, 1, 1), (64, 64, 32), (65, 63, 33), (130, 70, 288), (130, 70, 1056), (171, 288, 1280), (40, 1000, 257), (1700, 1500, 77), (1664, 1536, 64), (2370, 2000, 50)]


@pytest.mark.parametrize("Mdim,Ndim,Kdim", SIZES)
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("pad,offset", [(0, 0), (4, 4), (1, 1)])
def test_products(vl, guard, Mdim, Ndim, Kdim, kind, pad, offset):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Mdim + Kdim)

    def mat(r, c):
        ld = c + pad
        buf = torch.full((offset + r * ld,), float("nan"), device=DEV)
        out = buf.as_strided((r, c), (ld, 1), offset)
        out.copy_(torch.randn((r, c), generator=gen, device=DEV))
        return out

    A = mat(Kdim, Mdim) if kind == vl.PRODUCT_AT_B else mat(Mdim, Kdim)
    B = mat(Ndim, Kdim) if kind == vl.PRODUCT_A_BT else mat(Kdim, Ndim)
    a = to_f64(A).T if kind == vl.PRODUCT_AT_B else to_f64(A)
    b = to_f64(B).T if kind == vl.PRODUCT_A_BT else to_f64(B)
    C0 = torch.randn((Mdim, Ndim), generator=gen, device=DEV)
    for beta in (0, 1):
        C = guard.mat(Mdim, Ndim, torch.float32, ld=Ndim + pad, init=C0)
        vl.velora_dense_product(kind, A, B, C=C, beta=beta)
        assert_matches(C, a @ b + beta * to_f64(C0), 1e-5, "C", c=C_K1400)
    C = vl.velora_dense_product(kind, A, B, C=guard.mat(Mdim, Ndim, torch.bfloat16, ld=Ndim + pad))
    assert_matches(C, a @ b, TOL_GEMM, "C in bf16", c=C_K1400)


# Column blocks of 64 with a ragged last one; 1, 2, 4 and 8 blocks of 32 sub-tokens; fewer than nine slices (added up by the
# expansion) and more; one token.
@pytest.mark.parametrize("N,D,O,Dsub", [(1, 64, 65, 16), (700, 64, 130, 32), (3000, 640, 768, 16), (2500, 1000, 200, 8), (777, 1024, 96, 4)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
def test_weight_gradient_of_wide_layers(vl, guard, N, D, O, Dsub, z_dtype):
    case = vi.small_case(5 * N + O, N, D, O, dtype="f32", mean_offset=0.1)
    X, dY = case["X"].torch(DEV), case["dY"].torch(DEV)
    v = vl.velora_init_v(X, Dsub)
    M = vl.num_subtokens(D, Dsub)
    Z = vl.velora_compress(X, v, z_dtype=z_dtype)
    c = 3.84 * 3000 * 2.0 ** -24
    need = vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, N, D, O, Dsub)
    dW0 = torch.randn((O, D), device=DEV)
    for beta in (0, 1):
        dW = guard.mat(O, D, torch.float32, init=dW0)
        vl.velora_weight_grad(dY, Z, v, D, dW=dW, beta=beta, ws=guard.workspace(vl, need))
        ref = oracle.weight_grad(case["dY"].f64(), to_f64(Z), to_f64(v), D, dW0=to_f64(dW0) if beta else None)
        assert_matches(dW, ref, 1e-5, "dW", c=c)
    P = vl.velora_weight_grad_p(dY, Z, D, Dsub, P=guard.mat(O, M, torch.float32), ws=guard.workspace(vl, need))
    assert_matches(P, case["dY"].f64().T @ to_f64(Z), 1e-5, "P", c=c)
