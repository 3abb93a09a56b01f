"""Tensor-core products of few tiles: every tile width, 2, 3, 4, 5 and 8 CTAs that share a contraction, ragged in all three
directions, with accumulation, unaligned outputs, and the compress that rides on a split forward."""
import pytest
import torch

import oracle
import velora_inputs as vi
from _util import C_SUM, TOL_GEMM, TOL_Z, Guard, assert_matches, to_f64

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


# One k-block; 2 .. 8 CTAs per tile (3: rows of the exchange that do not divide evenly), with a short last share (71 and 33
# k-blocks); tiles of 64, 128, 192 and 256 columns, each alone and shared; more tiles than SMs; rows and columns that end inside a tile.
SIZES = [(100, 40, 8), (128, 64, 128), (386, 320, 9032), (615, 296, 4536), (130, 1000, 2104), (1000, 264, 1000), (300, 2000, 520),
         (2114, 576, 4096), (700, 1300, 3000), (3100, 768, 1024),
         (300, 768, 2048), (640, 1000, 3000), (640, 1000, 4096), (1500, 1000, 6000), (700, 1000, 4096), (4700, 1024, 512)]


@pytest.mark.parametrize("Mdim,Ndim,Kdim", SIZES)
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("c_dtype", [torch.bfloat16, torch.float32])
def test_products(vl, guard, Mdim, Ndim, Kdim, kind, c_dtype):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Mdim + Kdim)

    def mat(r, c):
        out = torch.full((r, -(-c // 8) * 8), float("nan"), dtype=torch.bfloat16, device=DEV)[:, :c]
        out.copy_(torch.randn((r, c), generator=gen, device=DEV))
        return out

    A = mat(Kdim, Mdim) if kind == vl.PRODUCT_AT_B else mat(Mdim, Kdim)
    B = mat(Ndim, Kdim) if kind == vl.PRODUCT_A_BT else mat(Kdim, Ndim)
    a = to_f64(A).T if kind == vl.PRODUCT_AT_B else to_f64(A)
    b = to_f64(B).T if kind == vl.PRODUCT_A_BT else to_f64(B)
    ref = a @ b
    C0 = torch.randn((Mdim, Ndim), generator=gen, device=DEV).to(c_dtype)
    for beta, ld in ((0, None), (1, None), (1, Ndim + 1)):
        C = guard.mat(Mdim, Ndim, c_dtype, ld=ld, init=C0)
        vl.velora_dense_product(kind, A, B, C=C, beta=beta)
        assert_matches(C, ref + beta * to_f64(C0), TOL_GEMM, "C", c=C_SUM)
    C1 = vl.velora_dense_product(kind, A, B, c_dtype=c_dtype)
    assert torch.equal(C1, vl.velora_dense_product(kind, A, B, c_dtype=c_dtype))


@pytest.mark.parametrize("N,D,O,Dsub", [(200, 4096, 3072, 64), (130, 1000, 2880, 8), (60, 2048, 2560, 512), (500, 1376, 4096, 1024)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
def test_forward_of_few_tiles(vl, guard, N, D, O, Dsub, z_dtype):
    case = vi.small_case(N + D, N, D, O, dtype="bf16", mean_offset=0.1)
    X, W = case["X"].torch(DEV), case["W"].torch(DEV)
    v = vl.velora_init_v(X, Dsub)
    ws = guard.workspace(vl, vl.velora_workspace_bytes(vl.OP_LINEAR_FORWARD, N, D, O, Dsub))
    Y, Z = vl.velora_linear_forward(X, W, v, Y=guard.mat(N, O), Z=guard.mat(N, vl.num_subtokens(D, Dsub), z_dtype), ws=ws)
    assert_matches(Y, oracle.linear_forward(case["X"].f64(), case["W"].f64()), TOL_GEMM, "Y")
    assert_matches(Z, oracle.compress(case["X"].f64(), to_f64(v)), TOL_Z if z_dtype == torch.float32 else TOL_GEMM, "Z")
