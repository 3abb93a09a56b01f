"""Sizes that each form of a kernel takes by its rule and that the tests of single operations leave out: fp32 products of several tiles
per CTA pair and several k-blocks, the CUDA-core product's large tiles with an fp32 result, every token tile of the adapter
forward, nine to sixteen splits of a narrow layer's gradient, and kernels that hold TMEM on two streams at once."""
import pytest
import torch

import oracle
import velora_inputs as vi
from _util import C_ROUNDED, C_SUM, TOL_GEMM, TOL_Z, Guard, assert_matches, to_f64

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


def _mat(r, c, pad, offset, gen):
    ld = c + pad
    out = torch.full((offset + r * ld,), float("nan"), device=DEV).as_strided((r, c), (ld, 1), offset)
    out.copy_(torch.randn((r, c), generator=gen, device=DEV))
    return out


# On the tensor cores: three and two tiles of 192 columns a pair with four and six k-blocks, two of 96 with two, the last ones ragged in all
# directions.  On the CUDA cores, where a contraction is short: tiles of 128 x 128 (at least 148 of them) and of 64 x 128.
# Bound: fp32 sums of K terms, 3.84 * K * 2^-24 of the column's rms.
@pytest.mark.parametrize("Mdim,Ndim,Kdim", [(5000, 1500, 200), (2001, 2500, 333), (1060, 2729, 120), (1700, 1500, 20), (2305, 2050, 13), (2000, 2000, 1)])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("pad,offset", [(0, 0), (4, 4), (1, 1)])
def test_fp32_products(vl, guard, Mdim, Ndim, Kdim, kind, pad, offset):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Mdim + Kdim)
    A = _mat(*((Kdim, Mdim) if kind == vl.PRODUCT_AT_B else (Mdim, Kdim)), pad, offset, gen)
    B = _mat(*((Ndim, Kdim) if kind == vl.PRODUCT_A_BT else (Kdim, Ndim)), pad, offset, gen)
    C0 = torch.randn((Mdim, Ndim), generator=gen, device=DEV)
    a, b = A.double(), B.double()
    ref = (a.T if kind == vl.PRODUCT_AT_B else a) @ (b.T if kind == vl.PRODUCT_A_BT else b)
    for beta in (0, 1):
        C = guard.mat(Mdim, Ndim, torch.float32, ld=Ndim + pad, init=C0)
        vl.velora_dense_product(kind, A, B, C=C, beta=beta)
        assert_matches(C, (ref + beta * C0.double()).cpu().numpy(), 1e-6, "C", c=3.84 * Kdim * 2.0 ** -24)


# fp32 multiply-adds in sequence are off by 1.33e-8 * sqrt(K) in norm at the least on data like these (|N(0, 1)|: 1.22e-7 at K = 64,
# 3.74e-7 at 768, 1.48e-6 at 12608; shifted by one: 1.20e-7, 4.15e-7, 1.67e-6).
@pytest.mark.parametrize("Mdim,Ndim,Kdim", [(4096, 4096, 64), (3000, 3000, 128), (2048, 2048, 256), (2048, 768, 768), (768, 3072, 12608)])
@pytest.mark.parametrize("what", ["magnitudes", "shifted"])
def test_fp32_products_of_one_sign_are_no_further_off_than_sums_in_sequence(vl, Mdim, Ndim, Kdim, what):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Kdim)
    A, B = (torch.randn((n, Kdim), generator=gen, device=DEV) for n in (Mdim, Ndim))
    A, B = (A.abs(), B.abs()) if what == "magnitudes" else (A + 1.0, B + 1.0)
    C = vl.velora_dense_product(vl.PRODUCT_A_BT, A, B)
    ref = A.double() @ B.double().T
    assert float((C.double() - ref).norm() / ref.norm()) <= 1.33e-8 * Kdim ** 0.5


# Tiles of 24, 32, 40, 48, 56 and 64 tokens, the last one ragged; a ring of three stages at 64 outputs.
@pytest.mark.parametrize("N", [2999, 4001, 5801, 7001, 8101, 9001])
@pytest.mark.parametrize("D,O,Dsub", [(1088, 64, 32), (520, 5, 8), (1024, 16, 512)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
def test_adapter_forward(vl, guard, N, D, O, Dsub, z_dtype):
    case = vi.small_case(N + D, N, D, O, dtype="bf16", mean_offset=0.25)
    X, W = case["X"].torch(DEV), case["W"].torch(DEV)
    v = vl.velora_init_v(X, Dsub)
    ws = guard.workspace(vl, vl.velora_workspace_bytes(vl.OP_LINEAR_FORWARD, N, D, O, Dsub))
    for _ in range(2):
        Y, Z = vl.velora_linear_forward(X, W, v, Y=guard.mat(N, O), Z=guard.mat(N, vl.num_subtokens(D, Dsub), z_dtype), ws=ws)
        assert_matches(Y, oracle.linear_forward(case["X"].f64(), case["W"].f64()), TOL_GEMM, "Y")
        assert_matches(Z, oracle.compress(case["X"].f64(), to_f64(v)), TOL_Z, "Z")
    assert vl.velora_workspace_status(ws) == 0


# 13 splits of five k-blocks, 16 with a last one of four, 16 with a last one of five out of eight; the last token block one token short.
@pytest.mark.parametrize("N,D,O,Dsub", [(4159, 512, 512, 64), (5055, 512, 1100, 64), (7999, 1000, 1030, 128)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("dw_dtype", [torch.float32, torch.bfloat16])
def test_narrow_layers_gradient_of_many_splits(vl, guard, N, D, O, Dsub, z_dtype, dw_dtype):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N)
    M = vl.num_subtokens(D, Dsub)
    dY = torch.zeros((N, -(-O // 8) * 8), dtype=torch.bfloat16, device=DEV)[:, :O]
    dY.copy_(torch.randn((N, O), generator=gen, device=DEV))
    Z = torch.randn((N, M), generator=gen, device=DEV).to(z_dtype)
    v = torch.randn(Dsub, generator=gen, device=DEV)
    need = vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, N, D, O, Dsub)
    P64 = dY.double().T @ Z.double()
    c = C_SUM if z_dtype == torch.bfloat16 else C_ROUNDED
    dW0 = torch.randn((O, D), generator=gen, device=DEV).to(dw_dtype)
    for beta in (0, 1):
        ref = (P64[:, :, None] * v.double()).reshape(O, M * Dsub)[:, :D] + beta * dW0.double()
        dW = guard.mat(O, D, dw_dtype, init=dW0)
        vl.velora_weight_grad(dY, Z, v, D, dW=dW, beta=beta, ws=guard.workspace(vl, need))
        assert_matches(dW, ref.cpu().numpy(), TOL_GEMM, "dW", c=c)
    P = vl.velora_weight_grad_p(dY, Z, D, Dsub, P=guard.mat(O, M, torch.float32), ws=guard.workspace(vl, need))
    assert_matches(P, P64.cpu().numpy(), TOL_GEMM, "P", c=c)


@pytest.mark.parametrize("N,D,O,Dsub", [(4159, 512, 512, 64), (8192, 515, 1152, 64)])
def test_narrow_layers_gradient_in_the_room_of_eight_splits(vl, guard, N, D, O, Dsub):
    """Half of the partial products' room is enough, with copies of the other product's operands behind it or without."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N)
    M = vl.num_subtokens(D, Dsub)
    dY = torch.randn((N, O), generator=gen, device=DEV).bfloat16()
    W = torch.randn((O, D), generator=gen, device=DEV).bfloat16()
    Z = torch.randn((N, M), generator=gen, device=DEV).bfloat16()
    v = torch.randn(Dsub, generator=gen, device=DEV)
    ref = ((dY.double().T @ Z.double())[:, :, None] * v.double()).reshape(O, M * Dsub)[:, :D]
    dX_ref = dY.double() @ W.double()
    full = vl.velora_workspace_bytes(vl.OP_LINEAR_BACKWARD_FACTORED, N, D, O, Dsub)
    for need in (full, full - 8 * O * 16 * 4):
        ws = guard.workspace(vl, need)
        for _ in range(2):
            dX, dW = vl.velora_linear_backward(dY, W, Z, v, dX=guard.mat(N, D), dW=guard.mat(O, D), ws=ws)
            assert_matches(dX, dX_ref.cpu().numpy(), TOL_GEMM, "dX")
            assert_matches(dW, ref.cpu().numpy(), TOL_GEMM, "dW")
        assert vl.velora_workspace_status(ws) == 0


def test_kernels_with_tensor_memory_on_two_streams(vl):
    """fp32 products beside partial factors and bf16 products, none of which waits for another: what each computes alone, bit for bit."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    A, B = torch.randn((3000, 400), generator=gen, device=DEV), torch.randn((1000, 400), generator=gen, device=DEV)
    Ah, Bh = A.bfloat16(), B.bfloat16()
    odd = torch.empty((4096, 1301), dtype=torch.bfloat16, device=DEV).copy_(torch.randn((4096, 1301), generator=gen, device=DEV))
    dY, Z = torch.randn((4096, 768), generator=gen, device=DEV), torch.randn((4096, 24), generator=gen, device=DEV)
    streams = [torch.cuda.Stream(DEV) for _ in range(2)]
    ws = [vl.velora_workspace_alloc(vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, 4096, 24 * 16, 1301, 16), DEV) for _ in range(2)]

    def left(stream=None):
        return [vl.velora_dense_product(vl.PRODUCT_A_BT, A, B, ws=ws[0], stream=stream), vl.velora_dense_product(vl.PRODUCT_A_BT, Ah, Bh, ws=ws[0], stream=stream)]

    def right(stream=None):
        return [vl.velora_weight_grad_p(y, Z, 24 * 16, 16, P=torch.empty((y.shape[1], 24), device=DEV), ws=ws[1], stream=stream) for y in (odd, dY)]

    alone = left() + right()
    torch.cuda.synchronize()
    together = []
    for _ in range(20):
        for s, f in zip(streams, (left, right)):
            with torch.cuda.stream(s):
                together.append(f())
    torch.cuda.synchronize()
    for i, outs in enumerate(together):
        for x, y in zip(outs, alone[:2] if i % 2 == 0 else alone[2:]):
            assert torch.equal(x, y)
    assert all(vl.velora_workspace_status(w) == 0 for w in ws)
