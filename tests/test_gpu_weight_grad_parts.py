"""The factor P = dY^T Z on the tensor cores to fp32 accuracy (fp32 dY, bf16 dY on odd rows): edges of slices, stages and tiles,
every storage of Z, and values that the bf16 parts cannot carry.  Bound: fp32 sums of N terms as in ``test_gpu_fp32_products``."""
import pytest
import torch

from _util import Guard, assert_matches

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


def _inputs(N, O, M, dtype, z, pad, offset, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    dY = torch.full((offset + N * (O + pad),), float("nan"), device=DEV, dtype=dtype).as_strided((N, O), (O + pad, 1), offset)
    dY.copy_(torch.randn((N, O), generator=gen, device=DEV))
    return dY, torch.randn((N, M), generator=gen, device=DEV).to(z)


# 16 sub-tokens and one column over a tile, the last slice one token; 17 and 32 sub-tokens; one token less than whole stages.
@pytest.mark.parametrize("N,O,M", [(3009, 4993, 16), (3841, 1153, 17), (8191, 383, 32), (1600, 11001, 3)])
@pytest.mark.parametrize("dtype,pad,offset", [(torch.bfloat16, 0, 0), (torch.bfloat16, 2, 3), (torch.float32, 0, 0), (torch.float32, 3, 0), (torch.float32, 7, 1)])
@pytest.mark.parametrize("z", [torch.float32, torch.bfloat16, torch.float8_e4m3fn])
def test_factor(vl, guard, N, O, M, dtype, pad, offset, z):
    dY, Z = _inputs(N, O, M, dtype, z, pad, offset, N + M)
    ws = guard.workspace(vl, vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, N, 16 * M, O, 16))
    ref = dY.double().T @ Z.double()
    P0 = torch.randn((O, M), device=DEV)
    for beta in (0, 1):
        P = guard.mat(O, M, torch.float32, ld=M + 1, init=P0)
        vl.velora_weight_grad_p(dY, Z, 16 * M, 16, P=P, beta=beta, ws=ws)
        assert_matches(P, (ref + beta * P0.double()).cpu().numpy(), 1e-6, "P", c=3.84 * N * 2.0 ** -24)
    assert vl.velora_workspace_status(ws) == 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_values_that_the_parts_cannot_carry(vl, guard, dtype):
    N, O, M = 4000, 1301, 9
    dY, Z = _inputs(N, O, M, dtype, torch.float32, 0, 0, 7)
    dY[5, 3], dY[6, 700], dY[6, 1300], dY[7, 1300] = float("inf"), float("nan"), float("inf"), float("-inf")
    dY[:, 10] = 0.0
    dY[:, 11] *= 2.0 ** -118
    Z[100, 2], Z[3999, 8] = float("-inf"), float("nan")
    P = guard.mat(O, M, torch.float32)
    vl.velora_weight_grad_p(dY, Z, 16 * M, 16, P=P)
    y, z = dY.double(), Z.double()
    ref = y.T @ z
    assert torch.equal(P.isnan(), ref.isnan())
    assert torch.equal(torch.where(P.isinf(), P, 0.0), torch.where(ref.isinf(), ref, 0.0).float())
    fin = ref.isfinite()
    scale = y.abs().nan_to_num(0, 0, 0).T @ z.abs().nan_to_num(0, 0, 0)
    # N roundings of 2^-24 at most, and numbers below the smallest normal fp32 one to its last place
    assert bool(((P.double() - ref).abs()[fin] <= (N * 2.0 ** -24 * scale + 2.0 ** -140)[fin]).all())


# One sub-token block of 16 columns of Z and one of 32; the last slice ragged.
@pytest.mark.parametrize("N,D,O,Dsub", [(4001, 1024, 3003, 64), (2200, 2048, 9001, 64)])
def test_packed_copy_gives_the_same_bits(vl, N, D, O, Dsub):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(N)
    dY, Z = _inputs(N, O, D // Dsub, torch.bfloat16, torch.float32, 0, 0, N)
    W = torch.randn((O, D), generator=gen, device=DEV).bfloat16()
    v = torch.randn(Dsub, generator=gen, device=DEV)
    _, dW = vl.velora_linear_backward(dY, W, Z, v)                      # packs dY for dX
    alone = vl.velora_weight_grad(dY, Z, v, D, ws=vl.velora_workspace_alloc(
        vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, N, D, O, Dsub), DEV))
    assert torch.equal(dW, alone)


@pytest.mark.parametrize("dtype,pad", [(torch.bfloat16, 2), (torch.bfloat16, 0), (torch.float32, 0), (torch.float32, 3)])
@pytest.mark.parametrize("ey,ez", [(0, -140), (30, -140), (70, -128), (60, -120), (-120, 60), (-70, -70)])
@pytest.mark.parametrize("where", ["operand", "token", "element"])
def test_very_small_operands(vl, guard, dtype, pad, ey, ez, where):
    """Numbers whose last bits no bf16 part holds against partners that make them show: a whole operand of them, whole tokens, single
    elements among ordinary ones."""
    N, O, M = 4000, 1301, 9
    dY, Z = _inputs(N, O, M, dtype, torch.float32, pad, 0, 9)
    small, large, e, f = (Z, dY, ez, ey) if ez <= ey else (dY, Z, ey, ez)
    large *= 2.0 ** f
    if where == "operand":
        small *= 2.0 ** e
    elif where == "token":
        small[5::3] *= 2.0 ** e
    else:
        small[::5, ::7] *= 2.0 ** e
        small[:, 8] = 0.0
        small[77, 8] = 2.0 ** e * 1.23456789
    P = guard.mat(O, M, torch.float32)
    vl.velora_weight_grad_p(dY, Z, 16 * M, 16, P=P)
    y, z = dY.double(), Z.double()
    ref = y.T @ z
    # N roundings of 2^-24 at most, and of numbers below the smallest normal fp32 one to the last place; in norm as fp32 sums have it
    assert bool(((P.double() - ref).abs() <= N * 2.0 ** -24 * (y.abs().T @ z.abs()) + N * 2.0 ** -149).all())
    if ey + ez > -100:
        for part in (slice(None), (slice(None), 8) if small is Z else 8):
            assert float((P[part].double() - ref[part]).norm() / ref[part].norm()) <= 1e-6


@pytest.mark.parametrize("dtype,pad", [(torch.bfloat16, 1), (torch.float32, 0)])
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M", [12, 24])
@pytest.mark.parametrize("what", ["magnitudes", "offset"])
def test_products_of_one_sign_add_up_as_fp32_sums_do(vl, guard, dtype, pad, z_dtype, M, what):
    """Sums that truncate show on products of one sign, where sums that round to nearest err by little more than their last rounding: 2^-24
    in norm (4.6e-8 to 5.3e-8 for fp32 multiply-adds in slices, any of these inputs)."""
    dY, Z = _inputs(12608, 768, M, dtype, z_dtype, pad, 0, 4)
    for t in (dY, Z):
        t.copy_(t.abs() if what == "magnitudes" else t + 1.0)
    P = vl.velora_weight_grad_p(dY, Z, 32 * M, 32)
    ref = dY.double().T @ Z.double()
    assert float((P.double() - ref).norm() / ref.norm()) <= 2.0 ** -24
