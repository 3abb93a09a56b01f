"""fp32 products on the tensor cores (three bf16 parts per operand): edges of their tiles, several tiles per CTA pair, rows on
odd boundaries, and the values that the parts cannot carry.
Bound: that of the fp32 sums of K terms in ``test_gpu_fp32_products``; a dropped part would be 2^-17 of a product and more."""
import pytest
import torch

from _util import Guard, assert_matches, to_f64

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


def _f64(vl, kind, A, B):
    a, b = A.double(), B.double()
    return (a.T if kind == vl.PRODUCT_AT_B else a) @ (b.T if kind == vl.PRODUCT_A_BT else b)


# Tiles of 96 columns, one a pair; of 192, one a pair; three waves of tiles one over in all directions; whole tiles and k-blocks.
@pytest.mark.parametrize("Mdim,Ndim,Kdim", [(1500, 1000, 333), (3000, 1000, 130), (2561, 3073, 65), (2048, 768, 768)])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("pad,offset", [(0, 0), (4, 4), (1, 1)])
def test_products(vl, guard, Mdim, Ndim, Kdim, kind, pad, offset):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Mdim + Kdim)
    A = _mat(*((Kdim, Mdim) if kind == vl.PRODUCT_AT_B else (Mdim, Kdim)), pad, offset, gen)
    B = _mat(*((Ndim, Kdim) if kind == vl.PRODUCT_A_BT else (Kdim, Ndim)), pad, offset, gen)
    C0 = torch.randn((Mdim, Ndim), generator=gen, device=DEV)
    ref = _f64(vl, kind, A, B)
    for beta in (0, 1):
        C = guard.mat(Mdim, Ndim, torch.float32, ld=Ndim + pad, init=C0)
        vl.velora_dense_product(kind, A, B, C=C, beta=beta)
        assert_matches(C, (ref + beta * C0.double()).cpu().numpy(), 1e-6, "C", c=3.84 * Kdim * 2.0 ** -24)


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("pad", [0, 1])
def test_values_that_the_parts_cannot_carry(vl, guard, kind, pad):
    """Infinities, NaN, the largest number (infinite as bf16), rows of numbers below 2^-110 and rows of zeros come out as fp32
    arithmetic has them, and leave every other output alone."""
    Mdim, Ndim, Kdim = 1500, 1000, 200
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    a = torch.randn((Mdim, Kdim), generator=gen, device=DEV)
    b = torch.randn((Ndim, Kdim), generator=gen, device=DEV)
    a[3, 7], a[40, 0], a[41, 199], a[700, 3], a[700, 4] = float("inf"), float("-inf"), float("nan"), float("inf"), float("-inf")
    a[1499, 100] = 3.4028234663852886e38
    b[11, 5], b[999, 64] = float("inf"), float("nan")
    b[:, 100] *= 2.0 ** -20                                   # keeps the products with the largest number finite
    a[200] *= 2.0 ** -118
    a[201] = 0.0
    a[202, 9] = 2.0 ** -140                                   # one tiny number among ordinary ones
    A, B = _mat(Mdim, Kdim, pad, 0, gen), _mat(Ndim, Kdim, pad, 0, gen)
    A.copy_(a)
    B.copy_(b)
    A = A.T.contiguous() if kind == vl.PRODUCT_AT_B else A
    B = B if kind == vl.PRODUCT_A_BT else B.T.contiguous()
    C = guard.mat(Mdim, Ndim, torch.float32, ld=Ndim + pad)
    vl.velora_dense_product(kind, A, B, C=C)
    ref = a.double() @ b.double().T
    assert torch.equal(C.isnan(), ref.isnan())
    assert torch.equal(torch.where(C.isinf(), C, 0.0), torch.where(ref.isinf(), ref, 0.0).float())
    fin = ref.isfinite()
    scale = (a.double().abs().nan_to_num(0, 0, 0) @ b.double().abs().nan_to_num(0, 0, 0).T)
    err = torch.where(fin, (C.double() - ref).abs(), 0.0)
    # 200 roundings of 2^-24 at most, and numbers below the smallest normal fp32 one to its last place
    assert bool((err <= torch.where(fin, 200 * 2.0 ** -24 * scale + 2.0 ** -140, float("inf"))).all())
    assert bool((C[201][fin[201]] == 0).all())


@pytest.mark.parametrize("what", ["infinite token", "NaN token", "2^-118"])
def test_every_output_of_a_long_contraction_is_computed_again(vl, guard, what):
    """A token that is not finite, or an operand of very small numbers, takes all outputs off the tensor cores; several tiles per CTA
    pair.  None may be left out, and no wait of the kernel may run out meanwhile."""
    Kdim, Mdim, Ndim = 40000, 2300, 2310
    gen = torch.Generator(device=DEV)
    gen.manual_seed(11)
    A = torch.randn((Kdim, Mdim), generator=gen, device=DEV)
    B = torch.randn((Kdim, Ndim), generator=gen, device=DEV)
    if what == "2^-118":
        A *= 2.0 ** -118
    else:
        B[31234] = float("inf") if what == "infinite token" else float("nan")
    ws = guard.workspace(vl, 256)
    C0 = torch.randn((Mdim, Ndim), generator=gen, device=DEV) * (2.0 ** -112 if what == "2^-118" else 1.0)
    C = guard.mat(Mdim, Ndim, torch.float32, init=C0)
    vl.velora_dense_product(vl.PRODUCT_AT_B, A, B, C=C, beta=1, ws=ws)
    assert vl.velora_workspace_status(ws) == 0
    if what == "2^-118":
        ref = A.double().T @ B.double() + C0.double()
        assert_matches(C * 2.0 ** 118, (ref * 2.0 ** 118).cpu().numpy(), 1e-5, "C", c=3.84 * Kdim * 2.0 ** -24)
    elif what == "infinite token":
        assert torch.equal(C, torch.where(A[31234] > 0, float("inf"), float("-inf"))[:, None].expand(Mdim, Ndim))
    else:
        assert bool(C.isnan().all())


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("ea,eb", [(-140, 0), (-140, 30), (-128, 70), (-120, 60), (60, -120), (-100, -30), (-70, -70)])
@pytest.mark.parametrize("where", ["operand", "row", "element"])
def test_very_small_operands(vl, guard, kind, ea, eb, where):
    """Numbers whose last bits no bf16 part holds, against partners so large (or small) that those bits show in the outputs: a whole
    operand of them, a row (or column) and single elements among ordinary ones, of either operand."""
    Mdim, Ndim, Kdim = 1500, 1000, 200
    gen = torch.Generator(device=DEV)
    gen.manual_seed(3)
    a = torch.randn((Mdim, Kdim), generator=gen, device=DEV)
    b = torch.randn((Ndim, Kdim), generator=gen, device=DEV)
    small, large, e, f = (a, b, ea, eb) if ea <= eb else (b, a, eb, ea)
    large *= 2.0 ** f
    if where == "operand":
        small *= 2.0 ** e
    elif where == "row":
        small[77] *= 2.0 ** e
    else:
        small[::5, ::7] *= 2.0 ** e
        small[77] = 0.0
        small[77, 11] = 2.0 ** e * 1.23456789
    A = a.T.contiguous() if kind == vl.PRODUCT_AT_B else a
    B = b if kind == vl.PRODUCT_A_BT else b.T.contiguous()
    C = guard.mat(Mdim, Ndim, torch.float32)
    vl.velora_dense_product(kind, A, B, C=C)
    ref = a.double() @ b.double().T
    # 200 roundings of 2^-24 at most, and of numbers below the smallest normal fp32 one to the last place
    bound = 200 * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 200 * 2.0 ** -149
    assert bool(((C.double() - ref).abs() <= bound).all())
    # in norm too, as fp32 sums of 200 terms have it (2.1e-7 for ordinary numbers), where the outputs are normal numbers
    if ea + eb > -100:
        for rows in (slice(None), 77):
            r, c = (ref[rows], C[rows]) if small is a else (ref[:, rows], C[:, rows])
            assert float((c.double() - r).norm() / r.norm()) <= 4e-7
