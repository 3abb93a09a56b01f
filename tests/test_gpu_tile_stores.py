"""bf16 products whose outputs leave as 32 x 64 tiles: ragged last tiles, in rows and columns, must not write a byte beyond the
matrix (guard bands), in the single-CTA kernel's widths and in the CTA-pair kernel.  Bound: as for every bf16 product."""
import pytest
import torch

from _util import TOL_GEMM, Guard, assert_matches

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def vl():
    import paper_2405_17991_b200 as pkg
    pkg.lib()
    return pkg


# One element; one over and one under the block's rows and columns; a short contraction with two sets of epilogue warps and several
# tiles per CTA; tiles of 192; pairs of CTAs, one over in both directions.
@pytest.mark.parametrize("Mdim,Ndim,Kdim", [(1, 1, 8), (31, 63, 16), (33, 65, 72), (129, 200, 136), (5000, 1029, 24), (4000, 760, 1096),
                                            (2305, 2561, 520)])
@pytest.mark.parametrize("kind", [0, 1])
def test_ragged_tiles(vl, Mdim, Ndim, Kdim, kind):
    guard = Guard(DEV)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(Mdim + Ndim)
    ld = -(-Ndim // 8) * 8
    A = torch.randn((Mdim, Kdim), generator=gen, device=DEV).bfloat16()
    B = torch.zeros((Ndim, Kdim) if kind == 0 else (Kdim, ld), device=DEV, dtype=torch.bfloat16)[:, :Kdim if kind == 0 else Ndim]
    B.copy_(torch.randn(B.shape, generator=gen, device=DEV))
    C = guard.mat(Mdim, Ndim, torch.bfloat16, ld=ld + 8)
    vl.velora_dense_product(kind, A, B, C=C)
    ref = A.double() @ (B.double().T if kind == 0 else B.double())
    assert_matches(C, ref.cpu().numpy(), TOL_GEMM, "C", c=4e-3)
    guard.check()
