"""Calls whose inputs are the outputs of the call before, queued without a host synchronisation: the bits are those of the same
calls with a synchronisation after each.  Kernels start while the one before them still runs, so a missing wait, or a load
that is served from before the wait, shows here and nowhere else.  Every buffer first holds the results of other inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def vl():
    import paper_2405_17991_b200 as pkg
    pkg.lib()
    return pkg


def _mat(n, d, dtype, pad):
    return torch.full((n, d + pad), float("nan"), dtype=dtype, device=DEV)[:, :d]


def _runs_agree(run, outputs, inputs):
    """run(step) issues the calls and calls step() after each; two sets of inputs, so that what lies in the buffers is stale."""
    def both(step):
        got = []
        for seed in (1, 2, 3):
            g = torch.Generator(device=DEV)
            g.manual_seed(seed)
            fresh = [torch.randn(t.shape, generator=g, device=DEV).to(t.dtype) for t in inputs]
            for t, f in zip(inputs, fresh):
                t.copy_(f)
            for _ in range(4):
                run(step)
            got.append([t.clone() for t in outputs])
        torch.cuda.synchronize()
        return got
    queued, stepped = both(lambda: None), both(torch.cuda.synchronize)
    for a, b in zip(queued, stepped):
        for i, (x, y) in enumerate(zip(a, b)):
            assert bool(torch.isfinite(x.float()).all()), i
            assert torch.equal(x, y), "output %d: %d of %d differ" % (i, int((x != y).sum()), x.numel())


# Widths of three layers in a row: CUDA-core fp32 products (split contractions among them); tensor-core products of few tiles,
# the CTA-pair kernel and the compress inside it; packed copies and staged rows; an adapter between two wide layers.
CHAINS = [(torch.float32, 0, 300, (64, 200, 130, 64)), (torch.float32, 1, 2000, (97, 300, 771, 97)), (torch.bfloat16, 0, 200, (512, 1376, 512, 512)),
          (torch.bfloat16, 0, 2100, (512, 3072, 1024, 512)), (torch.bfloat16, 0, 130, (1000, 3000, 256, 1000)),
          (torch.bfloat16, 1, 300, (257, 1031, 515, 257)), (torch.bfloat16, 0, 1500, (768, 16, 2048, 768)), (torch.bfloat16, 3, 700, (321, 17, 640, 321))]


@pytest.mark.parametrize("dtype,pad,N,widths", CHAINS)
@pytest.mark.parametrize("z_dtype", [torch.float32, torch.bfloat16])
def test_layers_in_a_row(vl, dtype, pad, N, widths, z_dtype):
    Dsub = 16
    pairs = list(zip(widths[:-1], widths[1:]))
    W = [_mat(o, d, dtype, pad) for d, o in pairs]
    H = [_mat(N, d, dtype, pad) for d in widths]
    G = [_mat(N, d, dtype, pad) for d in widths]
    Z = [torch.empty((N, vl.num_subtokens(d, Dsub)), dtype=z_dtype, device=DEV) for d, _ in pairs]
    dW = [_mat(o, d, torch.float32, pad) for d, o in pairs]
    Xhat = _mat(N, widths[0], dtype if z_dtype == torch.float32 else torch.bfloat16, pad)
    v = torch.full((Dsub,), Dsub ** -0.5, device=DEV)
    s = torch.empty(Dsub, device=DEV)
    ops = (vl.OP_LINEAR_FORWARD, vl.OP_LINEAR_BACKWARD_FACTORED, vl.OP_WEIGHT_GRAD_FACTORED, vl.OP_INIT_V)
    ws = vl.velora_workspace_alloc(max(vl.velora_workspace_bytes(op, N, d, o, Dsub) for d, o in pairs for op in ops), DEV)

    def run(step):
        for i, w in enumerate(W):
            vl.velora_linear_forward(H[i], w, v, Y=H[i + 1], Z=Z[i], ws=ws); step()
        G[-1].copy_(H[-1] * widths[1] ** -0.5); step()
        for i in reversed(range(len(W))):
            vl.velora_linear_backward(G[i + 1], W[i], Z[i], v, dX=G[i], dW=dW[i], ws=ws); step()
        vl.velora_subtoken_sum(G[0], Dsub, s=s, ws=ws); step()
        vl.velora_compress(G[0], v, Z=Z[0]); step()
        vl.velora_reconstruct(Z[0], v, widths[0], Xhat=Xhat); step()

    _runs_agree(run, H[1:] + G + Z + dW + [s, Xhat], [H[0]] + W)


# P accumulated over micro-batches and expanded at once, rows of P sharing cache lines between CTAs (odd pitch): the expansion
# starts while the reduction of the last micro-batch still writes.
@pytest.mark.parametrize("dtype,N,D,O,Dsub,ldp", [(torch.bfloat16, 512, 1040, 1024, 16, 67), (torch.bfloat16, 300, 4096, 300, 16, 257),
                                                  (torch.float32, 200, 640, 700, 16, 41), (torch.bfloat16, 900, 768, 24, 32, 25)])
def test_accumulated_factor_and_its_expansion(vl, dtype, N, D, O, Dsub, ldp):
    M = vl.num_subtokens(D, Dsub)
    dY, Z = [_mat(N, O, dtype, 0) for _ in range(3)], [torch.empty((N, M), device=DEV) for _ in range(3)]
    P = torch.zeros((O, ldp), device=DEV)[:, :M]
    dW = _mat(O, D, torch.float32, 0)
    v = torch.full((Dsub,), Dsub ** -0.5, device=DEV)
    ws = vl.velora_workspace_alloc(vl.velora_workspace_bytes(vl.OP_WEIGHT_GRAD_FACTORED, N, D, O, Dsub), DEV)

    def run(step):
        for i in range(3):
            vl.velora_weight_grad_p(dY[i], Z[i], D, Dsub, P=P, beta=1 if i else 0, ws=ws); step()
        vl.velora_expand_p(P, v, D, dW=dW); step()

    _runs_agree(run, [P, dW], dY + Z)
