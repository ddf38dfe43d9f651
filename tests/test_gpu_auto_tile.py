"""The automatic plane GEMM tile: where it takes CTA pairs, the outputs are those
of the one-SM tiles bit for bit (batches, binary64), and it keeps one SM per tile
for few or badly covered tiles."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def ozk():
    from paper_2609_27831_gb300 import build
    build.build()
    import paper_2609_27831_gb300 as pkg
    return pkg


@pytest.mark.parametrize("shape,tile", [((256, 256, 256, 53), 1), ((611, 347, 923, 113), 1), ((100, 3000, 8, 256), 1),
                                        ((512, 512, 64, 256), 2), ((700, 500, 40, 512), 2)])
def test_single_products(ozk, shape, tile):
    assert ozk.Plan(shape).info["gemm_tile"] == tile
    M, N, K, p = shape
    rng = np.random.Generator(np.random.PCG64(M))
    A = ozk.MPMatrix.from_host(synth.mp_matrix(rng, M, K, p, -8, 8))
    B = ozk.MPMatrix.from_host(synth.mp_matrix(rng, K, N, p, -8, 8))
    out = []
    for t in (0, 1):
        plan = ozk.Plan(shape, gemm_tile=t)
        C = ozk.MPMatrix.empty(M, N, p)
        plan.execute(A, B, C, plan.workspace())
        plan.check()
        out.append(C)
    for k in ("limbs", "exp", "sign"):
        assert torch.equal(getattr(out[0], k), getattr(out[1], k))


def test_batch(ozk):
    rng = np.random.Generator(np.random.PCG64(5))
    shapes = [(500, 260, 40, 256), (250, 511, 33, 113), (512, 250, 70, 512), (90, 64, 20, 53), (257, 768, 4, 256)]
    mats = [(ozk.MPMatrix.from_host(synth.mp_matrix(rng, M, K, p, -8, 8)),
             ozk.MPMatrix.from_host(synth.mp_matrix(rng, K, N, p, -8, 8))) for M, N, K, p in shapes]
    out = []
    for t in (0, 1):
        plan = ozk.Plan(shapes, gemm_tile=t)
        assert plan.info["gemm_tile"] == (2 if t == 0 else 1)
        C = [ozk.MPMatrix.empty(M, N, p) for M, N, K, p in shapes]
        plan.execute_batched([(A, B, c) for (A, B), c in zip(mats, C)], plan.workspace())
        plan.check()
        out.append(C)
    for x, y in zip(*out):
        assert torch.equal(x.limbs, y.limbs) and torch.equal(x.exp, y.exp) and torch.equal(x.sign, y.sign)


@pytest.mark.parametrize("M,N,K", [(1100, 900, 70), (70, 1000, 1030), (1030, 64, 1111)])
def test_binary64_gradients_are_exact(ozk, M, N, K):
    """Integer operands, whose products binary64 holds exactly; two of the three products of a step on pairs."""
    from paper_2609_27831_gb300 import autograd as ag
    rng = np.random.Generator(np.random.PCG64(M))
    X, Y, G = (torch.tensor(rng.integers(-30000, 30000, s).astype(np.float64)) for s in ((M, K), (K, N), (M, N)))
    xa, ya = X.cuda().requires_grad_(), Y.cuda().requires_grad_()
    out = ag.ozaki_matmul(xa, ya)
    out.backward(G.cuda())
    assert torch.equal(out.detach().cpu(), X @ Y)
    assert torch.equal(xa.grad.cpu(), G @ Y.T)
    assert torch.equal(ya.grad.cpu(), X.T @ G)
