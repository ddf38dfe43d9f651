"""Gradients of the binary64 mode, whose backward turns the cached planes, at the
edges of the transpose's 64 x 64 tiles and 8-value chunks: integer operands, whose
products binary64 holds exactly, so the gradients must be exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def ag():
    from paper_2609_27831_gb300 import build
    build.build()
    from paper_2609_27831_gb300 import autograd
    return autograd


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (7, 9, 8), (63, 65, 64), (64, 64, 64), (65, 63, 72), (8, 200, 129),
                                   (129, 1, 190), (130, 257, 67)])
def test_gradients_are_exact(ag, M, N, K):
    rng = np.random.Generator(np.random.PCG64(1000 * M + N))
    X, Y, G = (torch.tensor(rng.integers(-30000, 30000, s).astype(np.float64)) for s in ((M, K), (K, N), (M, N)))
    xa, ya = X.cuda().requires_grad_(), Y.cuda().requires_grad_()
    ag.ozaki_matmul(xa, ya).backward(G.cuda())
    assert torch.equal(xa.grad.cpu(), G @ Y.T)
    assert torch.equal(ya.grad.cpu(), X.T @ G)
