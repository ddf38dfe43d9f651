"""Retired binary64 caches are taken over by the next forward of the same shape:
results stay those of a fresh cache when shapes, streams and threads change
hands, and ozaki2_release_cache gives the memory back."""
import threading

import pytest

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


def _step(seed, M, N, K):
    from paper_2609_27831_gb300.autograd import ozaki_matmul
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g).requires_grad_()
    B = torch.randn(K, N, dtype=torch.float64, device="cuda", generator=g).requires_grad_()
    dC = torch.randn(M, N, dtype=torch.float64, device="cuda", generator=g)
    C = ozaki_matmul(A, B)
    return (C.detach(), *torch.autograd.grad(C, (A, B), dC))


SHAPES = [(70, 50, 90), (129, 64, 33), (70, 50, 90), (1, 7, 300)]


def test_reused_caches_give_the_fresh_results(ozk):
    want = []
    for i, s in enumerate(SHAPES):
        ozk.lib().ozaki2_release_cache()
        want.append(_step(i, *s))
    torch.cuda.synchronize()
    for rep in range(3):                                   # on other streams, without waiting between them
        got = []
        for i, s in enumerate(SHAPES):
            with torch.cuda.stream(torch.cuda.Stream()):
                got.append(_step(i, *s))
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            assert all(torch.equal(x, y) for x, y in zip(a, b))


def test_threads_never_share_a_cache(ozk):
    want = [_step(i, 64, 48, 80) for i in range(4)]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(10):
                got = _step(i, 64, 48, 80)
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(x, y) for x, y in zip(got, want[i])):
                    bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not bad


def test_release_gives_the_memory_back(ozk):
    _step(0, 1500, 1500, 1500)
    torch.cuda.synchronize()
    ozk.lib().ozaki2_release_cache()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    _step(1, 1500, 1500, 1500)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] < free0 - (100 << 20)   # kept for the next step
    ozk.lib().ozaki2_release_cache()
    assert torch.cuda.mem_get_info()[0] >= free0 - (16 << 20)
