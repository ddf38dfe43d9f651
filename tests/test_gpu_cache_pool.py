"""Retired binary64 caches are taken over by the next forward of the same shape:
results stay those of a fresh cache when shapes, streams and threads change
hands.  Only their plans are kept, in bounded number; the memory that a step
worked in is given back with its graph."""
import ctypes as C
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
        ozk.release_cache()
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


def _retired(ozk):
    n, b = C.c_int(), C.c_size_t()
    assert ozk.lib().ozaki2_retired_caches(C.byref(n), C.byref(b)) == 0
    return n.value, b.value


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_a_step_gives_its_memory_back(ozk):
    """Without a call to the library: what a step worked in is torch's again when its graph is gone,
    and only the plans' tables stay."""
    _step(0, 1500, 1500, 1500)
    ozk.release_cache()
    free0 = _free()
    _step(1, 1500, 1500, 1500)
    n, tables = _retired(ozk)
    assert n == 1 and 0 < tables < (8 << 20)
    assert _free() >= free0 - (16 << 20)
    ozk.release_cache()
    assert _retired(ozk) == (0, 0)


def test_the_library_s_own_memory_is_freed(ozk):
    """The calls without an allocator: cache_destroy frees what they worked in."""
    lib, n = ozk.lib(), 1500
    A, B, D, dA, dB = (torch.randn(n, n, dtype=torch.float64, device="cuda") for _ in range(5))
    out = torch.empty_like(A)

    def step():
        h, st = C.c_void_p(), torch.cuda.current_stream().cuda_stream
        assert lib.ozaki2_dgemm_fwd(n, n, n, A.data_ptr(), n, B.data_ptr(), n, out.data_ptr(), n, None, C.byref(h), st) == 0
        assert lib.ozaki2_dgemm_bwd(h, D.data_ptr(), n, dA.data_ptr(), n, dB.data_ptr(), n, st) == 0
        return h

    assert lib.ozaki2_cache_destroy(step()) == 0
    ozk.release_cache()
    free0 = _free()
    h = step()
    assert _free() < free0 - (100 << 20)
    assert lib.ozaki2_cache_destroy(h) == 0
    assert _free() >= free0 - (16 << 20)
    X, Y = A.clone().requires_grad_(), B.clone().requires_grad_()
    from paper_2609_27831_gb300.autograd import ozaki_matmul
    Z = ozaki_matmul(X, Y)                                 # the same through torch's memory
    gX, gY = torch.autograd.grad(Z, (X, Y), D)
    assert torch.equal(Z.detach(), out) and torch.equal(gX, dA) and torch.equal(gY, dB)


def test_the_pool_is_bounded_and_keyed(ozk):
    from paper_2609_27831_gb300.autograd import ozaki_matmul
    ozk.release_cache()
    want = _step(3, 40, 24, 16)
    for i in range(40):                                    # the 33rd shape on evicts the oldest
        _step(3, 8 + i, 8, 8)
        assert _retired(ozk)[0] == min(i + 2, 32)
    assert all(torch.equal(x, y) for x, y in zip(_step(3, 40, 24, 16), want))
    ozk.release_cache()
    A = torch.randn(8, 8, dtype=torch.float64, device="cuda", requires_grad=True)
    for i, kw in enumerate(({}, {"guard_bits": 20}, {"gemm_tile": 1}, {"crt_engine": 1}, {"grid": 3})):
        ozaki_matmul(A, A, **kw).sum().backward()          # other options: never taken over
        assert _retired(ozk)[0] == i + 1
    ozaki_matmul(A, A).sum().backward()
    assert _retired(ozk)[0] == 5                           # the same: taken over and given back


def test_no_memory_is_reported(ozk):
    A = torch.randn(8, 8, dtype=torch.float64, device="cuda")
    lib, h = ozk.lib(), C.c_void_p()
    none = ozk._lib.ALLOC_FN(lambda nbytes, user: None)
    st = torch.cuda.current_stream().cuda_stream
    args = (8, 8, 8, A.data_ptr(), 8, A.data_ptr(), 8, A.clone().data_ptr(), 8, None)
    assert lib.ozaki2_dgemm_fwd_alloc(*args, none, None, C.byref(h), st) == ozk._lib.OZ2_ENOMEM and not h.value
    assert lib.ozaki2_dgemm_fwd(*args, C.byref(h), st) == 0
    d = (h, A.data_ptr(), 8, torch.empty_like(A).data_ptr(), 8, torch.empty_like(A).data_ptr(), 8)
    assert lib.ozaki2_dgemm_bwd_alloc(*d, none, None, st) == ozk._lib.OZ2_ENOMEM
    assert lib.ozaki2_dgemm_bwd(*d, st) == 0
    assert lib.ozaki2_cache_destroy(h) == 0


def test_backward_on_another_stream_and_twice(ozk):
    from paper_2609_27831_gb300.autograd import ozaki_matmul
    want = _step(5, 300, 200, 400)
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn(300, 400, dtype=torch.float64, device="cuda", generator=g).requires_grad_()
    B = torch.randn(400, 200, dtype=torch.float64, device="cuda", generator=g).requires_grad_()
    D = torch.randn(300, 200, dtype=torch.float64, device="cuda", generator=g)
    for _ in range(5):
        out = ozaki_matmul(A, B)
        first = torch.autograd.grad(out, (A, B), D, retain_graph=True)
        node = out.grad_fn
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):                         # the engine would use the forward's stream
            second = node.apply(D)[:2] if hasattr(node, "apply") else type(node).backward(node, D)[:2]
        del out, node                                      # the planes' memory goes back while they are read
        junk = [torch.full((1 << 20,), 7.0, dtype=torch.float64, device="cuda") for _ in range(8)]
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip((*first, *second), want[1:] * 2)), junk[0][0]
