"""The CRT of accumulators of up to 12 digits (warp-level products of bytes, the
automatic choice there) against the tensor-core CRT of the same product
(crt_engine 1): the outputs are the same integers, compared bit for bit, at the
edges of the digit classes, the steps of 16 moduli and the blocks of 128 outputs."""
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


# with K = 5: digits 3 to 13 (classes of 8 and 12 and the first beyond), moduli 16 | 17, 32 | 33 and up to 45
@pytest.mark.parametrize("p,t", [(2, 5), (24, 24), (24, 59), (24, 60), (53, 88), (53, 89), (53, 92), (53, 93), (96, 116),
                                 (96, 117), (113, 127), (113, 139), (128, 156), (128, 157)])
@pytest.mark.parametrize("M,N", [(1, 1), (16, 8), (43, 3), (29, 53)])
def test_matches_the_tensor_core_crt(ozk, M, N, p, t):
    rng = np.random.Generator(np.random.PCG64(100 * t + M))
    A = ozk.MPMatrix.from_host(synth.mp_matrix(rng, M, 5, p, -9, 9))
    B = ozk.MPMatrix.from_host(synth.zero_rows(synth.mp_matrix(rng, 5, N, p, -9, 9), [2]))
    out = []
    for eng, mode in ((0, 0), (1, 1)):
        plan = ozk.Plan((M, N, 5, p), t_bits=t, crt_engine=eng)
        assert plan.info["crt_mode"] == mode
        ws = plan.workspace()
        ws.fill_(0x5A)
        C = ozk.MPMatrix.empty(M, N, p)
        plan.execute(A, B, C, ws)
        plan.check()
        out.append(C)
    C, D = out
    assert torch.equal(C.limbs, D.limbs) and torch.equal(C.exp, D.exp) and torch.equal(C.sign, D.sign)
