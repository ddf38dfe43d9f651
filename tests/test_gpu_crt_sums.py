"""The CRT sums on the tensor cores (crt_engine 2) against the CRT by a lane or
lanes per output (crt_engine 3: 64-bit multiply-adds of the digits of M_l, up to 12
digits byte products with a table of their own) of the same product: the outputs
are the same integers, compared bit for bit, at the edges of the sums kernel's K
blocks, column chunks, rings and tiles."""
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


def _operands(ozk, M, N, K, p, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return (ozk.MPMatrix.from_host(synth.mp_matrix(rng, M, K, p, -30, 30)),
            ozk.MPMatrix.from_host(synth.mp_matrix(rng, K, N, p, -30, 30)))


def _same(x, y):
    return torch.equal(x.limbs, y.limbs) and torch.equal(x.exp, y.exp) and torch.equal(x.sign, y.sign)


# t = p + 7 sets L and the columns formed.  Moduli: 32 | 33, 64 | 65, 96 | 97 and
# 128 | 129 (one to five K blocks, a last block of one modulus); columns formed:
# 64 to 256 (one chunk), 288 to 384 (two), from the first group on at p = 2048 up
# to t_bits 1270; the table in the ring (up to 6 K blocks at 224 columns) or
# streamed; t_bits 2111: the most moduli.
@pytest.mark.parametrize("p,kw", [(95, {}), (99, {}), (228, {}), (234, {}), (451, {}), (458, {}), (672, {}),
                                  (675, {}), (932, {}), (961, {}), (1119, {}), (1299, {}), (1410, {}), (1783, {}),
                                  (1858, {}), (2037, {}), (2048, {}), (53, {"t_bits": 2111}),
                                  (2048, {"t_bits": 869}), (2048, {"t_bits": 1100}), (2048, {"t_bits": 1270}),
                                  (2048, {"t_bits": 1271}),
                                  (2048, {"t_bits": 2111})])
@pytest.mark.parametrize("M,N", [(16, 8), (13, 11), (37, 531)])
def test_sums_match_the_crt_per_output(ozk, M, N, p, kw):
    A, B = _operands(ozk, M, N, 12, p, 1000 * p + N)
    out = []
    for eng, mode in ((3, 0), (2, 2)):
        plan = ozk.Plan((M, N, 12, p), crt_engine=eng, **kw)
        assert plan.info["crt_mode"] == mode
        ws = plan.workspace()
        ws.fill_(0x5A)
        C = ozk.MPMatrix.empty(M, N, p)
        plan.execute(A, B, C, ws)
        plan.check()
        out.append(C)
    assert _same(*out)


@pytest.mark.parametrize("p", [256, 700, 2048])
def test_several_tiles_per_block(ozk, p):
    """More tiles than SMs: three or four per block, accumulator slots and rings reused."""
    A, B = _operands(ozk, 250, 251, 8, p, p)
    out = []
    for eng, mode in ((3, 0), (2, 2)):
        plan = ozk.Plan((250, 251, 8, p), crt_engine=eng)
        assert plan.info["crt_mode"] == mode
        C = ozk.MPMatrix.empty(250, 251, p)
        plan.execute(A, B, C, plan.workspace())
        plan.check()
        out.append(C)
    assert _same(*out)


def test_many_short_runs(ozk):
    """More problems than SMs, of one tile to three: a block's next tile lies many runs ahead."""
    ps = (113, 256, 300, 512, 700)
    shapes = [((16, 8), (13, 11), (17, 17))[i % 3] + (4, ps[i % 5]) for i in range(400)]
    triples, singles = [], []
    for i, (M, N, K, p) in enumerate(shapes):
        A, B = _operands(ozk, M, N, K, p, i)
        triples.append((A, B, ozk.MPMatrix.empty(M, N, p)))
        singles.append(ozk.gemm(A, B, crt_engine=3))
    plan = ozk.Plan(shapes, crt_engine=2)
    plan.execute_batched(triples, plan.workspace())
    plan.check()
    for (_, _, C), S in zip(triples, singles):
        assert _same(C, S)


def test_batch_mixes_tables(ozk):
    """Runs of tiles of different problems on one block: resident and streamed tables, one and two
    column chunks in a launch sized by the longest, a run shorter than the grid."""
    shapes = [(130, 100, 6, 2048), (16, 8, 6, 113), (150, 151, 6, 256), (90, 170, 6, 1024), (33, 17, 6, 2048),
              (200, 140, 6, 512), (140, 150, 6, 1410), (16, 8, 6, 300)]
    triples, singles = [], []
    for i, (M, N, K, p) in enumerate(shapes):
        A, B = _operands(ozk, M, N, K, p, i)
        triples.append((A, B, ozk.MPMatrix.empty(M, N, p)))
        plan = ozk.Plan((M, N, K, p), crt_engine=3)
        assert plan.info["crt_mode"] == 0
        singles.append(ozk.MPMatrix.empty(M, N, p))
        plan.execute(A, B, singles[-1], plan.workspace())
        plan.check()
    plan = ozk.Plan(shapes, crt_engine=2)
    plan.execute_batched(triples, plan.workspace())
    plan.check()
    for (_, _, C), S in zip(triples, singles):
        assert _same(C, S)
