"""The plane GEMM's v_l store where N is not a multiple of 8 (rows of v_l only
2-byte aligned, written row by row) against the TMA store of the same product
with zero columns appended up to a multiple of 8: the reduced products v_l and
the outputs are the same integers, compared bit for bit."""
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


def _padded(B, n8):
    K, N = B["exp"].shape
    out = {"p": B["p"]}
    for k in ("limbs", "exp", "sign"):
        w = [(0, 0)] * (B[k].ndim - 1) + [(0, n8 - N)]
        out[k] = np.pad(B[k], w)
    return out


def _v(plan, ws, M, N):
    off, L = plan.layout()[0][4], plan.info["L"]
    pitch = -(-M * N // 8) * 8
    u = ws[off:off + 2 * L * pitch].view(torch.int16).view(L, pitch)
    return u[:, :M * N].reshape(L, M, N)


@pytest.mark.parametrize("tile", [1, 2])
@pytest.mark.parametrize("M,N,K,p", [(1, 1, 70, 113), (33, 7, 64, 256), (130, 31, 80, 256), (129, 33, 40, 113),
                                     (257, 250, 96, 256), (160, 255, 64, 53), (70, 257, 1100, 256),
                                     (300, 517, 33, 113), (31, 1093, 65, 53)])
def test_ragged_rows_match_the_aligned_store(ozk, M, N, K, p, tile):
    rng = np.random.Generator(np.random.PCG64(M * 1000 + N))
    A, B = synth.mp_matrix(rng, M, K, p, -8, 8), synth.mp_matrix(rng, K, N, p, -8, 8)
    n8 = -(-N // 8) * 8
    Ad, out = ozk.MPMatrix.from_host(A), []
    for cols, Bh in ((N, B), (n8, _padded(B, n8))):
        plan = ozk.Plan((M, cols, K, p), gemm_tile=tile)
        ws = plan.workspace()
        ws.fill_(0x5A)
        C = ozk.MPMatrix.empty(M, cols, p)
        plan.execute(Ad, ozk.MPMatrix.from_host(Bh), C, ws)
        plan.check()
        out.append((_v(plan, ws, M, cols)[:, :, :N], C.limbs[:, :, :N], C.exp[:, :N], C.sign[:, :N]))
    for got, want in zip(*out):
        assert torch.equal(got, want)


@pytest.mark.parametrize("tile", [1, 2])
@pytest.mark.parametrize("M,K", [(31, 1100), (300, 40)])
@pytest.mark.parametrize("N", [1, 2, 32, 33, 64, 65, 96, 97, 127, 128])
def test_narrow_outputs_match_the_wide_ones(ozk, M, N, K, tile):
    """Up to 128 columns the epilogue takes the chunks that hold any; with zero columns
    appended up to 256 it takes them all."""
    rng = np.random.Generator(np.random.PCG64(M * 1000 + N))
    A, B = synth.mp_matrix(rng, M, K, 200, -8, 8), synth.mp_matrix(rng, K, N, 200, -8, 8)
    Ad, out = ozk.MPMatrix.from_host(A), []
    for cols, Bh in ((N, B), (256, _padded(B, 256))):
        plan = ozk.Plan((M, cols, K, 200), gemm_tile=tile)
        ws = plan.workspace()
        ws.fill_(0x5A)
        C = ozk.MPMatrix.empty(M, cols, 200)
        plan.execute(Ad, ozk.MPMatrix.from_host(Bh), C, ws)
        plan.check()
        out.append((_v(plan, ws, M, cols)[:, :, :N], C.limbs[:, :, :N], C.exp[:, :N], C.sign[:, :N]))
    for got, want in zip(*out):
        assert torch.equal(got, want)


def test_batch_mixes_both_stores(ozk):
    """Problems with and without TMA-storable rows alternate on the same warps'
    staging buffers; each equals its own single product."""
    rng = np.random.Generator(np.random.PCG64(77))
    shapes = [(200, n, 70, p) for n, p in ((96, 113), (97, 256), (256, 53), (131, 113), (264, 256), (77, 53))] * 3
    triples, singles = [], []
    for M, N, K, p in shapes:
        A = ozk.MPMatrix.from_host(synth.mp_matrix(rng, M, K, p, -8, 8))
        B = ozk.MPMatrix.from_host(synth.mp_matrix(rng, K, N, p, -8, 8))
        triples.append((A, B, ozk.MPMatrix.empty(M, N, p)))
        singles.append(ozk.gemm(A, B))
    plan = ozk.Plan(shapes, grid=7)
    plan.execute_batched(triples, plan.workspace())
    plan.check()
    for (_, _, C), S in zip(triples, singles):
        assert torch.equal(C.limbs, S.limbs) and torch.equal(C.exp, S.exp) and torch.equal(C.sign, S.sign)
