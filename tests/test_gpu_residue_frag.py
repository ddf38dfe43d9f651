"""Residues of integers of up to 72 bytes (warp-level products, the automatic
choice there) against the byte GEMM of the same integers (res_engine 2): the
planes are the same bf16 integers, compared bit for bit, at the edges of the
word classes, steps, runs and tiles."""
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


def _planes(ozk, A, B, shape, fill, **kw):
    M, N, K, p = shape
    plan = ozk.Plan(shape, **kw)
    ws = plan.workspace()
    ws.fill_(fill)
    C = ozk.MPMatrix.empty(M, N, p)
    plan.execute(A, B, C, ws)
    plan.check()
    off, kp = plan.layout()
    G = plan.info["G"]
    pa = ws[off[2]:off[2] + 2 * G * M * kp].view(torch.int16).view(G, M, kp)[:, :, :K]
    pb = ws[off[3]:off[3] + 2 * G * N * kp].view(torch.int16).view(G, N, kp)[:, :, :K]
    return plan.info["res_mode"], pa, pb, C


# t: the last of a word class and the first of the next (128, 192, 320 and 576 bits
# of t + 1), K steps of 16 bytes; K: runs of 32, steps of 128, plane lines 16 and 32
# bytes aligned; lines: one, an odd count, more than a block's eight
@pytest.mark.parametrize("p,t", [(24, 40), (53, 127), (53, 128), (64, 127), (65, 100), (113, 191), (113, 192),
                                 (128, 260), (256, 319), (256, 320), (300, 383), (300, 384), (512, 575)])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (7, 9, 33), (8, 3, 128), (17, 10, 129), (5, 18, 200), (9, 33, 31)])
def test_planes_match_the_byte_gemm(ozk, M, N, K, p, t):
    rng = np.random.Generator(np.random.PCG64(100 * t + K))
    # exponents wide enough for integers of every length, rounded at every place, and for zeros
    A = synth.zero_rows(synth.mp_matrix(rng, M, K, p, -t // 2 - 8, t // 2 + 8), [M // 2] if M > 4 else [])
    B = synth.mp_matrix(rng, K, N, p, -t - 8, 8)
    Ad, Bd = ozk.MPMatrix.from_host(A), ozk.MPMatrix.from_host(B)
    m0, pa, pb, C = _planes(ozk, Ad, Bd, (M, N, K, p), 0x5A, t_bits=t)
    m2, qa, qb, D = _planes(ozk, Ad, Bd, (M, N, K, p), 0xA5, t_bits=t, res_engine=2)
    assert (m0, m2) == (0, 2)
    assert torch.equal(pa, qa) and torch.equal(pb, qb)
    assert torch.equal(C.limbs, D.limbs) and torch.equal(C.exp, D.exp) and torch.equal(C.sign, D.sign)


@pytest.mark.parametrize("t", [63, 127, 191, 319, 575])
def test_the_largest_byte_sums(ozk, t):
    """Integers of ones, +-(2^t - 1): every byte 255 (the top one 127 at whole bytes less a bit), the
    sums at their bounds; each plane against the residue itself."""
    M, N, K, p = 9, 10, 40, t
    nl = (p + 63) // 64
    rng = np.random.Generator(np.random.PCG64(t))

    def ones(rows, cols):
        limbs = np.full((nl, rows, cols), 2 ** 64 - 1, dtype=np.uint64)
        limbs[0] = np.uint64((2 ** 64 - 1) ^ ((1 << (64 * nl - p)) - 1))
        return {"p": p, "limbs": limbs, "exp": np.zeros((rows, cols), np.int32),
                "sign": rng.integers(0, 2, (rows, cols)).astype(np.int8)}

    A, B = ones(M, K), ones(K, N)
    mode, pa, pb, _ = _planes(ozk, ozk.MPMatrix.from_host(A), ozk.MPMatrix.from_host(B), (M, N, K, p), 0x5A, t_bits=t)
    assert mode == 0
    mods = ozk.Plan((M, N, K, p), t_bits=t).moduli()
    for planes, sign in ((pa, A["sign"]), (pb, B["sign"].T)):
        v = planes.cpu().view(torch.bfloat16).to(torch.int64).numpy()
        s = np.where(sign != 0, -1, 1)
        at = 0
        for m in mods:
            r = pow(2, t, m) - 1
            if m <= 255:
                x, at = v[at], at + 1
            else:
                r0, r1, rs = v[at:at + 3]
                assert np.array_equal(rs, r0 + r1) and r0.min() > -64 and r0.max() <= 64
                x, at = r0 + 128 * r1, at + 3
            assert np.array_equal(np.mod(x, m), np.mod(s * r, m)), m
            assert 2 * x.max() <= m and 2 * x.min() > -m, m
        assert at == v.shape[0]


@pytest.mark.parametrize("gmax", [20, 61])
def test_groups_of_moduli(ozk, gmax):
    """Planes streamed in groups: fewer moduli and tiles per launch, with and without the even one."""
    rng = np.random.Generator(np.random.PCG64(gmax))
    A = ozk.MPMatrix.from_host(synth.mp_matrix(rng, 20, 70, 256, -8, 8))
    B = ozk.MPMatrix.from_host(synth.mp_matrix(rng, 70, 13, 256, -8, 8))
    out = []
    for kw in ({}, {"plane_group": gmax}):
        plan = ozk.Plan((20, 13, 70, 256), **kw)
        C = ozk.MPMatrix.empty(20, 13, 256)
        plan.execute(A, B, C, plan.workspace())
        plan.check()
        out.append((plan.info["plane_groups"], C))
    assert out[0][0] == 1 and out[1][0] > 1
    (_, C), (_, D) = out
    assert torch.equal(C.limbs, D.limbs) and torch.equal(C.exp, D.exp) and torch.equal(C.sign, D.sign)
