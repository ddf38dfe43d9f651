"""Matrices inside larger buffers: a row stride above the columns and a limb plane
stride above the rows, which the C ABI accepts for every operand and result.  The
outputs are those of contiguous copies, bit for bit, and nothing around them is
written; through every residue and CRT kernel."""
import ctypes as C

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

FILL = 0x5A


@pytest.fixture(scope="module")
def ozk():
    from paper_2609_27831_gb300 import build
    build.build()
    import paper_2609_27831_gb300 as pkg
    return pkg


class _Strided:
    """A rows x cols matrix of nl limbs at an odd offset of filled buffers."""

    def __init__(self, ozk, rows, cols, p, pad, planes, m=None):
        nl, ld = (p + 63) // 64, cols + pad
        ps = rows * ld + planes
        buf = lambda n, dt: torch.full((n * torch.empty((), dtype=dt).element_size(),), FILL, dtype=torch.uint8,
                                       device="cuda").view(dt)
        self.raw = [buf(3 + nl * ps, torch.int64), buf(3 + ps, torch.int32), buf(3 + ps, torch.int8)]
        limbs, exp, sign = (b[3:] for b in self.raw)
        self.limbs = limbs.as_strided((nl, rows, cols), (ps, ld, 1), 3)
        self.exp, self.sign = (x.as_strided((rows, cols), (ld, 1), 3) for x in (exp, sign))
        if m is not None:
            self.limbs.copy_(m.limbs)
            self.exp.copy_(m.exp)
            self.sign.copy_(m.sign)
        self.desc = ozk._lib.Mat(limbs.data_ptr(), exp.data_ptr(), sign.data_ptr(), ld, ps)

    def untouched_around(self):
        for view, raw in zip((self.limbs, self.exp, self.sign), self.raw):
            view.zero_()
            inside = torch.zeros_like(raw)
            inside.as_strided(view.shape, view.stride(), 3).fill_(1)
            if not torch.all(raw.view(torch.uint8).view(raw.numel(), -1)[inside == 0] == FILL):
                return False
        return True


# p: residues in registers up to 72 bytes, byte GEMM beyond; CRT of up to 12 digits, one
# lane, sums with the short and the long finish
@pytest.mark.parametrize("p,kw", [(53, {}), (113, {}), (200, {}), (256, {}), (300, {}), (512, {}), (700, {}), (2048, {}),
                                  (256, {"crt_engine": 1, "res_engine": 1}), (256, {"crt_engine": 3, "res_engine": 2}),
                                  (700, {"crt_engine": 3, "res_engine": 3}), (113, {"engine": 1}), (113, {"engine": 2})])
@pytest.mark.parametrize("M,N,K,pads", [(37, 29, 70, (1, 3, 5)), (130, 40, 33, (7, 8, 1))])
def test_strided_matches_contiguous(ozk, M, N, K, pads, p, kw):
    rng = np.random.Generator(np.random.PCG64(p + M))
    A = ozk.MPMatrix.from_host(synth.zero_rows(synth.mp_matrix(rng, M, K, p, -30, 30), [3]))
    B = ozk.MPMatrix.from_host(synth.mp_matrix(rng, K, N, p, -30, 30))
    plan, want = ozk.Plan((M, N, K, p), **kw), ozk.MPMatrix.empty(M, N, p)
    ws = plan.workspace()
    plan.execute(A, B, want, ws)
    sa, sb = _Strided(ozk, M, K, p, pads[0], 11, A), _Strided(ozk, K, N, p, pads[1], 6, B)
    sc = _Strided(ozk, M, N, p, pads[2], 17)
    ozk.check(ozk.lib().ozaki2_execute(plan._h, C.byref(sa.desc), C.byref(sb.desc), C.byref(sc.desc), ws.data_ptr(),
                                       ws.numel(), torch.cuda.current_stream().cuda_stream), "ozaki2_execute")
    plan.check()
    for got, ref in zip((sc.limbs, sc.exp, sc.sign), (want.limbs, want.exp, want.sign)):
        assert torch.equal(got, ref)
    assert sa.untouched_around() and sb.untouched_around() and sc.untouched_around()
