"""The plane GEMM epilogue's packed fp32 reductions (centered and floor
remainders, factors in 7-bit halves), restated with every operation rounded to
fp32, over the moduli of the library: exact integers in their stated ranges."""
import numpy as np
import pytest

import paper_2609_27831_gb300 as ozk

C = np.float32(12582912.0)


@pytest.fixture(scope="module")
def moduli():
    return np.array(ozk.Plan((2, 2, 2, 2048)).moduli())


def _fma(a, b, c):
    # a b is exact in binary64 (24-bit factors), and so is the sum in these ranges
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(np.float32)


def _nearest(x, by):
    return (_fma(x, by, C) - C).astype(np.float32)


def _sub_qm(x, q, m):
    return (x.astype(np.float64) - q.astype(np.float64) * m).astype(np.float32)


def _centered(x, m):
    return _sub_qm(x, _nearest(x, np.float32(1) / np.float32(m)), m)


def _floored(x, m):
    mf = np.float32(m)
    h = np.float32(np.float32(-0.5) * (mf - np.float32(1))) / mf
    w = _fma(x, np.float32(1) / mf, np.float32(h))
    return _sub_qm(x, (w + C).astype(np.float32) - C, m)


def test_floor_remainder_of_one_limb_products(moduli):
    for m in moduli[moduli < 256]:
        b = int(0.52 * m) * int(m - 1) + 1
        x = np.arange(-b, b + 1)
        assert np.array_equal(_floored(x.astype(np.float32), m).astype(np.int64), x % m)


def test_floor_remainder_of_centered_two_limb_values(moduli):
    for m in moduli[moduli >= 256]:
        b = int(0.52 * m)
        x = np.arange(-b, b + 1)
        assert np.array_equal(_floored(x.astype(np.float32), m).astype(np.int64), x % m)


def test_centered_remainder_and_factor(moduli):
    rng = np.random.default_rng(1)
    for m in moduli:
        y = np.concatenate([rng.integers(-2**24 + 1, 2**24, 4000), [2**24 - 1, 1 - 2**24, 0]])
        r = _centered(y.astype(np.float32), m)
        ri = r.astype(np.int64)
        assert np.all((ri - y) % m == 0) and np.all(np.abs(ri) <= 0.52 * m)
        if m < 256:
            continue
        for f in (1, m - 1, int(rng.integers(2, m))):                # 128 cen(x f1) + x f0
            f0, f1 = f & 127, f >> 7
            z1 = _centered((r * np.float32(f1)).astype(np.float32), m)
            z = z1.astype(np.int64) * 128 + ri * f0
            assert np.all(np.abs(z) < 2**22) and np.all(np.abs(ri * f1) < 2**22)
            c = _centered(z.astype(np.float32), m).astype(np.int64)
            assert np.all((c - y * f) % m == 0) and np.all(np.abs(c) <= 0.52 * m)
