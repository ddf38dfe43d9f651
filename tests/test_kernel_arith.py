"""Arithmetic facts the CUDA kernels rely on, checked exhaustively on the CPU.

The residue kernel for integers of up to 72 bytes reduces the signed byte-product
sum y (one-limb modulus m, |y| <= 72 * 255 * 250 < 2^23) in packed fp32 with
q = round(y * rcp), rcp = 1/m rounded to fp32 as the library's host code
computes it, and takes r = y - q m as the centered residue without a correction
step; for odd m that holds exactly when q = round(y / m) for every such y, which
this test checks for all odd one-limb moduli of the method (Sec. 4.3's moduli
<= 255) and every reachable |y| (rounding to nearest is odd in y).  (The form for
longer integers reduces 32-bit sums by Barrett's method and needs none of this.)
"""
import numpy as np

from oracle import ozaki2_oracle as o


def test_fp32_rounded_quotient_is_exact_for_odd_one_limb_moduli():
    mods = [m for m in o.Params(1024, 2048).moduli if m <= 255]
    assert len(mods) == 54 and sum(m % 2 == 0 for m in mods) == 1      # 128 is the even one
    amax = 72 * 255 * 250
    assert amax < 0.973 * 2 ** 23 and 72 * 255 ** 2 < 2 ** 23      # fp32 holds every partial sum
    a = np.arange(amax + 1, dtype=np.int64)
    af = a.astype(np.float64)
    for m in mods:
        if m % 2 == 0:
            continue
        rcp = np.float64(np.float32(1.0 / m))      # as the host computes it
        prod = af * rcp                            # exact in binary64 (23 x 24 bits)
        assert not np.any(prod - np.floor(prod) == 0.5), m
        q = np.rint(prod).astype(np.int64)
        q_true = (2 * a + m) // (2 * m)            # round(a / m); no ties for odd m
        assert np.array_equal(q, q_true), m
        r = a - q * m
        assert r.min() >= -(m // 2) and r.max() <= m // 2, m


def test_fp32_rounded_quotient_is_exact_for_two_limb_moduli():
    """Two-limb moduli (odd primes in (255, 16191]): the kernel reduces the
    high-byte sum hi, |hi| <= 72 * 255 * 63, with the rounded quotient, then
    y = lo + 256 r_hi, |y| <= 72 * 255^2 + 256 * 8095 < 2^23 / (1 + 2^-29), the
    same way.  Exhaustive over that |y| (the larger range) for the smallest, the
    largest and a spread of the moduli in between."""
    mods = [m for m in o.Params(1024, 2048).moduli if m > 255]
    assert all(m % 2 == 1 for m in mods)
    pick = sorted(set([mods[0], mods[-1]] + mods[:: max(1, len(mods) // 10)]))
    assert max(mods) <= 16191
    amax = 72 * 255 * 255 + 256 * 8095
    assert amax * (1 + 2.0 ** -29) < 2 ** 23
    assert max(m >> 8 for m in mods) == 63 and 72 * 255 * 63 < amax
    a = np.arange(amax + 1, dtype=np.int64)
    af = a.astype(np.float64)
    for m in pick:
        rcp = np.float64(np.float32(1.0 / m))
        q = np.rint(af * rcp).astype(np.int64)
        assert np.array_equal(q, (2 * a + m) // (2 * m)), m


def test_ties_of_the_even_modulus_are_flipped():
    """m = 128, whose reciprocal and quotients are exact: rounding to nearest even
    leaves -64 for some multiples of 64, and only there; the kernel flips the sign
    of that bf16 value (-m/2, bits 0xC280) into +64."""
    y = np.arange(-72 * 255 * 250, 72 * 255 * 250 + 1, dtype=np.int64)
    r = y - 128 * np.rint(y / 128.0).astype(np.int64)
    assert r.min() == -64 and r.max() == 64 and np.all((y[r == -64] & 127) == 64)
    assert np.float32(-64.0).view(np.uint32) >> 16 == 0xC280
    flipped = np.where(r == -64, 64, r)
    assert np.array_equal(np.mod(flipped - y, 128), np.zeros_like(y)) and flipped.min() == -63


def test_byte_sums_of_the_crt_stay_exact():
    """The CRT of up to 12 digits: v_l and the bytes of M_l (and of floor(2^32 / m_l))
    below 2^8 and at most 48 moduli, so fp32 sums below 48 * 254 * 255 < 2^22; a digit's
    four byte sums y0 + 2^8 y1 fit 32 bits and lo + 2^16 hi 64, biased by 2^23's bits."""
    top = 48 * 254 * 255
    assert top < 2 ** 22
    bias = (0x4B000000 + (0x4B000000 << 8)) & 0xFFFFFFFF
    for y0, y1 in ((0, 0), (top, top), (1, top), (top, 0)):
        bits = [int(np.float32(y + 8388608.0).view(np.uint32)) for y in (y0, y1)]
        assert bits[0] == 0x4B000000 + y0
        assert (bits[0] + (bits[1] << 8) - bias) & 0xFFFFFFFF == y0 + (y1 << 8) < 2 ** 32
    assert sum(m <= 255 for m in o.Params(1024, 2048).moduli) >= 48


def test_tensor_core_two_limb_reduction_needs_no_correction():
    """The warp-specialised tensor-core residues reduce a two-limb modulus
    from the byte sums y0 (table halves |T0| <= 64) and y1 (|T1| <= 63) of at
    most 265 bytes: r1 = y1 - RN(y1 rcp) m, x = y0 + 128 r1, r = x - RN(x rcp) m,
    with no correction step.  Exhaustive over every |y1| <= 265 * 255 * 63 and
    every |x| <= 265 * 255 * 64 + 128 * 8095 for a spread of the moduli: the
    rounded quotient is round(y / m) and the remainder the centered residue."""
    mods = [m for m in o.Params(1024, 2048).moduli if m > 255]
    pick = sorted(set([mods[0], mods[-1]] + mods[:: max(1, len(mods) // 8)]))
    y1max = 265 * 255 * 63
    xmax = 265 * 255 * 64 + 128 * 8095
    assert max(y1max, xmax) < 2 ** 23
    for bound in (y1max, xmax):
        y = np.arange(-bound, bound + 1, dtype=np.int64)
        yf = y.astype(np.float64)
        for m in pick:
            rcp = np.float64(np.float32(1) / np.float32(m))     # RN(1/m), as the host computes it
            assert rcp == np.float64(np.float32(1.0 / m))
            q = np.rint(yf * rcp).astype(np.int64)              # y rcp is exact in binary64
            r = y - q * m
            assert r.min() >= -(m - 1) // 2 and r.max() <= (m - 1) // 2, m
            assert np.array_equal(np.mod(r - y, m), np.zeros_like(y)), m


def test_balanced_split_by_shifted_rounding():
    """split128: hi = RN((r - 0.5) / 128), lo = r - 128 hi is the balanced
    base-128 split (lo in (-64, 64]) for every |r| <= 8095."""
    r = np.arange(-8095, 8096, dtype=np.int64)
    h = (r.astype(np.float64) - 0.5) / 128.0
    assert not np.any(h - np.floor(h) == 0.5)
    hi = np.rint(h).astype(np.int64)
    lo = r - 128 * hi
    assert lo.min() == -63 and lo.max() == 64
    assert np.array_equal(lo + 128 * hi, r)


def _byte_perm(x, y, sel):
    """Byte permute: result byte n is byte (sel >> 4 n) & 7 of the pair
    (x low, y high), as the CUDA byte-permute intrinsic defines it."""
    src = [(x >> (8 * i)) & 0xFF for i in range(4)] + [(y >> (8 * i)) & 0xFF for i in range(4)]
    return sum(src[(sel >> (4 * n)) & 7] << (8 * n) for n in range(4))


def _f16_bits(v):
    """f16 bits derived from the value alone (sign, 5-bit exponent with bias
    15, 10 mantissa bits) for an integer |v| < 2^11."""
    if v == 0:
        return 0
    sgn = 0x8000 if v < 0 else 0
    a = abs(v)
    e = a.bit_length() - 1
    return sgn | ((15 + e) << 10) | (((a << 10) >> e) & 0x3FF)


def _f16(bits):
    return np.array([bits], dtype=np.uint16).view(np.float16)[0]


def _h2(word):
    return _f16(word & 0xFFFF), _f16(word >> 16)


def test_f16_bytes_of_the_tensor_core_residue_builders():
    """Both tensor-core residue kernels feed the bytes of |a_hat| to the MMA
    as f16.  The byte permute with 0x64646464 puts byte b under the exponent
    bits of 2^10 (0x64xx is 1024 + b: the mantissa's unit is 1 there); then
    the unsigned form subtracts 1024 (packed) and the signed form takes one
    packed fma with {s, s} and {-1024 s, -1024 s}.  Every intermediate is an
    integer below 2^11, so each step is exact in f16; checked for every byte,
    byte position and sign against f16 bits derived from the value."""
    for v in (1, 127, -64, 255, 1024, 1279, -1279):
        assert float(_f16(_f16_bits(v))) == v                   # the bits rule itself
    m1024 = _f16(0x6400)
    assert float(_f16(0x3C00)) == 1.0 and float(m1024) == 1024.0
    for sel, lo_pos in ((0x5140, 0), (0x7362, 2)):
        for b in range(256):
            for other in (0x00, 0xFF, 0x5A):
                x = (b << (8 * lo_pos)) | (other << (8 * (lo_pos + 1)))
                x |= 0xA5A50000 if lo_pos == 0 else 0x0000A5A5     # the bytes the selector skips
                lo, hi = _h2(_byte_perm(x, 0x64646464, sel))
                assert float(lo) == 1024 + b and float(hi) == 1024 + other
                # unsigned: one packed subtraction of {1024, 1024}
                u = (np.float16(lo - m1024), np.float16(hi - m1024))
                assert [int(t.view(np.uint16)) for t in u] == [_f16_bits(b), _f16_bits(other)]
                # signed: fma(p, s, -1024 s); the product and the sum are exact
                for s2, c2, sg in ((0x3C003C00, 0xE400E400, 1), (0xBC00BC00, 0x64006400, -1)):
                    s_lo, c_lo = _h2(s2)[0], _h2(c2)[0]
                    assert float(s_lo) == sg and float(c_lo) == -1024 * sg
                    r = np.float16(np.float16(lo * s_lo) + c_lo)
                    assert int(r.view(np.uint16)) == _f16_bits(sg * b)   # +0, never -0, for b = 0
