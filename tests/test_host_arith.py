"""Host checks of two exactness claims the tensor-pipe Galerkin kernel relies on (CPU only).

1. The raw-input prefetch divides a piece index q by the pieces per site, pps = 24 k + 9, as a
   multiply-high with m = floor((2^32 - 1) / pps) + 1: floor(q m / 2^32) = floor(q / pps) for
   every q < NB pps, NB = 4 or 8, k = 1 .. 24 (checked exhaustively).
2. The base-256 digit split of a double-float value v = hi + lo (|v| < 2, normalised) into
   7 digits, d = rint(hi), then (hi - d, lo) renormalised by one fast two-sum and scaled by
   256, is exact at every step: (hi + lo) after a step equals 256 (hi + lo - d) before it, as
   rationals; every digit has |d| <= 129 (exact in bfloat16), and the value minus its digit
   expansion sum_i d_i 2^(-6-8i) is at most 2^-55 (1 + 2^-16): the last step leaves
   |hi - d + lo| <= 1/2 + 2^-17 of weight 2^-54 (2^-55 itself occurs).  The FP32 operations
   are emulated with numpy float32 scalars (IEEE round to nearest even, like the kernel's _rn
   intrinsics and rintf).
"""
from fractions import Fraction

import numpy as np

F = np.float32


def test_prefetch_index_multiply_high_is_exact():
    for k in range(1, 25):
        pps = 2 * (2 * k) * 6 + 9
        m = (0xFFFFFFFF // pps + 1) & 0xFFFFFFFF
        for nb in (4, 8):
            q = np.arange(nb * pps, dtype=np.uint64)
            h = (q * np.uint64(m)) >> np.uint64(32)
            assert np.array_equal(h, q // np.uint64(pps)), (k, nb)


def _digits(hi, lo):
    """The kernel's digit loop on float32 scalars; returns digits and the (hi, lo) trail."""
    hi, lo = F(hi) * F(64.0), F(lo) * F(64.0)
    ds, trail = [], [(hi, lo)]
    for _ in range(7):
        d = F(np.rint(hi))
        r = F(hi - d)
        h2 = F(r + lo)
        l2 = F(lo - F(h2 - r))
        hi, lo = F(h2 * F(256.0)), F(l2 * F(256.0))
        ds.append(d)
        trail.append((hi, lo))
    return ds, trail


def _values():
    rng = np.random.default_rng(12)
    x = list(rng.uniform(-2.0, 2.0, 3000))
    x += list(rng.uniform(-1.0, 1.0, 1000) * 10.0 ** rng.uniform(-12, 0, 1000))
    x += [0.0, 1.0, -1.0, 1.9999999999, -1.9999999999, 2.0 ** -40, 0.5 + 2.0 ** -30]
    return x


def test_digit_split_is_exact():
    for x in _values():
        hi = F(x)
        lo = F(x - float(hi))          # normalised double-float pair of x
        ds, trail = _digits(hi, lo)
        for i, d in enumerate(ds):
            assert abs(float(d)) <= 129 and float(d) == int(d)
            before = Fraction(float(trail[i][0])) + Fraction(float(trail[i][1]))
            after = Fraction(float(trail[i + 1][0])) + Fraction(float(trail[i + 1][1]))
            assert after == 256 * (before - Fraction(float(d))), (x, i)
        v = Fraction(float(hi)) + Fraction(float(lo))
        expansion = sum(Fraction(int(d)) * Fraction(1, 2 ** (6 + 8 * i)) for i, d in enumerate(ds))
        assert abs(v - expansion) <= Fraction(1, 2 ** 55) * (1 + Fraction(1, 2 ** 16)), x


def test_digit_products_accumulate_exactly_in_fp32():
    """One staging batch's FP32 accumulator of weight d sums at most 7 digit pairs (i + j = d)
    over the 12 NB stacked rows, each product at most 129^2 in magnitude: below 2^24, so every
    partial sum of integers is exact in FP32 (NB = 8 and 4)."""
    for nb in (8, 4):
        assert 7 * (12 * nb) * 129 ** 2 < 2 ** 24
    # the fold's weights 2^(-12-8d), d < 7, are FP32 numbers (normal, exact powers of two)
    for d in range(7):
        w = F(2.0) ** F(-12 - 8 * d)
        assert float(w) == 2.0 ** (-12 - 8 * d) and np.isfinite(w) and w > np.finfo(F).tiny


def test_tile_reciprocals_of_the_stencil_are_exact():
    """u / t = (u ceil(2^16 / t)) >> 16 for thread indices u < 128 and tile extents t <= 128, and
    b / n = high word of b (floor((2^32 - 1) / n) + 1) while b n < 2^32 (the CTA's tile index)."""
    u = np.arange(128, dtype=np.int64)
    for t in range(1, 129):
        m = (65536 + t - 1) // t
        assert np.array_equal((u * m) >> 16, u // t)
    rng = np.random.default_rng(0)
    for n in list(range(2, 200)) + [1000, 4096, 65535]:
        m = 0xFFFFFFFF // n + 1
        b = np.unique(np.concatenate([np.arange(min(4 * n, 4096)),
                                      rng.integers(0, (2 ** 32 - 1) // n, 2000)])).astype(np.uint64)
        assert np.array_equal((b * np.uint64(m)) >> np.uint64(32), b // np.uint64(n))


def test_digit_split_by_magic_sums():
    """The kernel's digit split: v plus 1.546875 2^k (and 128 units) in units of 2^-14, 2^-30, 2^-46
    and 2^-54, the remainders renormalised by fast two-sums, digits as fp16 numbers s 2^-8 from the
    bytes of the sums' words.  Every remainder is exact as rationals, every digit has |s| <= 128,
    and the value minus its expansion sum_i s_i 2^(-6-8i) is at most 2^-55 (half of the last
    unit)."""
    def word(x):
        return int(np.array(x, dtype=F).view(np.uint32))

    def half(bits, scale, off):
        """scale * (fp16 of these bits) + off, exact in fp16; returns 2^8 times it."""
        y = Fraction(float(np.array(bits, dtype=np.uint16).view(np.float16))) * scale + off
        assert Fraction(float(np.float16(float(y)))) == y
        assert (y * 256).denominator == 1
        return int(y * 256)

    magic = [F(float.fromhex("0x1.8cp9") + float.fromhex("0x1p-7")),
             F(float.fromhex("0x1.8cp-7") + float.fromhex("0x1p-23")),
             F(float.fromhex("0x1.8cp-23") + float.fromhex("0x1p-39")),
             F(float.fromhex("0x1.8p-31") + float.fromhex("0x1.18p-40"))]
    units = [Fraction(1, 2 ** e) for e in (14, 30, 46, 54)]
    for m, u, man in zip(magic, units, (0xc60080, 0xc60080, 0xc60080, 0xc04600)):
        # exact constants, in a word whose bit 23 is clear
        assert Fraction(float(m)) == u * man and not word(m) >> 23 & 1
    rng = np.random.default_rng(3)
    xs = _values() + [s * (2 - 2.0 ** -23) for s in (1, -1)]
    # remainders at their largest: halves of the first two units, on both sides
    xs += [float(n) * 2.0 ** -14 + s * 2.0 ** -15 + t * 2.0 ** -31
           for n in rng.integers(-20000, 20000, 200) for s in (1, -1) for t in (1, 0, -1)]
    half_off = Fraction(-9, 2)
    for x in xs:
        hi = F(x)
        lo = F(x - float(hi))
        ds, h, l = [], hi, lo
        for i, (m, u) in enumerate(zip(magic, units)):
            before = Fraction(float(h)) + Fraction(float(l))
            if i == 3:
                h, l = F(h + l), F(0)     # the last remainder in one word
            a = F(h + m)
            n = Fraction(float(F(a - m)))
            w = word(a)
            if i < 3:
                ds += [half((w >> 8) & 0xFFFF, 1, -6),
                       half((w >> 16) & 0xFF00 | w & 0xFF, 4 ** i, half_off)]
                assert 256 * ds[-2] + ds[-1] == n / u
                r = F(h - F(a - m))
                h = F(r + l)
                l = F(l - F(h - r))
                assert Fraction(float(h)) + Fraction(float(l)) == before - n, (x, i)
            else:
                ds.append(half(w & 0xFFFF, 1, -6))
                assert ds[-1] == n / u
        assert all(abs(d) <= 128 for d in ds), (x, ds)
        v = Fraction(float(hi)) + Fraction(float(lo))
        expansion = sum(Fraction(d) * Fraction(1, 2 ** (6 + 8 * i)) for i, d in enumerate(ds))
        assert abs(v - expansion) <= Fraction(1, 2 ** 55), x
    # three batches of 48 stacked rows, 7 digit pairs each, stay exact in FP32
    assert 3 * 7 * 48 * 128 ** 2 < 2 ** 24


def test_integer_conversions_between_float_formats():
    """The conversions that stay off the FP64 pipe, as integer operations on the words: double to
    FP32 (nearest even), double to a double-float pair, a normalised pair to double (nearest), FP32
    to double -- bit for bit what the conversions give, within the exponents they claim."""
    rng = np.random.default_rng(0)
    f2u = lambda x: int(np.array(x, dtype=F).view(np.uint32))
    u2f = lambda u: float(np.array(u, dtype=np.uint32).view(F))
    d2u = lambda x: int(np.array(x, dtype=np.float64).view(np.uint64))
    u2d = lambda u: float(np.array(u, dtype=np.uint64).view(np.float64))
    n = 4000
    x = ((rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) |
         (rng.integers(1023 - 125, 1023 + 126, n).astype(np.uint64) << np.uint64(52)) |
         rng.integers(0, 1 << 52, n, dtype=np.uint64)).view(np.float64)
    for x in list(x) + [1.5 + 2.0 ** -24, 1.5 + 3 * 2.0 ** -24, 2 - 2.0 ** -25, 2 - 2.0 ** -53]:
        x = float(x)
        q = d2u(x)
        h, l = q >> 32, q & 0xFFFFFFFF
        ex, sign = (h >> 20) & 0x7FF, h & 0x80000000
        f0, t = ((ex - 896) << 23) | ((h & 0xFFFFF) << 3) | (l >> 29), l & 0x1FFFFFFF
        f = f0 + (1 if t > 1 << 28 or (t == 1 << 28 and f0 & 1) else 0)
        assert u2f(sign | f) == float(F(x)), x
        if 949 <= ex < 949 + 201:
            up = t >> 28
            hi = u2f(sign | (f0 + up))
            lo = float(F(t - (up << 29)) * F(u2f(sign | ((ex - 948) << 23))))
            H = float(F(x))
            assert (hi, lo) == (H, float(F(x - H))) or (t == 1 << 28 and hi + lo == x), x
        hi = float(F(x))
        ulp = float(np.spacing(F(abs(hi)))) / 2
        for lo in (float(F(x - hi)), 0.0, float(F(0.3 * (x - hi))), ulp, -ulp):
            u = f2u(hi)
            a = u & 0x7FFFFFFF
            e = a >> 23
            if 80 <= e < 230:
                p = float(F(lo) * F(u2f(((306 - e) << 23) | (u & 0x80000000))))
                s = (((a & 0x7FFFFF) | 0x800000) << 29) + int(np.rint(p))
                if 1 << 52 <= s < 1 << 53:
                    w = (((u & 0x80000000) | ((e + 896) << 20) | ((s >> 32) & 0xFFFFF)) << 32)
                    assert u2d(w | (s & 0xFFFFFFFF)) == hi + lo, (hi, lo)
            w = (((u & 0x80000000) | ((a >> 3) + 0x38000000)) << 32) | ((u << 29) & 0xFFFFFFFF)
            assert u2d(w) == hi


def test_small_quotients_by_float_division():
    """The Galerkin kernel's quotients a / b (a < 2^20): the float division of a + 1/2 by b, in
    error by up to 2 units in the last place, still truncates to floor(a / b)."""
    rng = np.random.default_rng(4)
    for b in list(range(1, 130)) + [144, 288, 768, 1000, 4096, 65536]:
        a = np.concatenate([np.arange(4096), rng.integers(0, 1 << 20, 2000),
                            b * rng.integers(0, (1 << 20) // b, 500), (1 << 20) - 1 - np.arange(64)])
        q = ((a.astype(F) + F(0.5)) / F(b)).astype(F)
        for step in (-2, 0, 2):
            p = (q.view(np.int32) + step).view(F)
            assert np.array_equal(p.astype(np.int64), a // b), (b, step)
