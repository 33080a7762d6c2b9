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
    """The kernel's digit split: v plus 1.5 2^k (and 128 units) in units of 2^-14, 2^-30, 2^-46 and
    2^-54, the remainders renormalised by fast two-sums, digits from the bytes of the sums' words.
    Every remainder is exact as rationals, every digit has |d| <= 128, and the value minus its
    expansion sum_i d_i 2^(-6-8i) is at most 2^-55 (half of the last unit)."""
    def word(x):
        return int(np.array(x, dtype=F).view(np.uint32))

    magic = [F(float.fromhex("0x1.8p9") + float.fromhex("0x1p-7")),
             F(float.fromhex("0x1.8p-7") + float.fromhex("0x1p-23")),
             F(float.fromhex("0x1.8p-23") + float.fromhex("0x1p-39")),
             F(float.fromhex("0x1.8p-31") + float.fromhex("0x1p-40"))]
    units = [Fraction(1, 2 ** e) for e in (14, 30, 46, 54)]
    for m, u, off in zip(magic, units, (128, 128, 128, 2 ** 14)):
        # exact constants: 1.5 2^23 units and the offset, in a word whose bit 23 is clear
        assert Fraction(float(m)) == u * (3 * 2 ** 22 + off) and not word(m) >> 23 & 1
    rng = np.random.default_rng(3)
    xs = _values() + [s * (2 - 2.0 ** -23) for s in (1, -1)]
    # remainders at their largest: halves of the first two units, on both sides
    xs += [float(n) * 2.0 ** -14 + s * 2.0 ** -15 + t * 2.0 ** -31
           for n in rng.integers(-20000, 20000, 200) for s in (1, -1) for t in (1, 0, -1)]
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
                ds += [((w >> 8) & 0xFFFF) - 2 ** 14, (w & 0xFF) - 128]
                assert 256 * ds[-2] + ds[-1] == n / u
                r = F(h - F(a - m))
                h = F(r + l)
                l = F(l - F(h - r))
                assert Fraction(float(h)) + Fraction(float(l)) == before - n, (x, i)
            else:
                ds.append((w & 0xFFFF) - 2 ** 14)
                assert ds[-1] == n / u
        assert all(abs(d) <= 128 for d in ds), (x, ds)
        v = Fraction(float(hi)) + Fraction(float(lo))
        expansion = sum(Fraction(d) * Fraction(1, 2 ** (6 + 8 * i)) for i, d in enumerate(ds))
        assert abs(v - expansion) <= Fraction(1, 2 ** 55), x
    # three batches of 48 stacked rows, 7 digit pairs each, stay exact in FP32
    assert 3 * 7 * 48 * 128 ** 2 < 2 ** 24
