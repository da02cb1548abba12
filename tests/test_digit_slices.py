"""The digit arithmetic of csrc/gemm_digits.cu on the host: an entry as a fixed-point integer, its
signed 8-bit digits, and their recombination -- exact, in range and within half a unit."""
import math
from fractions import Fraction

import numpy as np
import pytest


def fixed_point(v, E, S):
    """v 2^(8S - 2 - E) as an integer: truncated for S = 8, rounded half up in magnitude for S = 7."""
    q = abs(Fraction(v)) * Fraction(2) ** (8 * S - 2 - E)
    f = int(q) if S == 8 else (int(2 * q) + 1) // 2
    return -f if v < 0 else f


def biased_pair(h, l, E):
    """biased<7> of a float pair in units of 2^(E - 53), in float32 steps."""
    f = np.float32
    v = f(h * f(2.0 ** (22 - E)))
    t = f(v + f(12582912.0))
    r = f(v - f(t - f(12582912.0)))
    it = int(np.array(t).view(np.int32)) - (0x4b400000 - 0x01010101)
    ib = int(np.rint(f(r * f(2147483648.0)))) + int(np.rint(f(l * f(2.0 ** (53 - E))))) + 0x00808080
    assert -2 ** 31 <= ib < 2 ** 31
    return (it * 2147483648 + ib) % 2 ** 64


def digits(biased, S):
    return [((biased >> (8 * (S - 1 - a))) & 0xff) - 128 for a in range(S)]


BIAS = {8: 0x8080808080808080, 7: 0x0080808080808080}


@pytest.mark.parametrize("S", [7, 8])
def test_fp64_entries_recombine(S):
    rng = np.random.default_rng(1)
    vals = [0.0, 1.0, -1.0, np.nextafter(2.0, 0), -np.nextafter(2.0, 0), 2.0 ** -60, 5e-324, 1e-310]
    vals += list(rng.uniform(-2, 2, 300)) + list(rng.standard_normal(300) * 2.0 ** rng.uniform(-40, 0, 300))
    for v in vals:
        if abs(v) >= 2:
            continue
        f = fixed_point(v, 1, S)
        d = digits((f + BIAS[S]) % 2 ** 64, S)
        assert all(-128 <= x <= 127 for x in d)
        assert sum(x * 256 ** (S - 1 - a) for a, x in enumerate(d)) == f
        assert abs(Fraction(f) * Fraction(2) ** (1 - (8 * S - 2)) - Fraction(v)) <= Fraction(2) ** (1 - (8 * S - 2))


def test_float_pairs_recombine():
    rng = np.random.default_rng(2)
    vals = list(rng.uniform(-1, 1, 2000) * 2.0 ** rng.uniform(-30, 0, 2000))
    vals += [1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53), 0.5, 0.25 + 2.0 ** -26, 2.0 ** -23 * 1.5, 0.0]
    for v in vals:
        h = np.float32(v)
        l = np.float32(v - float(h))
        d = digits(biased_pair(h, l, 1), 7)
        got = Fraction(sum(x * 256 ** (6 - a) for a, x in enumerate(d))) * Fraction(2) ** (1 - 53)
        want = Fraction(float(h)) + Fraction(float(l))
        assert abs(got - want) <= Fraction(2) ** (1 - 53)   # two roundings of half a unit


def test_accumulators_stay_exact():
    # 128 atoms, up to 8 digit products of at most 2^14 per weight, and the 32-bit combinations
    assert 128 * 8 * 128 * 128 <= 2 ** 24
    s = [(w + 1) * 128 * 2 ** 14 for w in range(8)]
    assert s[0] * 256 + s[1] < 2 ** 31 and s[2] * 256 + s[3] < 2 ** 31
    # S = 7: weights 4 to 6 as one float in units of 2^-7 of weight 4 fits 31 bits
    assert s[4] * 128 + s[5] // 2 + s[6] // 512 < 2 ** 31
    assert math.log2(s[0]) + 24 + math.log2(2 ** 21 / 128) < 63   # sums of 2^21 atoms


def _worst(S):
    """Fixed-point integers whose digits are all extreme (127 or -128), and random ones."""
    rng = np.random.default_rng(S)
    out = []
    for pick in ([127] * S, [-128] * S, [127, -128] * 4, [-128, 127] * 4):
        d = [max(-63, min(63, pick[0]))] + list(pick[1:S])
        out.append(sum(v * 256 ** (S - 1 - a) for a, v in enumerate(d)))
    out += [int(v) for v in rng.integers(-2 ** 53, 2 ** 53, 200)]
    return out


@pytest.mark.parametrize("S,u", [(8, -58), (7, -50)])
def test_what_a_product_leaves_out(S, u):
    """D_ij x_j from the digit products with a + b < S and the last digits of both operands: within
    2^u of the bounds' product, the constant of csrc/digit_cols.cuh's threshold."""
    unit = Fraction(2) ** (8 * S - 2)          # operands in units of their bound / unit
    last = 1 if S == 8 else 2                  # S = 7 from float pairs: two roundings of half 2^(E - 53)
    for f in _worst(S):
        for h in _worst(S)[:40]:
            df, dh = digits((f + BIAS[S]) % 2 ** 64, S), digits((h + BIAS[S]) % 2 ** 64, S)
            kept = sum(df[a] * dh[b] * 256 ** (2 * S - 2 - a - b) for a in range(S) for b in range(S - a))
            err = abs(Fraction(kept - f * h)) / unit ** 2 + (last * abs(Fraction(h)) + abs(Fraction(f)) + last) / unit ** 2
            assert err <= Fraction(2) ** u


def test_what_a_chunk_of_one_sign_rounds():
    """S = 7: weights 4 to 6 of a 128-atom chunk as one float, all digits extreme: with the products
    left out still within 2^-50 of the bounds' product per entry."""
    for n in (1, 16, 128):
        s = [n * (w + 1) * 128 * 128 for w in range(7)]
        f = np.float32(s[6]) * np.float32(2.0 ** -9)
        f = np.float32(np.float64(s[5]) * 0.5 + np.float64(f))
        f = np.float32(np.float64(s[4]) * 128 + np.float64(f))
        exact = Fraction(s[4]) * 128 + Fraction(s[5], 2) + Fraction(s[6], 512)
        got = Fraction(int(np.rint(f)))
        # in units of 2^-7 of weight 4; weight 4 is 2^-32 of weight 0, 2^12 of which is the bound
        err = abs(got - exact) / 2 ** 7 / 2 ** 32 / 2 ** 12
        assert err + n * Fraction(6 * 2 ** 14, 2 ** 68) + n * Fraction(3, 2 ** 54) <= n * Fraction(1, 2 ** 50) + Fraction(1, 2 ** 52)


def fixed_float(v, E):
    """csrc/gemm_digits.cu's fixed_float: v 2^(61 - E), truncated, from the bits of a float."""
    b = int(np.float32(v).view(np.uint32))
    ex = (b >> 23) & 0xff
    sh = max(ex, 1) - 89 - E
    m = (b & 0x7fffff) | (0x800000 if ex else 0)
    f = m << sh if sh >= 0 else m >> min(-sh, 31)
    return -f if b >> 31 else f


def test_float_pairs_in_eight_digits():
    rng = np.random.default_rng(3)
    vals = list(rng.uniform(-1, 1, 1000) * 2.0 ** rng.uniform(-40, 0, 1000)) + [0.0, 1.0 - 2.0 ** -53, 2.0 ** -30]
    for v in vals:
        h = np.float32(v)
        l = np.float32(v - float(h))
        f = fixed_float(h, 0) + fixed_float(l, 0)
        d = digits((f + BIAS[8]) % 2 ** 64, 8)
        assert sum(x * 256 ** (7 - a) for a, x in enumerate(d)) == f and abs(d[0]) <= 64
        assert abs(Fraction(f) / 2 ** 61 - Fraction(float(h)) - Fraction(float(l))) < 2 * Fraction(1, 2 ** 61)
