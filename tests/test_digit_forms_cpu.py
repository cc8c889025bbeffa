"""The exact digit splits and the value bounds of the tensor-core kernels, emulated on the
CPU in the kernels' own steps: fix64 (seven 8-bit digits of an IEEE double,
csrc/legendre_tc64.cu), digits6 and split6 (six digits of the mixed analysis' operands,
csrc/legendre_tc_ana.cu), and bound_kernel's FP32 walk against the recursion in double on
rings up to either pole (cos theta >= 0 in every pair).
"""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest

F = np.float32


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def pow2_fraction(k):
    return Fraction(2) ** k


# ---- fix64 ------------------------------------------------------------------------------


def fix64_digits(w):
    b = bits(w)
    hw, lw = b >> 32, b & 0xFFFFFFFF
    e = (hw >> 20) & 0x7FF
    hi = ((((hw & 0xFFFFF) | 0x100000) << 10) | (lw >> 22)) & 0xFFFFFFFF
    m = (hi << 32) | ((lw << 10) & 0xFFFFFFFF)
    f = m >> max(0, min(63, 1022 - e))
    if hw >> 31:
        f = -f
    f = (f + 0x8080808080808080) & (2**64 - 1)
    return [((f >> (8 * (7 - i))) & 255) - 128 for i in range(7)]


def values(limit, n=4000):
    rng = np.random.default_rng(1)
    x = rng.uniform(-limit, limit, n) * 2.0 ** -rng.integers(0, 70, n)
    edges = [limit, np.nextafter(limit, 0), 0.5, 0.25 - 2.0**-54, 2.0**-55, 2.0**-56, 1.5 * 2.0**-56, 2.0**-57, 0.0, 1e-300, 5e-324,
             sum(127 * 2.0 ** (-7 - 8 * i) for i in range(6)), sum(128 * 2.0 ** (-7 - 8 * i) for i in range(1, 6))]
    x = np.concatenate([x, edges, -np.array(edges)])
    return x[np.abs(x) <= limit]


def test_fix64():
    for w in values(127.0 / 128):
        d = fix64_digits(float(w))
        assert all(-128 <= v <= 127 for v in d)
        got = sum(Fraction(v) * pow2_fraction(-7 - 8 * i) for i, v in enumerate(d))
        assert abs(got - Fraction(float(w))) <= pow2_fraction(-56) + pow2_fraction(-63)  # (cut to 2^-63 first)


def test_fix64_of_scaled_inputs():
    """Inputs are scaled below 1/2: the first digit stays within 64, and so do the level sums
    (512 entries, level 3's four products) within 2^25 quanta at the very worst, 2^24 up to level 2."""
    for w in values(0.5 - 2.0**-54):
        assert abs(fix64_digits(float(w))[0]) <= 64
    # level k: digits (i, k - i) of Lambda (first digit <= 121, by the bound's margin) and the input
    lam, inp = [121] + [128] * 6, [64] + [128] * 6
    sums = [sum(lam[i] * inp[k - i] for i in range(k + 1)) for k in range(4)]
    assert 512 * sums[0] <= 2**23 and 512 * sums[1] <= 2**24
    assert 256 * sums[2] <= 2**24  # analysis: 128 pairs, two values each


# ---- digits6 and split6 --------------------------------------------------------------------

QUANTA6 = [7, 15, 23, 31, 40, 49]


def digits6(x, e):
    b = bits(x)
    hi, lo = b >> 32, b & 0xFFFFFFFF
    E = (hi >> 20) & 0x7FF
    sh = max(1026 - E - e, 1)
    m = (((hi & 0xFFFFF) | 0x100000) << 32) | lo
    f = (m + (1 << (sh - 1))) >> sh if E > 0 and sh < 63 else 0
    if hi >> 31:
        f = -f
    f = (f + (1 << 41) + (1 << 33) + (1 << 25) + (1 << 17) + (1 << 8)) & (2**64 - 1)
    fh, fl = f >> 32, f & 0xFFFFFFFF
    sfh = fh - 2**32 if fh >= 2**31 else fh
    return [sfh >> 10, ((fh >> 2) & 255) - 128, (((fh << 32 | fl) >> 26) & 255) - 128, ((fl >> 18) & 255) - 128,
            ((fl >> 9) & 511) - 256, (fl & 511) - 256]


@pytest.mark.parametrize("e", [0, -300, 17, 900])
def test_digits6(e):
    for w in values(1.0 - 2.0**-40):
        x = math.ldexp(float(w), -e) if abs(e) < 400 else float(w) * 2.0**-e
        if x != 0.0 and abs(x) < 2.0**-1022:
            continue  # denormals give zero
        d = digits6(x, e)
        assert abs(d[0]) <= 128 and all(-128 <= v <= 127 for v in d[1:4]) and all(-256 <= v <= 255 for v in d[4:])
        got = sum(Fraction(v) * pow2_fraction(-q) for v, q in zip(d, QUANTA6))
        assert abs(got - Fraction(x) * pow2_fraction(e)) <= pow2_fraction(-50)


def split6(h, lo):
    s0 = F(98304.0)
    d, r = [], h
    for k, s in enumerate([0, -8, -16, -24, -33, -42]):
        c = F(s0 * F(2.0**s))
        v = F(F(r + c) - c)
        d.append(v)
        r = F(r - v)
        if k == 2:
            r = F(r + lo)
    return d


def test_split6():
    rng = np.random.default_rng(2)
    for _ in range(4000):
        v = rng.uniform(-1, 1) * 2.0 ** -rng.integers(0, 30)
        h = F(v)
        lo = F((v - float(h)) * rng.choice([0.0, 1.0, -1.0]))  # normalised: at most half an ulp of h
        if abs(float(h)) >= 1.0 - 2.0**-20:
            continue
        d = split6(h, lo)
        for x, q, top in zip(d, QUANTA6, [128, 128, 128, 192, 256, 256]):
            n = Fraction(float(x)) * pow2_fraction(q)
            assert n.denominator == 1 and abs(n) <= top
            assert F(np.uint32(np.array([x]).view(np.uint32)[0] & 0xFFFF0000).view(F)) == x  # a bf16 number
        # the low word enters a remainder below 2^-24 in one FP32 sum below 2^-23, and digit 5
        # rounds to 2^-50
        got = sum(Fraction(float(x)) for x in d)
        assert abs(got - (Fraction(float(h)) + Fraction(float(lo)))) <= pow2_fraction(-48) + pow2_fraction(-50)


def test_sums_of_512_products_are_exact():
    """Every product of digits i, j <= 5 over 512 entries stays within 2^24 quanta (level 6's
    product of two digits 3 alone may not)."""
    lam, inp = [128, 128, 128, 192, 256, 256], [128, 128, 128, 128, 256, 256]
    for i in range(6):
        for j in range(6 - i):
            assert 512 * lam[i] * inp[j] <= 2**24 or (i, j) in ((3, 2),)
    assert 512 * 192 * 128 <= 2**24 * 0.75  # (3, 2): digit 3 takes the low word, digit 2 does not


# ---- the bound -----------------------------------------------------------------------------


def coefficients(lmax, m, s):
    """a_l, b_l of p_{l+1} = (a_l x + b_l) p_l - p_{l-1} from a_{lmax+1} downwards."""
    l0 = max(m, abs(s))
    l = np.arange(l0, lmax + 1, dtype=np.longdouble)
    a2 = (l + 1) ** 2 / ((l + 1 - m) * (l + 1 + m)) * (2 * l + 1) * (2 * l + 3) / ((l + 1 - s) * (l + 1 + s))
    a, q = np.empty(len(l)), np.sqrt(a2[-1])
    for k in range(len(l) - 1, -1, -1):
        q = a2[k] / q
        a[k] = q
    with np.errstate(all="ignore"):
        f = np.where(l == 0, 0, m * s / (l * (l + 1))).astype(float)
    return a, a * f


def log2_start(m, s, th, a0):
    l0, kap = (m, s) if m >= abs(s) else (abs(s), m if s > 0 else -m)
    k = abs(s) if m >= abs(s) else m
    r = (math.lgamma(2 * l0 + 1) - math.lgamma(l0 + k + 1) - math.lgamma(l0 - k + 1)) / math.log(2)
    return (0.5 * (math.log2((2 * l0 + 1) / (4 * math.pi)) + r) + l0 * (np.log2(np.sin(th)) - 1) + kap * np.log2(np.tan(th / 2))
            - 0.5 * math.log2(a0))


def walk(a, b, y, v0, minus, fp32):
    """Largest |p_l| of the difference form from start values 2^v0, in FP32 as the kernel's
    walk (values p 2^(64 sc)) or in double (2^(600 sc))."""
    t, step, up = (F, 64, 32) if fp32 else (np.float64, 600, 300)
    e = np.floor(v0) + 1
    sc = np.floor((e + step // 2) / step).astype(int)
    p = (2.0 ** (v0 - step * sc)).astype(t)
    d, vmax, y = p.copy(), np.zeros_like(p), y.astype(t)

    def true(p):
        w = np.where(sc == 0, 1.0, np.where(sc == -1, 2.0**-64, 0.0)) if fp32 else (sc == 0)
        return np.abs(p) * w.astype(t)

    for k in range(len(a)):
        vmax = np.maximum(vmax, true(p))
        if fp32:  # fma in the wider type, rounded once
            ca, cb = float(F(a[k])), float(F(a[k] - 2.0 + (-b[k] if minus else b[k])))
            u = (-ca * y.astype(float) + cb).astype(F)
            d = (u.astype(float) * p.astype(float) + d.astype(float)).astype(F)
        else:
            d = ((a[k] - 2.0 + (-b[k] if minus else b[k])) - a[k] * y) * p + d
        p = p + d
        if k % 4 == 3:
            r = (sc < 0) & (np.abs(p) > 2.0**up)
            p, d, sc = np.where(r, p * t(2.0**-step), p), np.where(r, d * t(2.0**-step), d), sc + r
    return np.maximum(vmax, true(p)).astype(float)


@pytest.mark.parametrize("lmax,ms", [(300, (0, 1, 7, 150, 299)), (4095, (0, 1, 2, 4, 25, 300)), (8191, (0, 2, 40))])
@pytest.mark.parametrize("spin", [0, 2])
def test_bound_holds_up_to_the_poles(lmax, ms, spin):
    """The bound 2^lexp (the walk's maximum and 1/16, up to a power of two) leaves fix64's
    127/128 room on every ring: next to the poles, at Lambda_lmax's nodes and mid-latitude."""
    near = np.concatenate([np.linspace(3e-4, 6e-4, 40), np.array([2.4048, 5.5201, 8.6537, 11.7915]) / (lmax + 1.5)])
    th = np.concatenate([near, np.linspace(0.01, 1.57, 60)])
    x = np.cos(np.concatenate([th, np.pi - near]))  # lone southern rings: folded to cos theta >= 0
    th = np.concatenate([th, near])
    x = np.abs(x)
    for m in ms:
        a, b = coefficients(lmax, m, spin)
        bound, true = np.zeros(len(th)), np.zeros(len(th))
        for minus in range(2 if spin else 1):
            v0 = log2_start(m, -spin if minus else spin, th, a[0])
            bound = np.maximum(bound, walk(a, b, 1.0 - x, v0, minus, True))
            true = np.maximum(true, walk(a, b, 2.0 * np.sin(th / 2) ** 2, v0, minus, False))
        lexp = np.maximum(-90, np.ceil(np.log2(np.maximum(bound, 1e-30) * 1.0625)))
        assert (true <= 127.0 / 128 * 2.0**lexp).all()
