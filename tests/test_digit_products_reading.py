"""The integer arithmetic of the FP64-accurate products and of the fixed-point
reflector, restated in Python integers and compared with exact values.

The restatements follow csrc/oz.cuh (digits, join, the eight-digit product),
csrc/oz_matvec.cu (cut, the seven-digit product with column weights) and
csrc/fx.cuh (fx_reflect) step by step.  Bounds, per real term and relative to
the product of the two largest parts: a pair of digits i + j = s weighs 256^-s and
is below 2^14 of the 2^61 (2^53) that the largest part is at least, so that what
the eight (seven) digits leave out is below 7 (6) 2^62 / 2^122 plus a 250th, 2^-57
(2^-49); cutting adds 2^-62 (2^-51).
"""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest

M32, M64 = (1 << 32) - 1, (1 << 64) - 1


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _exponent(x):
    return _bits(x) >> 52 & 0x7FF


def _balanced(v, n):
    """n signed base-256 digits of v, the largest first, through biased bytes"""
    b = v + sum(128 << 8 * i for i in range(n))
    assert 0 <= b < 1 << 8 * n
    return [(b >> 8 * (n - 1 - i) & 255) - 128 for i in range(n)]


# ---- eight digits (oz.cuh) ----------------------------------------------------

def _digits62(x, E):
    b = _bits(x)
    e = b >> 52 & 0x7FF
    d = min(E - e, 63) if e else 63
    m = (b & (1 << 52) - 1) | 1 << 52
    q = ((m << 10 >> d) + 1) >> 1
    return -q if b >> 63 else q


def _join(hi, lo, p2):
    """oz::join in 32-bit words: the double nearest to (hi 2^32 + lo) 2^p2"""
    hi += lo >> 32
    sg = M32 if hi < 0 else 0
    w2, w1, w0 = (hi >> 32 & M32) ^ sg, (hi & M32) ^ sg, (lo & M32) ^ sg
    t = w0 + (sg & 1)
    w0, t = t & M32, w1 + (t >> 32)
    w1, w2 = t & M32, w2 + (t >> 32) & M32
    e = 1023 + 95 + p2
    if w2 == 0:
        w2, w1, w0, e = w1, w0, 0, e - 32
    if w2 == 0:
        w2, w1, e = w1, w0, e - 32
    lz = 32 - w2.bit_length()
    funnel = lambda h, l: ((h << 32 | l) << (lz & 31)) >> 32 & M32
    m1, m0 = funnel(w2, w1), funnel(w1, w0)
    e -= lz
    r = (m1 << 32 | m0) >> 11
    r += m0 >> 10 & 1
    r += ((e - 1 & 0xFFF) << 20 | (sg & 0x80000000)) << 32
    if m1 == 0 or e <= 0:
        return 0.0
    assert e < 2047
    return struct.unpack("<d", struct.pack("<Q", r & M64))[0]


def _nearest(v, p2):
    """v 2^p2 rounded to a double, halves away from zero"""
    if v == 0:
        return 0.0
    s = max(abs(v).bit_length() - 53, 0)
    q = (abs(v) + (1 << s >> 1)) >> s
    return math.copysign(math.ldexp(q, s + p2), v)


def _product8(a, b):
    """sum a_k b_k of 64 reals as one stage forms it"""
    ea, eb = max(map(_exponent, a)), max(map(_exponent, b))
    da = [_balanced(_digits62(x, ea), 8) for x in a]
    db = [_balanced(_digits62(x, eb), 8) for x in b]
    v = [sum(x[i] * y[s - i] for x, y in zip(da, db) for i in range(s + 1)) for s in range(8)]
    assert all(abs(t) <= 1 << 23 for t in v)            # exact in FP32
    p = [v[2 * i] * 256 + v[2 * i + 1] for i in range(4)]
    assert all(abs(t) < 1 << 31 for t in p)
    return _join(p[0] * 65536 + p[1], p[2] * 65536 + p[3], ea + eb - 2112)


def _rows(rng, n, kind):
    a, b = rng.standard_normal(n), rng.standard_normal(n)
    if kind == "graded":         # in opposite directions, over a factor 2^40
        g = np.exp2(rng.integers(-20, 21, n))
        a, b = a * g, b / g
    elif kind == "cancelling":
        a[n // 2:], b[n // 2:] = -a[: n // 2], b[: n // 2] * (1 + 1e-14 * rng.standard_normal(n // 2))
    elif kind == "full":         # mantissas of ones
        a = np.copysign(np.nextafter(2.0, 1.0), a)
        b = np.copysign(np.nextafter(2.0, 1.0), b)
    return a, b


@pytest.mark.parametrize("kind", ["flat", "graded", "cancelling", "full"])
def test_eight_digit_products(kind):
    rng = np.random.default_rng(3)
    for _ in range(60):
        a, b = _rows(rng, 64, kind)
        exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
        top = float(np.max(np.abs(a)) * np.max(np.abs(b)))
        err = abs(Fraction(_product8(a.tolist(), b.tolist())) - exact)
        assert err <= Fraction(top) * 64 * Fraction(1, 2 ** 57) + abs(exact) * Fraction(1, 2 ** 53)


def test_digits_are_a_rounded_integer():
    rng = np.random.default_rng(4)
    for _ in range(4000):
        x = math.ldexp(rng.uniform(-2, 2), int(rng.integers(-70, 1)))
        E = _exponent(x) + int(rng.integers(0, 70))
        q, d = _digits62(x, E), _balanced(_digits62(x, E), 8)
        assert sum(c << 8 * (7 - i) for i, c in enumerate(d)) == q and abs(d[0]) <= 64
        assert abs(Fraction(q) - Fraction(x) * Fraction(2) ** (61 - (E - 1023))) <= Fraction(1, 2)


def test_join_rounds_every_sum_to_nearest():
    rng = np.random.default_rng(5)
    def check(v):
        for hi, lo in ((v >> 32, v & M32), ((v >> 32) + 7, (v & M32) - (7 << 32)), ((v >> 32) - 9, (v & M32) + (9 << 32))):
            assert _join(hi, lo, -60) == _nearest(v, -60), hex(v)
    for k in range(1, 90):
        for t in (0, 1, 2, 3, 5, 1 << 10, 1 << 11, 3 << 9):   # all ones, carries through every word
            for v in ((1 << k) - t, (1 << k) + t):
                check(v)
                check(-v)
    for _ in range(20000):
        check(int(rng.integers(-1 << 62, 1 << 62)) << int(rng.integers(0, 28)) >> int(rng.integers(0, 80)))


# ---- seven digits, entries in two parts, weighted columns (oz_matvec.cu) ----------

def _split(x):
    """hi and lo of 24 bits each, both cut off"""
    m, e = np.frexp(x)
    hi = np.ldexp(np.trunc(m * 2.0 ** 24), e - 24)
    m, e = np.frexp(x - hi)
    return hi, np.ldexp(np.trunc(m * 2.0 ** 24), e - 24)


def _f32(x):
    b = struct.unpack("<I", struct.pack("<f", x))[0]
    return b >> 31, b >> 23 & 0xFF, b & 0x7FFFFF


def _cut(hi, lo, E):
    sg, eh, fh = _f32(hi)
    _, el, fl = _f32(lo)
    mh, ml = (fh << 8 | 1 << 31 if eh else 0), (fl << 8 | 1 << 31 if el else 0)
    q = (mh << 32) >> min(E - eh + 10, 64)
    q += ml >> min((E - el - 22) & M32, 32)
    return -q if sg else q


def _product7(a, x, col):
    hi, lo = _split(a)
    er = max([1] + [_f32(h)[1] + c for h, c in zip(hi, col)])
    ex = max(_exponent(v) - c for v, c in zip(x, col))
    da = [_balanced(_cut(h, l, er - c), 7) for h, l, c in zip(hi, lo, col)]
    dx = [_balanced((_digits62(v, ex + c) + 128) >> 8, 7) for v, c in zip(x, col)]
    v = [sum(p[i] * q[s - i] for p, q in zip(da, dx) for i in range(s + 1)) for s in range(7)]
    top = sum(v[s] << 8 * (2 - s) for s in range(3))
    low = sum(v[s] << 8 * (6 - s) for s in range(3, 7))
    return _join(top, low, er + ex - 1208)


@pytest.mark.parametrize("kind", ["flat", "graded", "cancelling"])
@pytest.mark.parametrize("weighted", [False, True])
def test_seven_digit_products(kind, weighted):
    rng = np.random.default_rng(6)
    for _ in range(20):
        n = 256
        a, x = _rows(rng, n, kind)
        hi, lo = _split(a)
        col = [0] * n
        if weighted:   # the columns' scales from X, at most zero
            e = [math.frexp(v)[1] for v in x]
            col = [max(c - max(e), -64) for c in e]
        stored = [Fraction(float(h)) + Fraction(float(l)) for h, l in zip(hi, lo)]
        exact = sum(s * Fraction(float(v)) for s, v in zip(stored, x))
        w = np.exp2(np.array(col, dtype=float))
        top = float(np.max(np.abs(a) * w) * np.max(np.abs(x) / w))
        err = abs(Fraction(_product7(a, x.tolist(), col)) - exact)
        assert err <= Fraction(top) * n * Fraction(1, 2 ** 49) + abs(exact) * Fraction(1, 2 ** 53)
        if weighted and kind == "graded":   # the sizes of the terms themselves, to a factor of two each
            assert top <= 16 * float(np.max(np.abs(a * x)))


# ---- the reflector in integers (fx.cuh) ----------------------------------------------

def _mul64hi(a, b):
    return a * b >> 64


def _reflect(ar, ai, N, sN):
    if N == 0:
        return 0, (0, 0), (0, 0), 0
    b = N.bit_length()
    ev = (sN - b) >> 1
    sh = 64 + 2 * ev - sN
    nn = (N << sh if sh >= 0 else N >> -sh) & M64
    qf = np.float32(1) / np.sqrt(np.float32(np.float32(nn >> 32) * np.float32(2.0 ** -32)))
    q = int(np.float32(qf * np.float32(2.0 ** 30)))
    q60 = q << 30
    e = (1 << 60) - _mul64hi(nn, q * q)
    eh = e >> 14
    e2 = eh * eh >> 32
    rs = q60 + (_mul64hi(q60, e << 20) >> 17) + (((q >> 15) * ((3 * e2) >> 3)) >> 15)
    xn = _mul64hi(nn, rs)
    one = 1 << 60
    nx, ny = ar < 0, ai < 0
    ax, ay = min(abs(ar) << ev, one - 1), min(abs(ai) << ev, one - 1)
    ty = _mul64hi(ay << 4, rs) >> 1
    tau2 = ((one + _mul64hi(ax << 4, rs)) >> 1, -ty if nx != ny else ty)
    beta = xn if nx else -xn
    D = min(ax + xn, 2 * one - 1)
    d = _mul64hi(D << 2, D << 2) + _mul64hi(ay << 2, ay << 2)
    yf = np.float32(1) / np.float32(np.float32(d >> 32) * np.float32(2.0 ** -28))
    y = int(np.float32(yf * np.float32(2.0 ** 28)))
    e = (1 << 58) - _mul64hi(d << 1, y << 33)
    eh = e >> 12
    e2 = eh * eh >> 32
    inv = (y << 32) + (_mul64hi(y << 32, e << 22) >> 16) + (((y >> 13) * e2) >> 15)
    cx, cy = _mul64hi(D << 3, inv), _mul64hi(ay << 3, inv)
    return ev, tau2, (-cx if nx else cx, cy if ny else -cy), beta


def test_integer_reflector_against_exact_values():
    """tau / 2, the scale / 2 and beta in 2^-60: within 16 units, about 2^-56 of their sizes."""
    rng = np.random.default_rng(7)
    for _ in range(4000):
        top = int(rng.integers(3, 59))
        x = [complex(*rng.integers(-(1 << top), 1 << top, 2).tolist()) for _ in range(int(rng.integers(1, 6)))]
        if rng.random() < 0.2:
            x[0] = 0j if len(x) > 1 else x[0]
        N = sum(int(v.real) ** 2 + int(v.imag) ** 2 for v in x)
        ar, ai = int(x[0].real), int(x[0].imag)
        ev, tau2, sc2, beta = _reflect(ar, ai, N, 120)
        if N == 0:
            continue
        norm = Fraction(math.isqrt(N << 200), 1 << 100)
        u = Fraction(2) ** ev                    # units of 2^(-60 - ev)
        assert Fraction(1, 2) <= norm * u / 2 ** 60 < 1 + Fraction(1, 2 ** 50)
        sg = 1 if ar >= 0 else -1
        eb = -sg * norm
        dr, di = ar - eb, Fraction(ai)
        d2 = dr * dr + di * di
        want = ((1 + abs(ar) / norm) / 2, sg * ai / norm / 2, dr / d2 * 2 ** 60 / u / 2, -di / d2 * 2 ** 60 / u / 2)
        got = [Fraction(v, 2 ** 60) for v in (*tau2, *sc2)]
        for g, w in zip(got, want):
            assert abs(g - w) <= Fraction(16, 2 ** 60), (ar, ai, N)
        assert abs(Fraction(beta) - eb * u) <= 16
