"""Writes hankel_fit.h: fixed-point polynomials for the modulus-phase functions
of the Hankel functions H_0 and H_1 for z >= 8, and for sine and cosine on an
eighth of a turn to each side.

For real z > 0 (DLMF 10.17, Abramowitz & Stegun 9.2.5-9.2.6),
    J_nu(z) = sqrt(2/(pi z)) (P_nu(z) cos chi - Q_nu(z) sin chi),
    Y_nu(z) = sqrt(2/(pi z)) (P_nu(z) sin chi + Q_nu(z) cos chi),
    chi = z - (nu/2 + 1/4) pi,
so P_nu = sqrt(pi z/2) (J_nu cos chi + Y_nu sin chi) and
Q_nu = sqrt(pi z/2) (Y_nu cos chi - J_nu sin chi).  P_nu and z Q_nu are
smooth, even functions of 1/z; on each interval [za, zb) they are fitted as
polynomials in x = (v - vm) / vh, v = 1/z^2, mapped onto [-1, 1]: Chebyshev
interpolation at Chebyshev points from 40-digit values (mpmath), converted to
monomial coefficients for Horner's rule.  The intervals are widened by 1e-6, so
that |x| < 1 also where z was compared with an end after rounding to FP32.
sin(pi/4 g) / g and cos(pi/4 g) are fitted the same way in x = g^2 on [0, 1].

The polynomials are evaluated in 60-bit fixed point: the highest coefficients,
whose sums stay below 2^-28, by 32-bit multiplications, the others by the
products of fx.cuh.  Every fit is checked: an integer emulation of the header's
statements is compared with 40-digit values at 161 points of the interval and
must stay within 1e-17 absolute.

Run from this directory (needs mpmath and numpy):  python gen_hankel_fit.py
(the header is committed; the build does not run this script).
"""
import os

import mpmath as mp

mp.mp.dps = 40
INTERVALS = [(8, 12, 9), (12, 20, 8), (20, 30, 6), (30, 60, 6), (60, None, 5)]   # (za, zb, degree)
NPTS = 64
PAD = mp.mpf(1) / 10 ** 6
TOL = 1e-17


def pq(nu, z):
    """P_nu - 1 and z Q_nu"""
    if z is None:
        return mp.mpf(0), mp.mpf(4 * nu * nu - 1) / 8
    j, y = mp.besselj(nu, z), mp.bessely(nu, z)
    chi = z - (mp.mpf(nu) / 2 + mp.mpf(1) / 4) * mp.pi
    c, s = mp.cos(chi), mp.sin(chi)
    f = mp.sqrt(mp.pi * z / 2)
    return f * (j * c + y * s) - 1, f * (y * c - j * s) * z


def cheb_fit(f, deg, lo, hi):
    """monomial coefficients on [lo, hi], in the variable itself"""
    xs = [mp.cos(mp.pi * (k + mp.mpf(1) / 2) / NPTS) for k in range(NPTS)]
    F = [f((lo + hi) / 2 + (hi - lo) / 2 * x) for x in xs]
    cheb = [mp.fsum(F[k] * mp.cos(j * mp.pi * (k + mp.mpf(1) / 2) / NPTS) for k in range(NPTS)) * (2 if j else 1) / NPTS
            for j in range(deg + 1)]
    # T_j in t = (2 x - lo - hi) / (hi - lo), by the recurrence on coefficient lists
    a, b = 2 / mp.mpf(hi - lo), -mp.mpf(lo + hi) / (hi - lo)
    T = [[mp.mpf(1)], [b, a]]
    for _ in range(2, deg + 1):
        p, q = T[-1], T[-2]
        n = [mp.mpf(0)] * (len(p) + 1)
        for i, c in enumerate(p):
            n[i] += 2 * b * c
            n[i + 1] += 2 * a * c
        for i, c in enumerate(q):
            n[i] -= c
        T.append(n)
    out = [mp.mpf(0)] * (deg + 1)
    for j in range(deg + 1):
        for i, c in enumerate(T[j]):
            out[i] += cheb[j] * c
    return out


def rnd(x):
    return int(mp.nint(x))


class Horner:
    """Integer coefficients and statements of one polynomial (|x| <= 1)."""

    def __init__(self, mono):
        deg = len(mono) - 1
        tails = [mp.fsum(abs(c) for c in mono[k:]) for k in range(deg + 1)]
        scale = lambda t: int(mp.floor(mp.mpf("30.9") - mp.log(t, 2)))
        self.m = next((k for k in range(1, deg + 1) if scale(tails[k]) >= 59), deg + 1)
        self.deg = deg
        if self.m <= deg:
            self.S = scale(tails[self.m])
            self.lo = {k: rnd(mono[k] * mp.mpf(2) ** (self.S + k - self.m)) for k in range(self.m, deg + 1)}
            assert all(abs(c) < 2 ** 31 for c in self.lo.values())
        self.hi = {k: rnd(mono[k] * mp.mpf(2) ** 60) for k in range(0, min(self.m, deg + 1))}

    def emulate(self, X):
        """X = x 2^60"""
        x31 = min(X >> 29, 2 ** 31 - 1)
        if self.m <= self.deg:
            a = self.lo[self.deg]
            for k in range(self.deg - 1, self.m - 1, -1):
                a = ((a * x31) >> 32) + self.lo[k]
            acc = ((a * x31) >> (self.S - 29)) + self.hi[self.m - 1]
            k = self.m - 2
        else:
            acc = self.hi[self.deg]
            k = self.deg - 1
        for j in range(k, -1, -1):
            acc = fxmul(acc, X) + self.hi[j]
        return acc

    def code(self, name):
        hexs = lambda c: f"{c}ll"
        out = []
        if self.m <= self.deg:
            e = f"{self.lo[self.deg]}"
            for k in range(self.deg - 1, self.m - 1, -1):
                e = f"__mulhi({e}, x31) + {self.lo[k]}" if e.lstrip("-").isdigit() else f"__mulhi({e}, x31) + {self.lo[k]}"
            out.append(f"  {name} = (((long long)({e}) * x31) >> {self.S - 29}) + {hexs(self.hi[self.m - 1])};")
            k = self.m - 2
        else:
            out.append(f"  {name} = {hexs(self.hi[self.deg])};")
            k = self.deg - 1
        for j in range(k, -1, -1):
            out.append(f"  {name} = fx_mul(fx({name}), x) + {hexs(self.hi[j])};")
        return out


def fxmul(a, b):
    """fx.cuh's product of two Q60 numbers"""
    def split(v):
        h = (v + 2 ** 29) >> 30
        l = v & (2 ** 30 - 1)
        return h, l - 2 ** 30 if l >= 2 ** 29 else l
    (ah, al), (bh, bl) = split(a), split(b)
    return ah * bh + ((2 ** 29 + ah * bl + al * bh) >> 30)


def check(h, f, lo, hi, what):
    worst = 0.0
    for i in range(161):
        X = rnd((mp.mpf(lo) + (mp.mpf(hi) - lo) * i / 160) * mp.mpf(2) ** 60)
        worst = max(worst, float(abs(mp.mpf(h.emulate(X)) / mp.mpf(2) ** 60 - f(mp.mpf(X) / mp.mpf(2) ** 60))))
    if worst > TOL:
        raise SystemExit(f"{what}: error {worst:.2e} > {TOL}")
    return worst


def main():
    here = os.path.dirname(os.path.abspath(__file__))
    lines = [
        "// Generated by gen_hankel_fit.py (do not edit): polynomials in 60-bit fixed",
        "// point (value 2^60) for P_nu and z Q_nu (nu = 0, 1; Hankel's modulus-phase",
        "// functions) in x = (1/z^2 - vm) ivh on [za, zb), and for sin(pi/4 g) / g and",
        "// cos(pi/4 g) in x = g^2; x31 is x 2^31.  The worst errors are those of the",
        "// integer evaluation against 40-digit values.",
        "#pragma once",
        '#include "fx.cuh"',
        "",
    ]
    for i, (za, zb, deg) in enumerate(INTERVALS):
        va = 1 / (mp.mpf(za) * (1 - PAD)) ** 2
        vb = 1 / (mp.mpf(zb) * (1 + PAD)) ** 2 if zb else -va * PAD
        vm, vh = (va + vb) / 2, (va - vb) / 2
        zof = lambda x: 1 / mp.sqrt(vm + vh * x) if vm + vh * x > mp.mpf(10) ** -12 else None
        fits = {}
        for nu in (0, 1):
            for w, name in ((0, "P"), (1, "zQ")):
                f = lambda x: pq(nu, zof(x))[w] + (1 - w)
                h = Horner(cheb_fit(f, deg, -1, 1))
                fits[f"{name}{nu}"] = (h, check(h, f, -1 if zb else -1 + 4 * PAD, 1, f"[{za}, {zb}) {name}{nu}"))
        lines.append(f"// [{za}, {zb if zb else 'inf'}): degree {deg}; worst errors " +
                     ", ".join(f"{k} {v[1]:.1e}" for k, v in fits.items()))
        lines.append(f"constexpr double HK_IVH{i} = {float(1 / vh)!r}, HK_SH{i} = {float(3 - vm / vh)!r};   // 3 + x = v ivh + sh")
        lines.append(f"__device__ __forceinline__ void hankel_fit{i}(Fx x, int x31, long long& P0, long long& zQ0, "
                     "long long& P1, long long& zQ1) {")
        for k in ("P0", "zQ0", "P1", "zQ1"):
            lines += fits[k][0].code(k)
        lines += ["}", ""]
    q = mp.pi / 4
    fs = lambda x: mp.sin(q * mp.sqrt(x)) / mp.sqrt(x) if x > 0 else q
    fc = lambda x: mp.cos(q * mp.sqrt(x))
    hs, hc = Horner(cheb_fit(fs, 7, 0, 1)), Horner(cheb_fit(fc, 7, 0, 1))
    es, ec = check(hs, fs, 0, 1, "sine"), check(hc, fc, 0, 1, "cosine")
    lines.append(f"// sin(pi/4 g) / g and cos(pi/4 g), x = g^2 in [0, 1]: degree 7; worst errors {es:.1e}, {ec:.1e}")
    lines.append("__device__ __forceinline__ void hankel_sincos_fit(Fx x, int x31, long long& s, long long& c) {")
    lines += hs.code("s") + hc.code("c") + ["}", ""]
    with open(os.path.join(here, "hankel_fit.h"), "w") as fh:
        fh.write("\n".join(lines))
    print("wrote hankel_fit.h")


if __name__ == "__main__":
    main()
