"""Generate poly64.cuh: FP64 polynomials of the cosine cutoff (Eq. 8) and its derivative and
the table of 2^(j/32) for the FP64 tanh, from mpmath at 50 digits.

Run with mpmath available:  python gen_poly64.py > poly64.cuh
The script checks the polynomials in FP64 (Horner's scheme, multiply-adds rounded twice)
before writing.
"""
import sys

import mpmath as mp
import numpy as np

mp.mp.dps = 50
DEG = 8  # truncation below 1e-18 of the largest value on z in [0, 1/4]


def sin_part(z):
    """(1/4) sin(pi y) / y at z = y^2."""
    y = mp.sqrt(z)
    return mp.pi / 4 if y == 0 else mp.sin(mp.pi * y) / (4 * y)


def cos_part(z):
    """(pi/4) cos(pi y) at z = y^2."""
    return mp.pi / 4 * mp.cos(mp.pi * mp.sqrt(z))


def fit(f):
    return [float(c) for c in mp.chebyfit(f, [0, mp.mpf(1) / 4], DEG + 1)]  # highest degree first


def horner(c, z):
    v = np.full_like(z, c[0])
    for a in c[1:]:
        v = v * z + a
    return v


def check(c, f):
    z = np.linspace(0.0, 0.25, 501)
    want = np.array([float(f(mp.mpf(float(v)))) for v in z])
    assert np.abs(horner(c, z) - want).max() < 4e-16


def nest(c):
    e = repr(c[0])
    for a in c[1:]:
        e = f"fma({e}, z, {a!r})"
    return e


def emit():
    p, q = fit(sin_part), fit(cos_part)
    check(p, sin_part)
    check(q, cos_part)
    out = ["// Generated by gen_poly64.py -- do not edit.",
           "// FP64 cosine cutoff (Eq. 8): with y = r / r_c - 1/2 and z = y^2,",
           "//   f_c / 2 = 1/4 - y P(z),   f_c' / 2 = -Q(z) / r_c,",
           f"// degree {DEG} Chebyshev fits on z in [0, 1/4]; and 2^(j/32), j = 0 ... 31, for tanh.",
           "#pragma once", "", "namespace nep {", "",
           "__device__ __forceinline__ double cut_p64(double z)", "{", f"    return {nest(p)};", "}", "",
           "__device__ __forceinline__ double cut_q64(double z)", "{", f"    return {nest(q)};", "}", "",
           "static __device__ const double kExp2Table[32] = {"]
    exact = [mp.power(2, mp.mpf(j) / 32) for j in range(32)]
    t = [repr(float(v)) for v in exact]
    out += ["    " + ", ".join(t[k:k + 4]) + "," for k in range(0, 32, 4)]
    out += ["};", "// the entries' rounding, relative", "static __device__ const double kExp2Rest[32] = {"]
    t = [repr(float((v - mp.mpf(float(v))) / v)) for v in exact]
    out += ["    " + ", ".join(t[k:k + 4]) + "," for k in range(0, 32, 4)]
    out += ["};", "// ln 2 / 32 in two parts (the first with 21 trailing zero bits) and 32 / ln 2"]
    ln = mp.log(2) / 32
    hi = np.float64(float(ln)).view(np.uint64) & np.uint64(0xffffffffffe00000)
    hi = float(hi.view(np.float64))
    out += [f"constexpr double kLn2Hi = {hi!r}, kLn2Lo = {float(ln - mp.mpf(hi))!r}, kLn2Inv = {float(1 / ln)!r};",
            "", "}  // namespace nep"]
    return "\n".join(out) + "\n"


if __name__ == "__main__":
    sys.stdout.write(emit())
