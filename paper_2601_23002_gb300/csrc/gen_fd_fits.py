"""Generates fd_fit_tables.h: piecewise polynomials for the inverse
Fermi-Dirac integral, the Thomas-Fermi free-energy function and the
Perdew-Zunger exchange-correlation functions.

For y = I_{1/2}(eta) (the reduced density pi^2 n / (sqrt2 T^(3/2)) of the
finite-T Thomas-Fermi term F_s^TF of Eq. 1) and s = ln y, the CUDA kernels
need
    eta(s)                              (v_TF = T eta)
    p(s) = (2/3) I_{3/2}(eta(s)) / y    (f_TF = sqrt2/pi^2 T^(5/2) y (eta - p))

FP32 table: equal intervals of s on [S_LO, S_HI), power series in the
interval's x in [-1, 1] (interpolated at the Chebyshev nodes); outside, the
kernels use the leading terms of the non-degenerate series and of the
Sommerfeld expansion.

FP64 tables: SUB equal intervals of every binade [2^e, 2^(e+1)) of the
argument itself, so that the interval and the local variable (mantissa minus
the interval's middle, exact) come from the argument's bits, without a
logarithm; power series, the two functions' coefficients interleaved.
    fd64: (eta, p) of y on [2^FD_ELO, 2^FD_EHI)
    xc64: (e_xc, v_xc) of u = n / n_1, n_1 = 3/(4 pi) the density of r_s = 1
          (where the two correlation branches meet: an interval's end), on
          [2^XC_ELO, 2^XC_EHI)
Outside, eta and p come from the series
    y small: eta = ln u + sum_k a_k u^k, p = 1 + sum_k b_k u^k, u = y / Gamma(3/2)
    y large: Sommerfeld through e0^-4, e0 = (3 y / 2)^(2/3)
whose a_k, b_k this script computes, and e_xc, v_xc from their formulas.

Reference values: I_nu(eta) = -Gamma(nu+1) Li_{nu+1}(-e^eta) by mpmath for
eta <= 40, and the Sommerfeld series (exact to far below double precision for
half-integer nu at eta > 40, where the exponentially small part vanishes).
This generator is part of the library build tooling; it does not use the
test oracle.  Run: python gen_fd_fits.py  (writes fd_fit_tables.h beside it).
"""
from __future__ import annotations

import os
import sys
from multiprocessing import Pool

import mpmath as mp

mp.mp.dps = 34

S_LO, S_HI = -32.0, 24.0
W32, D32 = 1.0, 7
SUB, D64 = 16, 8
FD_ELO, FD_EHI = -14, 17
XC_ELO, XC_EHI = -20, 6


def fd_int(nu, eta):
    nu = mp.mpf(nu)
    eta = mp.mpf(eta)
    if eta <= 40:
        return -mp.gamma(nu + 1) * mp.re(mp.polylog(nu + 1, -mp.exp(eta)))
    tot = mp.mpf(1)
    for k in range(1, 10):
        c = 2 * (1 - mp.mpf(2) ** (1 - 2 * k)) * mp.zeta(2 * k)
        c *= mp.gamma(nu + 2) / mp.gamma(nu + 2 - 2 * k)
        tot += c * eta ** (-2 * k)
    return eta ** (nu + 1) / (nu + 1) * tot


def eta_of_s(s):
    y = mp.exp(mp.mpf(s))
    u = y / mp.gamma(mp.mpf(1.5))
    if y < 1:
        guess = mp.log(u) + u / mp.sqrt(8)
    else:
        guess = (mp.mpf(1.5) * y) ** (mp.mpf(2) / 3)
    f = lambda e: mp.log(fd_int(0.5, e)) - mp.mpf(s)
    return mp.findroot(f, guess, tol=mp.mpf(10) ** (-30))


def funcs(s):
    e = eta_of_s(s)
    y = mp.exp(mp.mpf(s))
    p = mp.mpf(2) / 3 * fd_int(1.5, e) / y
    return e, p


def fd_of_y(y):
    return funcs(mp.log(y))


# Perdew-Zunger 1981, unpolarised; B and D from the continuity of e_c and
# de_c/dr_s at r_s = 1 (as the kernels' own formula)
def xc_of_u(u):
    g, b1, b2 = mp.mpf("-0.1423"), mp.mpf("1.0529"), mp.mpf("0.3334")
    A, C = mp.mpf("0.0311"), mp.mpf("0.0020")
    den1 = 1 + b1 + b2
    D = -g * (b1 / 2 + b2) / den1 ** 2 - A - C
    B = g / den1 - D
    rs = u ** (-mp.mpf(1) / 3)
    n = 3 * u / (4 * mp.pi)
    ex = -mp.mpf(3) / 4 * (3 / mp.pi) ** (mp.mpf(1) / 3) * n ** (mp.mpf(1) / 3)
    if u <= 1:
        den = 1 + b1 * mp.sqrt(rs) + b2 * rs
        ec = g / den
        dec = -g * (b1 / (2 * mp.sqrt(rs)) + b2) / den ** 2
    else:
        ln = mp.log(rs)
        ec = A * ln + B + C * rs * ln + D * rs
        dec = A / rs + C * ln + C + D
    return ex + ec, 4 * ex / 3 + ec - rs / 3 * dec


def power_fit(values, nodes):
    """Monomial coefficients of the polynomial through (nodes, values)."""
    n = len(nodes)
    V = mp.matrix(n, n)
    for i, x in enumerate(nodes):
        for k in range(n):
            V[i, k] = x ** k
    c = mp.lu_solve(V, mp.matrix(values))
    return [c[k] for k in range(n)]


def horner(c, x):
    r = mp.mpf(0)
    for ck in reversed(c):
        r = r * x + ck
    return r


def cheb_nodes(deg, half):
    return [half * mp.cos(mp.pi * (j + mp.mpf(0.5)) / (deg + 1)) for j in range(deg + 1)]


def fit_pair(args):
    """Coefficients of the two functions of `kind` on middle +- half (times
    scale), and the worst error between the nodes."""
    kind, mid, half, scale, deg = args
    mid, half, scale = mp.mpf(mid), mp.mpf(half), mp.mpf(scale)
    f = {"s": lambda x: funcs(mid + half * x), "fd": lambda t: fd_of_y(scale * (mid + t)),
         "xc": lambda t: xc_of_u(scale * (mid + t))}[kind]
    nodes = cheb_nodes(deg, mp.mpf(1) if kind == "s" else half)
    vals = [f(x) for x in nodes]
    c1 = power_fit([v[0] for v in vals], nodes)
    c2 = power_fit([v[1] for v in vals], nodes)
    e1 = e2 = mp.mpf(0)
    for q in ("-0.97", "-0.41", "0.13", "0.77"):
        x = mp.mpf(q) * (mp.mpf(1) if kind == "s" else half)
        a, b = f(x)
        e1 = max(e1, abs(horner(c1, x) - a) / max(1 if kind != "xc" else 0, abs(a)))
        e2 = max(e2, abs(horner(c2, x) - b) / max(1 if kind != "xc" else 0, abs(b)))
    return c1, c2, e1, e2


def series_coefficients():
    """a_k, b_k (k = 1..3) of eta - ln u and p - 1 in powers of u, from
    u(z) = -Li_{3/2}(-z), z = e^eta, and p = Li_{5/2}(-z)/Li_{3/2}(-z)."""
    # z = u + z2 u^2 + z3 u^3 + z4 u^4 by inverting u = sum (-1)^(k+1) z^k / k^(3/2)
    def compose(order):
        z = [mp.mpf(0)] * (order + 1)
        z[1] = mp.mpf(1)
        for m in range(2, order + 1):
            # coefficient of u^m in sum_k (-1)^(k+1) z^k/k^1.5 must vanish
            def coef(zz):
                tot, pw = mp.mpf(0), [mp.mpf(1)] + [mp.mpf(0)] * order
                for k in range(1, m + 1):
                    pw = [sum(pw[i] * zz[j - i] for i in range(j + 1)) for j in range(order + 1)]
                    tot += (-1) ** (k + 1) * pw[m] / mp.mpf(k) ** mp.mpf(1.5)
                return tot
            z[m] = -coef(z)
        return z
    order = 4
    z = compose(order)
    # ln(z/u) = ln(1 + r), r = z2 u + z3 u^2 + z4 u^3
    r = [mp.mpf(0)] + z[2:]
    mul = lambda a, b: [sum(a[i] * b[j - i] for i in range(j + 1)) for j in range(order)]
    r2 = mul(r, r)
    r3 = mul(r2, r)
    a = [r[k] - r2[k] / 2 + r3[k] / 3 for k in range(order)]
    # p u = sum (-1)^(k+1) z^k / k^(5/2)
    tot, pw = [mp.mpf(0)] * (order + 1), [mp.mpf(1)] + [mp.mpf(0)] * order
    for k in range(1, order + 1):
        pw = [sum(pw[i] * z[j - i] for i in range(j + 1)) for j in range(order + 1)]
        tot = [t + (-1) ** (k + 1) * q / mp.mpf(k) ** mp.mpf(2.5) for t, q in zip(tot, pw)]
    return a[1:4], tot[2:5]


def fmt(v, single):
    return (f"{float(v):.9e}f" if single else f"{float(v):.17g}")


def main():
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fd_fit_tables.h")
    n32 = int(round((S_HI - S_LO) / W32))
    jobs32 = [("s", S_LO + (i + 0.5) * W32, W32 / 2, 1, D32) for i in range(n32)]

    def binades(kind, lo, hi):
        return [(kind, 1 + (j + mp.mpf(0.5)) / SUB, mp.mpf(1) / (2 * SUB), mp.mpf(2) ** e, D64)
                for e in range(lo, hi) for j in range(SUB)]

    jfd, jxc = binades("fd", FD_ELO, FD_EHI), binades("xc", XC_ELO, XC_EHI)
    with Pool() as pool:
        r32 = pool.map(fit_pair, jobs32, chunksize=2)
        rfd = pool.map(fit_pair, jfd, chunksize=4)
        rxc = pool.map(fit_pair, jxc, chunksize=8)
    worst = [[float(max(r[k] for r in rr)) for k in (2, 3)] for rr in (r32, rfd, rxc)]
    a, b = series_coefficients()
    lines = [
        "/* Generated by gen_fd_fits.py -- do not edit.",
        " * fd32_tab: power series in x in [-1, 1] (eta's, then p's) on intervals of s = ln y for",
        " * eta(s) = I_{1/2}^{-1}(e^s) and p(s) = (2/3) I_{3/2}(eta(s)) / e^s on [FD_S_LO, FD_S_HI):",
        f" * {n32} intervals of width {W32}, degree {D32}; max rel err eta {worst[0][0]:.2e}, p {worst[0][1]:.2e}.",
        f" * fd64_tab: (eta, p) of y on {SUB} intervals per binade of [2^{FD_ELO}, 2^{FD_EHI}), degree {D64}, coefficient pairs;",
        f" * max rel err eta {worst[1][0]:.2e}, p {worst[1][1]:.2e}.",
        f" * xc64_tab: (e_xc, v_xc) of u = 4 pi n / 3 on {SUB} intervals per binade of [2^{XC_ELO}, 2^{XC_EHI});",
        f" * max rel err {worst[2][0]:.2e}, {worst[2][1]:.2e}.",
        " * FD_A*, FD_B*: eta = ln u + sum a_k u^k, p = 1 + sum b_k u^k, u = y / Gamma(3/2), below the table.",
        " */",
        "#pragma once",
        f"#define FD_S_LO ({S_LO})",
        f"#define FD_S_HI ({S_HI})",
        f"#define FD32_W ({W32}f)",
        f"#define FD32_NINT {n32}",
        f"#define FD32_NC {D32 + 1}",
        f"#define BIN64_LG {SUB.bit_length() - 1}",
        f"#define BIN64_NC {D64 + 1}",
        f"#define FD64_ELO ({FD_ELO})",
        f"#define FD64_NINT {len(rfd)}",
        f"#define XC64_ELO ({XC_ELO})",
        f"#define XC64_NINT {len(rxc)}",
    ]
    lines += [f"#define FD_A{k + 1} ({float(v):.17g})" for k, v in enumerate(a)]
    lines += [f"#define FD_B{k + 1} ({float(v):.17g})" for k, v in enumerate(b)]

    def arr(name, tab, single, typ):
        lines.append(f"static __device__ __align__(16) const {typ} {name}[{len(tab)}][{len(tab[0])}] = {{")
        for row in tab:
            lines.append("  {" + ", ".join(fmt(v, single) for v in row) + "},")
        lines.append("};")

    pairs = lambda rr: [[v for q in zip(r[0], r[1]) for v in q] for r in rr]
    arr("fd64_tab", pairs(rfd), False, "double")
    arr("xc64_tab", pairs(rxc), False, "double")
    arr("fd32_tab", [r[0] + r[1] for r in r32], True, "float")
    with open(out, "w") as f:
        f.write("\n".join(lines) + "\n")
    sys.stderr.write(f"worst errors {worst}\n")
    print("wrote", out)


if __name__ == "__main__":
    main()
