"""Generate the tables of the fixed-point Hankel evaluator (writes hankel_fixed.inc).

The polynomials interpolate at Chebyshev points in 60-digit arithmetic.  The first six alternate in
sign, c_0 - y (c_1 - y (c_2 - ...)), with positive coefficients c_j and Horner sums, so the device
evaluates them with unsigned 64-bit fractions:

* sin(pi x / 2) / (2 x) and cos(pi x / 2) / 2 in y = x^2 on [0, 1/4]                 (unit 2^-64)
* beyond Z_ASYM, in y = 256 / z^2, with P_nu, Q_nu as in gen_hankel_coeffs.py:
    2^11 (1 - P_0) / y, 4 (-z Q_0), 2^11 (P_1 - 1) / y, 2 z Q_1                      (unit 2^-64)

and below Z_ASYM, on the intervals BOUNDS of z, P_0 - 1, Q_0, P_1 - 1, Q_1 as polynomials in
t = 2^sh (u - u_lo), u = 1/z (sh: t < 1/2), with signed coefficients and sums of unit 2^-64, all
below 1/2.

The interpolation error of every table is checked to stay below 2^-60 of the quantity it stands
for (E, F, P, Q).  Run:  python gen_hankel_fixed.py   (needs mpmath; the output is committed)
"""
import os
import struct

import mpmath as mp

from gen_hankel_coeffs import PQ, Z_ASYM

mp.mp.dps = 60
DEG_S, DEG_C, DEG_PQ = 7, 7, 7
BOUNDS = [1.5, 1.75, 2.0, 2.5, 3.25, 4.25, 5.75, 8.0, 12.0, Z_ASYM]
DEG_N = 10


def cheb_interp(f, hi, deg):
    """Monomial coefficients in y of the degree-deg interpolant on [0, hi] at Chebyshev points."""
    n = deg + 1
    y = [hi * (1 + mp.cos(mp.pi * (2 * j + 1) / (2 * n))) / 2 for j in range(n)]
    V = mp.matrix(n, n)
    for i in range(n):
        for j in range(n):
            V[i, j] = y[i] ** j
    c = mp.lu_solve(V, mp.matrix([f(v) for v in y]))
    return [c[j] for j in range(n)]


def table(name, f, hi, deg, weight):
    """C initializer of one table; weight(y): size of the quantity per unit of the table."""
    c = cheb_interp(f, hi, deg)
    err = max(abs(mp.polyval(c[::-1], y) - f(y)) * weight(y)
              for y in [hi * (k + mp.mpf(1) / 3) / 200 for k in range(200)])
    assert err < mp.mpf(2) ** -60, (name, mp.log(err, 2))
    out = []
    for j, v in enumerate(c):
        v = v * (-1) ** j
        q = int(mp.nint(v * mp.mpf(2) ** 64))
        assert 0 <= q < 2 ** 64, (name, j, v)
        out.append(f"0x{q:016x}ull")
    return f"// error {mp.nstr(err, 2)}\n#define {name} {{{', '.join(out)}}}"


def near_tables():
    """Per interval: u_lo, sh and the four rows of coefficients (integers of unit 2^-64)."""
    lo_, sh_, rows, worst = [], [], [], mp.mpf(0)
    n = DEG_N + 1
    for a, b in zip(BOUNDS[:-1], BOUNDS[1:]):
        lo = int(mp.floor(mp.mpf(2) ** 64 / b)) - 2 ** 16  # the 1/z given may be a few ulp off
        w = mp.mpf(1) / a - mp.mpf(lo) / 2 ** 64
        sh = int(mp.floor(mp.log(mp.mpf(1) / 2 / w, 2)))
        tmax = w * 2 ** sh
        assert tmax * (1 + mp.mpf(2) ** -50) < mp.mpf(1) / 2
        t = [tmax * (1 + mp.cos(mp.pi * (2 * j + 1) / (2 * n))) / 2 for j in range(n)]
        zt = lambda v: 1 / (mp.mpf(lo) / 2 ** 64 + v / 2 ** sh)  # noqa: B023, E731
        V = mp.matrix(n, n)
        for i in range(n):
            for j in range(n):
                V[i, j] = t[i] ** j
        probes = [tmax * (k + mp.mpf(1) / 3) / 40 for k in range(40)]
        row = []
        for nu in (0, 1):
            at, ref = [PQ(nu, zt(v)) for v in t], [PQ(nu, zt(v)) for v in probes]
            for which in (0, 1):
                off = 1 if which == 0 else 0
                c = mp.lu_solve(V, mp.matrix([v[which] - off for v in at]))
                c = [c[j] for j in range(n)]
                worst = max([worst] + [abs(mp.polyval(c[::-1], v) - (r[which] - off)) for v, r in zip(probes, ref)])
                for k in range(n):  # Horner sums from coefficient k on
                    assert sum(abs(c[j]) * tmax ** (j - k) for j in range(k, n)) < mp.mpf(1) / 2, (a, nu, which, k)
                row.append([int(mp.nint(v * mp.mpf(2) ** 64)) for v in c])
        lo_.append(lo)
        sh_.append(sh)
        rows.append(row)
    assert worst < mp.mpf(2) ** -60, mp.log(worst, 2)
    L = [f"// below {Z_ASYM!r}: error {mp.nstr(worst, 2)}",
         f"#define HX_NIV {len(rows)}", f"#define HX_DEG_N {DEG_N}"]
    his = [struct.unpack("<Q", struct.pack("<d", b))[0] for b in BOUNDS[1:-1]]
    assert all(h & 0xffffffff == 0 for h in his), "bounds must have a zero low word"
    L.append("// high words of the inner interval bounds")
    L.append("#define HX_IV_HI {" + ", ".join(str(h >> 32) for h in his) + "}")
    L.append("#define HX_NEAR_LO {" + ", ".join(f"0x{v:016x}ull" for v in lo_) + "}")
    L.append("#define HX_NEAR_SH {" + ", ".join(map(str, sh_)) + "}")
    L.append("// [interval][P_0 - 1, Q_0, P_1 - 1, Q_1][coefficient]")
    body = ", ".join("{" + ", ".join("{" + ", ".join(f"{v}ll" for v in r) + "}" for r in row) + "}" for row in rows)
    L.append("#define HX_NEAR {" + body + "}")
    return L


def main():
    sy = mp.sqrt
    L = ["// Generated by gen_hankel_fixed.py -- do not edit."]
    L.append(table("HX_SIN", lambda y: mp.sin(mp.pi * sy(y) / 2) / (2 * sy(y)), mp.mpf(1) / 4, DEG_S,
                   lambda y: 2 * sy(y)))
    L.append(table("HX_COS", lambda y: mp.cos(mp.pi * sy(y) / 2) / 2, mp.mpf(1) / 4, DEG_C, lambda y: 2))
    hi = mp.mpf(256) / mp.mpf(Z_ASYM) ** 2
    z = lambda y: 16 / sy(y)
    L.append(table("HX_P0", lambda y: 2 ** 11 * (1 - PQ(0, z(y))[0]) / y, hi, DEG_PQ, lambda y: y / 2 ** 11))
    L.append(table("HX_Q0", lambda y: -4 * z(y) * PQ(0, z(y))[1], hi, DEG_PQ, lambda y: 1 / (4 * z(y))))
    L.append(table("HX_P1", lambda y: 2 ** 11 * (PQ(1, z(y))[0] - 1) / y, hi, DEG_PQ, lambda y: y / 2 ** 11))
    L.append(table("HX_Q1", lambda y: 2 * z(y) * PQ(1, z(y))[1], hi, DEG_PQ, lambda y: 1 / (2 * z(y))))
    L += near_tables()
    c = int(mp.floor(2 / mp.pi * mp.mpf(2) ** 96))
    L.append("// 2/pi in units of 2^-96, most significant word first")
    L.append(f"#define HX_2_OVER_PI {{0x{c >> 64:08x}u, 0x{c >> 32 & 0xffffffff:08x}u, 0x{c & 0xffffffff:08x}u}}")
    L += [f"#define HX_DEG_S {DEG_S}", f"#define HX_DEG_C {DEG_C}", f"#define HX_DEG_PQ {DEG_PQ}"]
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "hankel_fixed.inc")
    open(out, "w").write("\n".join(L) + "\n")


if __name__ == "__main__":
    main()
