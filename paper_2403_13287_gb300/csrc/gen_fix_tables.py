"""Write fix_tables.h: the integer tables of the fixed-point split fluxes
(lskum_fixed.cuh).

1. erf(s)/2 and exp(-s^2)/(2 sqrt(pi)), Taylor coefficients on the grid
s_k = k/2048, k = 0..8192 (s up to 4). With s = s_k + d and u = 2^12 d in
[-1, 1], each function is c_0 + u (c_1 + u (c_2 + u (c_3 + u c_4))),
c_i = f^(i)(s_k) 2^(-12 i) / i!. The first omitted term is below 2^-62. The
coefficients are integers, c_0 2^62, c_1 2^75 (64 bits), c_2 2^56, c_3 2^57,
c_4 2^58 (32 bits): the scales at which the evaluation adds them. A row is
64 bytes: c_0, c_1 of both functions, then c_2, c_3, c_4 of both, then two
padding words.

exp(-s^2) and erf are related to Hermite polynomials H_n (physicists'):
d^n/ds^n exp(-s^2) = (-1)^n H_n(s) exp(-s^2), erf' = 2/sqrt(pi) exp(-s^2).

2. 2^(j/4096) 2^62, j = 0..4095, for the table-driven exp (P. T. P. Tang,
ACM Trans. Math. Software 15 (1989) 144-157).

3. log2 of a mantissa m in [1, 2): for the interval j of 1024, r_j is the
reciprocal of its middle rounded to 32 bits (r_j 2^32) and the table holds
-log2(r_j) 2^60; log2(m) = -log2(r_j) + log2(m r_j) with m r_j - 1 = z,
|z| < 1.0005 2^-11, by the series of log2(1 + z) to z^5 in u = 2^11 z.

The values are computed with mpmath at 50 significant digits and rounded to
the nearest integer.

Run from the repository root:  python paper_2403_13287_gb300/csrc/gen_fix_tables.py
"""
import os

import mpmath as mp

mp.mp.dps = 50
STEP = 2048          # grid points per unit of s
KMAX = 4 * STEP      # s_k up to 4
DEG = 4
SCALE = [62, 75, 56, 57, 58]
EXP_N = 4096
LOG_N = 1024


def hermite(n, x):
    h0, h1 = mp.mpf(1), 2 * x
    if n == 0:
        return h0
    for k in range(1, n):
        h0, h1 = h1, 2 * x * h1 - 2 * k * h0
    return h1


def coefficients(k):
    s = mp.mpf(k) / STEP
    g = mp.e ** (-s * s)
    e = [(-1) ** n * hermite(n, s) * g / mp.factorial(n) for n in range(DEG + 1)]
    half_erf = [mp.erf(s) / 2] + [e[n - 1] / (n * mp.sqrt(mp.pi)) for n in range(1, DEG + 1)]
    gauss = [v / (2 * mp.sqrt(mp.pi)) for v in e]
    out = []
    for f in (half_erf, gauss):
        out.append([int(mp.nint(mp.ldexp(f[n], SCALE[n] - 12 * n))) for n in range(DEG + 1)])
    return out


def main():
    here = os.path.dirname(os.path.abspath(__file__))
    lines = [
        "// Generated by gen_fix_tables.py (mpmath, 50 digits): do not edit.",
        "#pragma once",
        "",
        "#define LSKUM_FIX_KMAX %d" % KMAX,
        "",
        "struct FixRow {",
        "    int64_t t0, t1, e0, e1;         // c_0 2^62, c_1 2^75 of erf(s)/2 and of exp(-s^2)/(2 sqrt(pi))",
        "    int32_t t2, t3, t4, e2, e3, e4; // c_2 2^56, c_3 2^57, c_4 2^58",
        "    int32_t pad[2];",
        "};",
        "",
        "LSKUM_FIX_TABLE FixRow kFixErf[%d] = {" % (KMAX + 1),
    ]
    for k in range(KMAX + 1):
        t, e = coefficients(k)
        assert all(abs(v) < 2 ** 31 for v in t[2:] + e[2:]) and abs(t[1]) < 2 ** 63
        lines.append("    {%s, {0, 0}}," % ", ".join("%d%s" % (v, "ll" if i < 4 else "") for i, v in
                                                   enumerate(t[:2] + e[:2] + t[2:] + e[2:])))
    lines += ["};", "", "// 2^(j/%d) 2^62" % EXP_N, "LSKUM_FIX_TABLE int64_t kFixExp2[%d] = {" % EXP_N]
    vals = ["%dll" % int(mp.nint(mp.ldexp(mp.mpf(2) ** (mp.mpf(j) / EXP_N), 62))) for j in range(EXP_N)]
    for j in range(0, EXP_N, 4):
        lines.append("    " + ", ".join(vals[j:j + 4]) + ",")
    lines.append("};")
    a1 = mp.log(2) / (2 * EXP_N)
    lines += [
        "",
        "// 2^(u/8192) = 1 + u (a_1 + u (a_2 + u a_3)), |u| <= 1, a_n = (ln2/8192)^n / n!:",
        "// a_1 2^75, a_2 2^58, a_3 2^59; log2(e) 2^62",
        "#define LSKUM_FIX_A1 %dll" % int(mp.nint(mp.ldexp(a1, 75))),
        "#define LSKUM_FIX_A2 %d" % int(mp.nint(mp.ldexp(a1 ** 2 / 2, 58))),
        "#define LSKUM_FIX_A3 %d" % int(mp.nint(mp.ldexp(a1 ** 3 / 6, 59))),
        "#define LSKUM_FIX_LOG2E %dll" % int(mp.nint(mp.ldexp(1 / mp.log(2), 62))),
    ]
    lines += ["", "// r_j 2^32 and -log2(r_j) 2^60", "struct FixLogRow {", "    int64_t log2c;", "    uint32_t r, pad;", "};",
              "LSKUM_FIX_TABLE FixLogRow kFixLog2[%d] = {" % LOG_N]
    for j in range(LOG_N):
        r = int(mp.nint(mp.ldexp(1 / (1 + (mp.mpf(j) + mp.mpf(1) / 2) / LOG_N), 32)))
        lines.append("    {%dll, %du, 0}," % (int(mp.nint(mp.ldexp(-mp.log(mp.ldexp(mp.mpf(r), -32)) / mp.log(2), 60))), r))
    lines.append("};")
    c = [(-1) ** (n + 1) / (n * mp.log(2)) * mp.mpf(2) ** (-11 * n) for n in range(1, 6)]
    lines.append("// log2(1 + z) = u (c_1 + u (c_2 + u (c_3 + u (c_4 + u c_5)))): c_1 2^72, c_2 2^84, c_3 2^64, c_4 2^66, c_5 2^68; ln2 2^63")
    for n, q in zip(range(1, 6), (72, 84, 64, 66, 68)):
        lines.append("#define LSKUM_FIX_LOG_C%d %d%s" % (n, int(mp.nint(mp.ldexp(c[n - 1], q))), "ll" if n < 3 else ""))
    lines.append("#define LSKUM_FIX_LN2 %dll" % int(mp.nint(mp.ldexp(mp.log(2), 63))))
    with open(os.path.join(here, "fix_tables.h"), "w") as f:
        f.write("\n".join(lines) + "\n")


if __name__ == "__main__":
    main()
