"""Write forward_f64.h and forward_df.h: the tables of the double-precision and
float-pair forward passes, computed in 40-digit arithmetic with mpmath.

    python paper_2206_03719_gb300/csrc/gen_forward_f64.py

Quantile: Phi^-1(p) for p in [2^-(OCT+1), 1/2), one degree-6 polynomial per
segment: octave k = 1..OCT is p in [2^-(k+1), 2^-k), cut in SEG segments of
equal width.  In a segment t in [-1/2, 1/2) runs linearly over p.  Each
polynomial interpolates at seven Chebyshev nodes.  Stored coefficient-major
([(k - 1) * SEG + segment]): c_0 as a double, c_1..c_3 as pairs of floats,
c_4..c_6 as floats.

Exponential: 2^(j / EXPN), j = 0..EXPN-1, and the coefficients of
2^(f / EXPN) - 1 on |f| <= 1/2 (Taylor to f^3, the f^4 term economised onto
f^2), for f in units of 2^-22 (the stepper's integer split of the log price).

Float pairs: the same segments at degree 5 (c_0..c_2 as pairs, the others as
floats) and 2^(j / EXPN_DF) as pairs.
"""
import os

import mpmath as mp
import numpy as np

mp.mp.dps = 40
OCT, SEG, DEG = 10, 64, 6
EXPN = 2048
DEG_DF, EXPN_DF = 5, 1024


def quantile(p):
    return -mp.sqrt(2) * mp.erfinv(1 - 2 * p)


def segment(k, i, DEG=DEG):
    """coefficients of the segment's polynomial in t, and its error"""
    left = mp.mpf(2) ** -(k + 1) * (1 + mp.mpf(i) / SEG)
    width = mp.mpf(2) ** -(k + 1) / SEG
    nodes = [mp.cos(mp.pi * (j + mp.mpf(0.5)) / (DEG + 1)) / 2 for j in range(DEG + 1)]
    A = mp.matrix(DEG + 1, DEG + 1)
    b = mp.matrix(DEG + 1, 1)
    for r, t in enumerate(nodes):
        for j in range(DEG + 1):
            A[r, j] = t ** j
        b[r] = quantile(left + width * (t + mp.mpf(0.5)))
    sol = mp.lu_solve(A, b)
    c = list(sol)
    worst = mp.mpf(0)
    for s in (-0.5, -0.37, -0.2, 0.0, 0.11, 0.3, 0.45, 0.5):
        v = mp.mpf(0)
        for x in reversed(c):
            v = v * s + x
        worst = max(worst, abs(v - quantile(left + width * (mp.mpf(s) + mp.mpf(0.5)))))
    return c, float(worst)


def pair(x):
    """(hi, lo) floats of an mp value"""
    hi = np.float32(float(x))
    return hi, np.float32(float(mp.mpf(x) - mp.mpf(float(hi))))


def main():
    rows = [[] for _ in range(DEG + 1)]
    worst = 0.0
    for k in range(1, OCT + 1):
        for i in range(SEG):
            c, e = segment(k, i)
            worst = max(worst, e / max(1.0, abs(float(c[0]))))
            for j in range(DEG + 1):
                rows[j].append(c[j])
    print("largest segment error, max(1, |z|) relative: %.3g" % worst)
    L = mp.log(2) / EXPN
    S = mp.mpf(2) ** -22
    a1, a2, a3 = L * S, (L ** 2 / 2 + L ** 4 / 96) * S ** 2, L ** 3 / 6 * S ** 3
    here = os.path.dirname(os.path.abspath(__file__))
    f2 = lambda x: "{%.9ef, %.9ef}" % pair(x)  # noqa: E731
    with open(os.path.join(here, "forward_f64.h"), "w") as f:
        f.write("// forward_f64.h -- written by gen_forward_f64.py (40-digit mpmath); do not edit.\n"
                "#pragma once\n\nnamespace lsmc {\n\n"
                "constexpr int kQsOct = %d, kQsSeg = %d;  // octaves, segments\n"
                "constexpr int kExpN = %d, kExpNLog2 = %d;\n"
                "constexpr double kExpUnit = %.17e;  // kExpN / ln 2, as a pair\n"
                "constexpr double kExpUnitLo = %.17e;\n"
                "constexpr double kExpUnitInv = %.17e;\n"
                "constexpr float kExpA1 = %.9ef, kExpA1Lo = %.9ef;\n"
                "constexpr float kExpA2 = %.9ef, kExpA2Lo = %.9ef;\n"
                "constexpr float kExpA3 = %.9ef;\n\n"
                "struct F64Tables {\n"
                "  double q0[kQsOct * kQsSeg];     // quantile segments: c_0\n"
                "  float2 qp[3][kQsOct * kQsSeg];  // c_1, c_2, c_3 as pairs\n"
                "  float qf[3][kQsOct * kQsSeg];   // c_4, c_5, c_6\n"
                "  double exp2[kExpN];             // 2^(j / kExpN)\n"
                "};\n\n" % ((OCT, SEG, EXPN, EXPN.bit_length() - 1, float(1 / L),
                              float(1 / L - mp.mpf(float(1 / L))), float(L)) + pair(a1) + pair(a2) +
                             (float(a3),)))
        f.write("static __device__ const F64Tables kF64Tables = {\n    {\n")
        for i in range(0, len(rows[0]), 4):
            f.write("        " + " ".join("%.17e," % float(v) for v in rows[0][i:i + 4]) + "\n")
        f.write("    },\n    {\n")
        for r in rows[1:4]:
            f.write("        {\n")
            for i in range(0, len(r), 4):
                f.write("            " + " ".join(f2(v) + "," for v in r[i:i + 4]) + "\n")
            f.write("        },\n")
        f.write("    },\n    {\n")
        for r in rows[4:]:
            f.write("        {\n")
            for i in range(0, len(r), 6):
                f.write("            " + " ".join("%.9ef," % float(v) for v in r[i:i + 6]) + "\n")
            f.write("        },\n")
        f.write("    },\n    {\n")
        e = [float(mp.mpf(2) ** (mp.mpf(j) / EXPN)) for j in range(EXPN)]
        for i in range(0, EXPN, 4):
            f.write("        " + " ".join("%.17e," % v for v in e[i:i + 4]) + "\n")
        f.write("    },\n};\n\n}  // namespace lsmc\n")


def main_df():
    rows = [[] for _ in range(DEG_DF + 1)]
    for k in range(1, OCT + 1):
        for i in range(SEG):
            for j, c in enumerate(segment(k, i, DEG_DF)[0]):
                rows[j].append(c)
    L = mp.log(2) / EXPN_DF
    here = os.path.dirname(os.path.abspath(__file__))
    with open(os.path.join(here, "forward_df.h"), "w") as f:
        f.write("// forward_df.h -- written by gen_forward_f64.py (40-digit mpmath); do not edit.\n"
                "#pragma once\n\nnamespace lsmc {\n\n"
                "constexpr int kDfExpN = %d, kDfExpNLog2 = %d;\n"
                "constexpr double kDfExpUnit = %.17e;  // kDfExpN / ln 2\n"
                "constexpr float kDfExpA1 = %.9ef, kDfExpA1Lo = %.9ef;\n"
                "constexpr float kDfExpA2 = %.9ef, kDfExpA2Lo = %.9ef, kDfExpA3 = %.9ef;\n\n"
                "struct DfForward {\n"
                "  float2 qp[3][%d];  // quantile segments: c_0, c_1, c_2 as pairs\n"
                "  float qf[%d][%d];   // c_3, c_4, c_5\n"
                "  float2 exp2[kDfExpN];  // 2^(j / kDfExpN)\n"
                "};\n\n" % ((EXPN_DF, EXPN_DF.bit_length() - 1, float(1 / L)) + pair(L) +
                            pair(L ** 2 / 2) + (float(L ** 3 / 6), OCT * SEG, DEG_DF - 2, OCT * SEG)))
        f.write("static __device__ const DfForward kDfForward = {\n    {\n")
        f2 = lambda x: "{%.9ef, %.9ef}" % pair(x)  # noqa: E731
        for r in rows[:3]:
            f.write("        {\n")
            for i in range(0, len(r), 4):
                f.write("            " + " ".join(f2(v) + "," for v in r[i:i + 4]) + "\n")
            f.write("        },\n")
        f.write("    },\n    {\n")
        for r in rows[3:]:
            f.write("        {\n")
            for i in range(0, len(r), 6):
                f.write("            " + " ".join("%.9ef," % float(v) for v in r[i:i + 6]) + "\n")
            f.write("        },\n")
        f.write("    },\n    {\n")
        for i in range(0, EXPN_DF, 4):
            f.write("        " + " ".join(f2(mp.mpf(2) ** (mp.mpf(j) / EXPN_DF)) + ","
                                          for j in range(i, i + 4)) + "\n")
        f.write("    },\n};\n\n}  // namespace lsmc\n")


if __name__ == "__main__":
    main()
    main_df()
