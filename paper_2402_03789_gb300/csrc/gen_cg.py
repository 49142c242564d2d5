"""Emit cg_tables.cuh: unrolled real-basis Clebsch-Gordan contractions.

Build step of the CUDA library (run by the package's build()).  The real
coupling tensors follow the convention the library documents in
include/sevennet.h:
  * complex CG <l1 m1 l2 m2 | l3 m3> from the Racah formula (exact rationals);
  * carried to the real spherical-harmonic basis (z polar axis, m = -l..l,
    Condon-Shortley complex harmonics, real Y_{l,m>0} = sqrt2 (-1)^m Re Y_l^m,
    Y_{l,m<0} = sqrt2 (-1)^m Im Y_l^|m|) by the unitary U_l;
  * the non-zero real or imaginary part kept, scaled to sum C^2 = 2 l3 + 1,
    sign fixed so the first entry in (m1, m2, m3) order with |C| > 1e-9 is > 0.

For each coupling (l1, l2, l3) with l <= LMAX it writes a specialisation
    CG<l1,l2,l3>::G(Y, G)        G[m1][m3] = sum_m2 C[m1,m2,m3] Y[m2]
    CG<l1,l2,l3>::M(T, m)        m[m3] = sum_{m1,m2} C[m1,m2,m3] T[m1][m2]
    CG<l1,l2,l3>::S(S, gY)       gY[m2] += sum_{m1,m3} C[m1,m2,m3] S[m1][m3]
with every structurally zero coefficient dropped.
"""

from fractions import Fraction
import math
import os
import sys

LMAX = 3


def _f(n):
    return math.factorial(n)


def racah_cg(j1, m1, j2, m2, J, M):
    """<j1 m1 j2 m2 | J M> (integer j) as a float, via the Racah formula."""
    if M != m1 + m2 or abs(m1) > j1 or abs(m2) > j2 or abs(M) > J:
        return 0.0
    if not (abs(j1 - j2) <= J <= j1 + j2):
        return 0.0
    pre = Fraction((2 * J + 1) * _f(J + j1 - j2) * _f(J - j1 + j2) * _f(j1 + j2 - J),
                   _f(j1 + j2 + J + 1))
    pre *= _f(J + M) * _f(J - M) * _f(j1 - m1) * _f(j1 + m1) * _f(j2 - m2) * _f(j2 + m2)
    s = Fraction(0)
    for k in range(0, j1 + j2 + J + 2):
        args = [k, j1 + j2 - J - k, j1 - m1 - k, j2 + m2 - k, J - j2 + m1 + k, J - j1 - m2 + k]
        if min(args) < 0:
            continue
        den = 1
        for a in args:
            den *= _f(a)
        s += Fraction((-1) ** k, den)
    return float(s) * math.sqrt(float(pre))


def u_matrix(l):
    """U[m][m'] (indices offset by l): real = U complex."""
    s = 1.0 / math.sqrt(2.0)
    U = [[0j] * (2 * l + 1) for _ in range(2 * l + 1)]
    for m in range(-l, l + 1):
        if m == 0:
            U[l][l] = 1.0 + 0j
        elif m > 0:
            U[m + l][m + l] = (-1) ** m * s
            U[m + l][-m + l] = s + 0j
        else:
            a = -m
            U[m + l][-a + l] = 1j * s
            U[m + l][a + l] = -1j * (-1) ** a * s
    return U


def real_cg_table(l1, l2, l3):
    U1, U2, U3 = u_matrix(l1), u_matrix(l2), u_matrix(l3)
    n1, n2, n3 = 2 * l1 + 1, 2 * l2 + 1, 2 * l3 + 1
    Cc = [[[racah_cg(l1, a - l1, l2, b - l2, l3, c - l3) for c in range(n3)]
           for b in range(n2)] for a in range(n1)]
    T = [[[0j] * n3 for _ in range(n2)] for _ in range(n1)]
    for a in range(n1):
        for b in range(n2):
            for c in range(n3):
                acc = 0j
                for x in range(n1):
                    if U1[a][x] == 0:
                        continue
                    for y in range(n2):
                        if U2[b][y] == 0:
                            continue
                        for z in range(n3):
                            if U3[c][z] == 0 or Cc[x][y][z] == 0:
                                continue
                            acc += U3[c][z] * Cc[x][y][z] * U1[a][x].conjugate() * U2[b][y].conjugate()
                T[a][b][c] = acc
    re = max(abs(T[a][b][c].real) for a in range(n1) for b in range(n2) for c in range(n3))
    im = max(abs(T[a][b][c].imag) for a in range(n1) for b in range(n2) for c in range(n3))
    part = (lambda z: z.real) if re >= im else (lambda z: z.imag)
    R = [[[part(T[a][b][c]) for c in range(n3)] for b in range(n2)] for a in range(n1)]
    norm = sum(R[a][b][c] ** 2 for a in range(n1) for b in range(n2) for c in range(n3))
    sc = math.sqrt(n3 / norm)
    R = [[[R[a][b][c] * sc for c in range(n3)] for b in range(n2)] for a in range(n1)]
    first = next(R[a][b][c] for a in range(n1) for b in range(n2) for c in range(n3)
                 if abs(R[a][b][c]) > 1e-9)
    sign = 1.0 if first > 0 else -1.0
    out = {}
    for a in range(n1):
        for b in range(n2):
            for c in range(n3):
                v = sign * R[a][b][c]
                if abs(v) > 1e-9:
                    out[(a, b, c)] = v
    return out


def _lit(v):
    return "%.9ef" % v


def emit(path):
    lines = [
        "// Generated by gen_cg.py -- real-basis Clebsch-Gordan contractions.",
        "// Do not edit; rerun the generator.",
        "#pragma once",
        "",
        "template <int L1, int L2, int L3> struct CG;",
        "",
    ]
    nnz_total = {}
    for l1 in range(LMAX + 1):
        for l2 in range(LMAX + 1):
            for l3 in range(abs(l1 - l2), min(l1 + l2, LMAX) + 1):
                tab = real_cg_table(l1, l2, l3)
                nnz_total[(l1, l2, l3)] = len(tab)
                n3 = 2 * l3 + 1
                lines.append(f"// coupling {l1} x {l2} -> {l3}: {len(tab)} non-zero coefficients")
                lines.append(f"template <> struct CG<{l1}, {l2}, {l3}> {{")
                lines.append(f"  static constexpr int NNZ = {len(tab)};")
                lines.append("  static __device__ __forceinline__ void G(const float* __restrict__ Y, float* __restrict__ g) {")
                for a in range(2 * l1 + 1):
                    for c in range(n3):
                        terms = [(b, v) for (aa, b, cc), v in sorted(tab.items()) if aa == a and cc == c]
                        if not terms:
                            expr = "0.0f"
                        else:
                            expr = " + ".join(f"{_lit(v)} * Y[{b}]" for b, v in terms)
                        lines.append(f"    g[{a * n3 + c}] = {expr};")
                lines.append("  }")
                lines.append("  static __device__ __forceinline__ void M(const float* __restrict__ T, float* __restrict__ m) {")
                for c in range(n3):
                    terms = [(a, b, v) for (a, b, cc), v in sorted(tab.items()) if cc == c]
                    expr = " + ".join(f"{_lit(v)} * T[{a * (2 * l2 + 1) + b}]" for a, b, v in terms)
                    lines.append(f"    m[{c}] = {expr};")
                lines.append("  }")
                lines.append("  static __device__ __forceinline__ void S(const float* __restrict__ s, float* __restrict__ gy) {")
                for bb in range(2 * l2 + 1):
                    terms = [(a, c, v) for (a, b2, c), v in sorted(tab.items()) if b2 == bb]
                    for a, c, v in terms:
                        lines.append(f"    gy[{bb}] = fmaf({_lit(v)}, s[{a * n3 + c}], gy[{bb}]);")
                lines.append("  }")
                lines.append("};")
                lines.append("")
    couplings = [f"X({a}, {b}, {c})" for a in range(LMAX + 1) for b in range(LMAX + 1)
                 for c in range(abs(a - b), min(a + b, LMAX) + 1)]
    lines.append("// every coupling with l <= LMAX in canonical (l1, l2, l3) order")
    lines.append("#define SN_FOR_EACH_COUPLING(X) " + " ".join(couplings))
    low = [f"X({a}, {b}, {c})" for a in range(3) for b in range(3) for c in range(abs(a - b), min(a + b, 2) + 1)]
    lines.append("// the couplings with every l <= 2")
    lines.append("#define SN_FOR_EACH_COUPLING_L2(X) " + " ".join(low))
    lines.append("")
    with open(path, "w") as fh:
        fh.write("\n".join(lines) + "\n")
    return nnz_total


if __name__ == "__main__":
    out = sys.argv[1] if len(sys.argv) > 1 else os.path.join(os.path.dirname(__file__), "cg_tables.cuh")
    nnz = emit(out)
    print("wrote", out, "couplings:", len(nnz))
