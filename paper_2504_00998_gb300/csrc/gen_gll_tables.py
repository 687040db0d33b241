"""Writes fe_gll_tables.h: the shape-only 1D tables of the Hamiltonian sweep kernel and of the
Gauss-quadrature potential kernel.

They depend on the degree p only; the mesh enters through scalars at run time.  K1, M1 are the
exactly integrated 1D stiffness and mass matrices of the Lagrange basis on the p + 1
Gauss-Lobatto-Legendre nodes of [-1, 1], sig_k = 1 / sqrt(m_k) (m_k = w_k, or 2 w_0 at a node
shared by two cells).  GB[q][i] = l_i(g_q) interpolates from the GLL nodes to the p + 1
Gauss-Legendre points g_q of [-1, 1] (the potential integrated by Gauss quadrature).

The sweep kernel (fe_sweep.cuh) takes the symmetrically scaled tables, in double:
  KH[j][k] = sig_j K1[j][k] sig_k,  GH[j][k] = sig_j G1[j][k] sig_k  (G1 = int l_j l_k'),
  TH[j] = sqrt(p (p + 1) / (2 (2 p + 1))) sig_j w_j P_p(x_j):
the exact mass differs from the GLL-lumped one only in the L_p . L_p product (the rule is exact
to degree 2 p - 1; <L_p, L_p> is 2 / (2 p + 1) exactly and 2 / p by the rule), so
M1 = diag(w) - g (w P_p)(w P_p)^T with g = (p / 2)^2 (2 / p - 2 / (2 p + 1)).
NH[j] = 1 / sig_j is the constant function in the scaled variables (KH NH = 0).  The rules are computed the way the library's mesh set-up computes them
(three-term Legendre recurrence, Newton from the same starting points, (p+1)-point Gauss
quadrature of the products) and rounded to float.

Run: python gen_gll_tables.py  (writes fe_gll_tables.h beside this script).
"""
import math
import os


def legendre(n, x):
    p0, p1 = 1.0, x
    if n == 0:
        return 1.0, 0.0
    for k in range(2, n + 1):
        p0, p1 = p1, ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k
    dp = n * (x * p1 - p0) / (x * x - 1.0) if abs(x * x - 1.0) > 1e-300 else 0.0
    return p1, dp


def gll_rule(p):
    x = [0.0] * (p + 1)
    x[0], x[p] = -1.0, 1.0
    for i in range(1, p):
        t = -math.cos(math.pi * i / p)
        for _ in range(100):
            P, dP = legendre(p, t)
            d2 = (2.0 * t * dP - p * (p + 1.0) * P) / (1.0 - t * t)
            dt = dP / d2
            t -= dt
            if abs(dt) < 1e-16:
                break
        x[i] = t
    w = [2.0 / (p * (p + 1.0) * legendre(p, xi)[0] ** 2) for xi in x]
    return x, w


def gauss_rule(q):
    xs, ws = [], []
    for i in range(q):
        t = math.cos(math.pi * (i + 0.75) / (q + 0.5))
        for _ in range(100):
            P, dP = legendre(q, t)
            dt = P / dP
            t -= dt
            if abs(dt) < 1e-16:
                break
        P, dP = legendre(q, t)
        xs.append(t)
        ws.append(2.0 / ((1.0 - t * t) * dP * dP))
    return xs, ws


def lagrange(xn, i, t):
    v, d = 1.0, 0.0
    for j in range(len(xn)):
        if j == i:
            continue
        f = (t - xn[j]) / (xn[i] - xn[j])
        d = d * f + v / (xn[i] - xn[j])
        v *= f
    return v, d


def hat_tables(p):
    n1 = p + 1
    xi, w = gll_rule(p)
    gq, gw = gauss_rule(n1)
    K1 = [[0.0] * n1 for _ in range(n1)]
    G1 = [[0.0] * n1 for _ in range(n1)]
    for a in range(n1):
        ld = [lagrange(xi, i, gq[a]) for i in range(n1)]
        for i in range(n1):
            for j in range(n1):
                K1[i][j] += gw[a] * ld[i][1] * ld[j][1]
                G1[i][j] += gw[a] * ld[i][0] * ld[j][1]
    sig = [1.0 / math.sqrt(2.0 * w[0] if k in (0, p) else w[k]) for k in range(n1)]
    KH = [[sig[j] * K1[j][k] * sig[k] for k in range(n1)] for j in range(n1)]
    GH = [[sig[j] * G1[j][k] * sig[k] for k in range(n1)] for j in range(n1)]
    c = math.sqrt(p * (p + 1.0) / (2.0 * (2.0 * p + 1.0)))
    TH = [c * sig[j] * w[j] * legendre(p, xi[j])[0] for j in range(n1)]
    return KH, GH, TH, [1.0 / v for v in sig]


def gauss_interp(p):
    xi, _ = gll_rule(p)
    gq = sorted(gauss_rule(p + 1)[0])   # ascending, as the points of a cell are ordered
    return [[lagrange(xi, i, gq[q])[0] for i in range(p + 1)] for q in range(p + 1)]


def emit_double(name, A):
    rows = ",\n    ".join("{" + ", ".join(repr(v) for v in r) + "}" for r in A)
    return f"__device__ constexpr double {name}[{len(A)}][{len(A[0])}] = {{\n    {rows}}};\n"


def main():
    out = ["// Generated by gen_gll_tables.py (do not edit): the GLL-to-Gauss interpolation GB and the",
           "// tables KH, GH, TH, NH of the sweep kernel for p = 1..6 (see the script for their",
           "// definition).",
           "#pragma once", "", "namespace fe {", ""]
    for p in range(1, 7):
        out.append(emit_double(f"kGaussB{p}", gauss_interp(p)))
        KH, GH, TH, NH = hat_tables(p)
        out.append(emit_double(f"kHatK{p}", KH))
        out.append(emit_double(f"kHatG{p}", GH))
        out.append(emit_double(f"kHatT{p}", [TH]))
        out.append(emit_double(f"kHatN{p}", [NH]))
    out.append("""// GB[q][i] of degree P
template <int P>
__device__ __forceinline__ constexpr double gauss_b(int q, int i) {
  if constexpr (P == 1) return kGaussB1[q][i];
  else if constexpr (P == 2) return kGaussB2[q][i];
  else if constexpr (P == 3) return kGaussB3[q][i];
  else if constexpr (P == 4) return kGaussB4[q][i];
  else if constexpr (P == 5) return kGaussB5[q][i];
  else return kGaussB6[q][i];
}
// KH[j][k], GH[j][k], TH[j] and NH[j] of degree P
template <int P>
__device__ __forceinline__ constexpr double hat_k(int j, int k) {
  if constexpr (P == 1) return kHatK1[j][k];
  else if constexpr (P == 2) return kHatK2[j][k];
  else if constexpr (P == 3) return kHatK3[j][k];
  else if constexpr (P == 4) return kHatK4[j][k];
  else if constexpr (P == 5) return kHatK5[j][k];
  else return kHatK6[j][k];
}
template <int P>
__device__ __forceinline__ constexpr double hat_g(int j, int k) {
  if constexpr (P == 1) return kHatG1[j][k];
  else if constexpr (P == 2) return kHatG2[j][k];
  else if constexpr (P == 3) return kHatG3[j][k];
  else if constexpr (P == 4) return kHatG4[j][k];
  else if constexpr (P == 5) return kHatG5[j][k];
  else return kHatG6[j][k];
}
template <int P>
__device__ __forceinline__ constexpr double hat_t(int j) {
  if constexpr (P == 1) return kHatT1[0][j];
  else if constexpr (P == 2) return kHatT2[0][j];
  else if constexpr (P == 3) return kHatT3[0][j];
  else if constexpr (P == 4) return kHatT4[0][j];
  else if constexpr (P == 5) return kHatT5[0][j];
  else return kHatT6[0][j];
}
template <int P>
__device__ __forceinline__ constexpr double hat_n(int j) {
  if constexpr (P == 1) return kHatN1[0][j];
  else if constexpr (P == 2) return kHatN2[0][j];
  else if constexpr (P == 3) return kHatN3[0][j];
  else if constexpr (P == 4) return kHatN4[0][j];
  else if constexpr (P == 5) return kHatN5[0][j];
  else return kHatN6[0][j];
}

}  // namespace fe""")
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fe_gll_tables.h")
    with open(path, "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
