"""Generate straight-line Cartesian expansion code for the CUDA kernels.

Writes ``expansion_gen.cuh``: for every order p = 0..4 a set of
``__device__`` functions, templated on the arithmetic type T, over
*scaled* symmetric coefficients (multi-index alpha = (a,b,c); scaled means
divided by alpha! = a! b! c!):

  sfmm_mono_K(v, out)     out[alpha] = v^alpha / alpha!        |alpha| <= K
  sfmm_derivs_K(u, rinv, D)  D[gamma] = d^gamma (1/|r|)        |gamma| <= K
                          from the unit vector u = r/|r| and rinv = 1/|r|
                          (McMurchie-Davidson recurrence in u, then the
                          factor rinv^(|gamma|+1): no overflow in FP32)
  sfmm_m2l_p(D, Q, C)     C[0..NM) += M_beta, C[NM..NM+NF) += F_gamma
                          (Sect. 2.2; Q scaled moments, dipole optional)
  sfmm_l2p_p(am, C, out)  potential and acceleration polynomials at a
  sfmm_m2m_p(gm, Qc, Qp)  Qp[alpha] += sum_{beta<=alpha} gm[alpha-beta] Qc[beta]
  constant tables for the lane-parallel L2L translation (App. A.2)

and the same interaction on the independent components only.  1/|r| is
harmonic, so D_{..z+2} = -D_{x+2..} - D_{..y+2..}: every derivative, and with
it every coefficient M_beta, F_gamma, is a sum of those with at most one z
(2k+1 of degree k).  Moments fold onto the same set:

  sfmm_fold_p(Q, q)          q[0] = Q_0, then the folded moments of degree
                             2..p (no dipole: the row's centre is the centre
                             of mass)
  sfmm_derivs_fold_K(x, y, z, rinv, D)    the D_gamma the interaction reads,
                             from r (products of rinv up to rinv^(2K+1))
  sfmm_uderivs_fold_K(u, rinv, D)         the same from the unit vector
  sfmm_m2l_fold_p(D, q, C)   C[0..(p+1)^2) += sums of M, without the sign;
                             then the entries E of F_gamma =
                             (-1)^|gamma| (M_gamma + E_gamma): the terms of
                             M_gamma (the unsigned sum; none for |gamma| =
                             p+1) are terms of F_gamma too, and E_gamma has
                             those of |alpha| = p+1-|gamma| (none for
                             |gamma| = p: the dipole's)
  sfmm_unfold_p[NC][SFMM_NX_p][2]         the coefficient vector from those
                             sums: (entry, factor) pairs, factor 0 unused

The layout of a coefficient vector C of order p is [M_beta for |beta| <= p]
followed by [F_gamma for 1 <= |gamma| <= p+1]; multi-indices are ordered by
degree, then a descending, then b descending.

Run: python gen_expansion.py  (build() runs it before compiling).
"""
import os
from math import factorial

PMAX = 4


def mis(K, lo=0):
    return [(a, b, n - a - b) for n in range(lo, K + 1) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


def idx_of(K, lo=0):
    return {g: i for i, g in enumerate(mis(K, lo))}


def deg(g):
    return sum(g)


def sub(a, b):
    return tuple(x - y for x, y in zip(a, b))


def add(a, b):
    return tuple(x + y for x, y in zip(a, b))


def geq(a, b):
    return all(x >= y for x, y in zip(a, b))


def lit(v):
    """A literal of type T (cast from a double literal)."""
    return "T(%r)" % float(v)


def gen_mono(K):
    I = idx_of(K)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_mono_%d(T vx, T vy, T vz, T* o) {" % K]
    lines.append("  o[0] = T(1);")
    comp = ["vx", "vy", "vz"]
    for g in mis(K, 1):
        t = next(i for i in range(3) if g[i] > 0)
        prev = list(g)
        prev[t] -= 1
        f = g[t]
        if f == 1:
            lines.append("  o[%d] = o[%d] * %s;" % (I[g], I[tuple(prev)], comp[t]))
        else:
            lines.append("  o[%d] = o[%d] * (%s * %s);" % (I[g], I[tuple(prev)], comp[t], lit(1.0 / f)))
    lines.append("}")
    return "\n".join(lines)


def gen_derivs(K):
    """D_gamma for |gamma| <= K via R^(m)_gamma in the unit vector u."""
    I = idx_of(K)
    stmts = []
    have = {}

    def R(m, g):
        key = (m, g)
        if key in have:
            return have[key]
        if deg(g) == 0:
            df = 1
            for k in range(2 * m - 1, 1, -2):
                df *= k
            val = lit(((-1) ** m) * df)
            have[key] = val
            return val
        t = next(i for i in range(3) if g[i] > 0)
        g1 = list(g)
        g1[t] -= 1
        a = R(m + 1, tuple(g1))
        name = "R%d_%d%d%d" % (m, g[0], g[1], g[2])
        expr = "u%s * %s" % ("xyz"[t], a)
        if g[t] > 1:
            g2 = list(g)
            g2[t] -= 2
            b = R(m + 1, tuple(g2))
            expr = "fma(u%s, %s, %s * %s)" % ("xyz"[t], a, lit(g[t] - 1), b)
        stmts.append("  const T %s = %s;" % (name, expr))
        have[key] = name
        return name

    body = []
    for g in mis(K):
        R(0, g)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_derivs_%d(T ux, T uy, T uz, T rinv, T* D) {" % K]
    lines += stmts
    # powers of rinv
    lines.append("  T s = rinv;")
    for n in range(K + 1):
        for g in mis(n, n):
            lines.append("  D[%d] = %s * s;" % (I[g], have[(0, g)]))
        if n < K:
            lines.append("  s = s * rinv;")
    lines.append("}")
    return "\n".join(lines)


def gen_m2l(p, skip_dipole):
    """C[M_beta] += (-1)^|b| sum_{|a|<=p-|b|} D[a+b] Q[a];
    C[NM + F_gamma] += (-1)^|g| sum_{|a|<=p+1-|g|} D[a+g] Q[a]."""
    ID = idx_of(p + 1)
    IQ = idx_of(p)
    NM = len(mis(p))
    IF = idx_of(p + 1, 1)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_m2l_%d%s(const T* D, const T* Q, T* C) {"
             % (p, "_nodip" if skip_dipole else "")]
    for b in mis(p):
        terms = [(a, ID[add(a, b)]) for a in mis(p - deg(b)) if not (skip_dipole and deg(a) == 1)]
        lines.append("  { T s = D[%d] * Q[0];" % terms[0][1])
        for a, d in terms[1:]:
            lines.append("    s = fma(D[%d], Q[%d], s);" % (d, IQ[a]))
        op = "+=" if deg(b) % 2 == 0 else "-="
        lines.append("    C[%d] %s s; }" % (IQ[b], op))
    for g in mis(p + 1, 1):
        terms = [(a, ID[add(a, g)]) for a in mis(p + 1 - deg(g)) if not (skip_dipole and deg(a) == 1)]
        lines.append("  { T s = D[%d] * Q[0];" % terms[0][1])
        for a, d in terms[1:]:
            lines.append("    s = fma(D[%d], Q[%d], s);" % (d, IQ[a]))
        op = "+=" if deg(g) % 2 == 0 else "-="
        lines.append("    C[%d] %s s; }" % (NM + IF[g], op))
    lines.append("}")
    return "\n".join(lines)


def gen_l2p(p):
    """phi = sum_b am[b] M_b ; acc_d = sum_b am[b] F_{b+e_d} (signs and G
    applied by the caller: Phi = -G phi, a = +G acc)."""
    IQ = idx_of(p)
    NM = len(mis(p))
    IF = idx_of(p + 1, 1)
    lines = ["template <typename T, typename C_T> __device__ __forceinline__ void sfmm_l2p_%d(const T* am, const C_T* C, T* out) {" % p]
    lines.append("  T phi = T(0), ax = T(0), ay = T(0), az = T(0);")
    for b in mis(p):
        i = IQ[b]
        lines.append("  phi = fma(am[%d], T(C[%d]), phi);" % (i, i))
        for d, nm in enumerate(("ax", "ay", "az")):
            e = [0, 0, 0]
            e[d] = 1
            lines.append("  %s = fma(am[%d], T(C[%d]), %s);" % (nm, i, NM + IF[add(b, tuple(e))], nm))
    lines.append("  out[0] = phi; out[1] = ax; out[2] = ay; out[3] = az;")
    lines.append("}")
    return "\n".join(lines)


def gen_m2m(p):
    IQ = idx_of(p)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_m2m_%d(const T* gm, const T* Qc, T* Qp) {" % p]
    for a in mis(p):
        terms = [(IQ[sub(a, b)], IQ[b]) for b in mis(p) if geq(a, b)]
        lines.append("  { T s = Qp[%d];" % IQ[a])
        for gi, bi in terms:
            lines.append("    s = fma(gm[%d], Qc[%d], s);" % (gi, bi))
        lines.append("    Qp[%d] = s; }" % IQ[a])
    lines.append("}")
    return "\n".join(lines)


def gen_m2m_steps(p):
    """Lane-parallel M2M: step k of moment j holds the k-th term of gen_m2m's
    sum, monomial + 256 child moment (0xffff: no more terms); exponents of
    moment j as a + 8 b + 64 c."""
    IQ = idx_of(p)
    rows = [[IQ[sub(a, b)] + 256 * IQ[b] for b in mis(p) if geq(a, b)] for a in mis(p)]
    n, steps = len(rows), max(len(r) for r in rows)
    stride = (n + 31) // 32 * 32
    body = ",\n  ".join("{" + ", ".join("%d" % (rows[j][k] if j < n and k < len(rows[j]) else 0xffff)
                                         for j in range(stride)) + "}" for k in range(steps))
    exps = ", ".join("%d" % (g[0] + 8 * g[1] + 64 * g[2]) for g in mis(p))
    return ("#define SFMM_MT_%d %d  /* steps of the M2M translation */\n" % (p, steps)
            + "static __device__ const unsigned short sfmm_m2m_steps_%d[%d][%d] = {\n  %s};\n" % (p, steps, stride, body)
            + "static __device__ const unsigned short sfmm_moment_exp_%d[%d] = {%s};\n" % (p, n, exps))


def gen_tables(p):
    """Lane-parallel L2L: target coefficient j is its own source plus
    h^(gamma_i - beta_j)/()! C_i over the other sources i of its block (M or F)
    with gamma_i >= beta_j; step k of lane j holds i + 256 t, t the index of
    the monomial in sfmm_mono_{p+1} (0xffff: no more terms)."""
    IM = mis(p)
    IF = mis(p + 1, 1)
    allc = [("M", g) for g in IM] + [("F", g) for g in IF]
    Imono = idx_of(p + 1)
    n = len(allc)
    rows = [[i + 256 * Imono[sub(g, b)] for i, (bi, g) in enumerate(allc) if bi == bj and g != b and geq(g, b)]
            for bj, b in allc]
    steps, stride = max(1, max(len(r) for r in rows)), (n + 31) // 32 * 32
    body = ",\n  ".join("{" + ", ".join("%d" % (rows[j][k] if j < n and k < len(rows[j]) else 0xffff)
                                         for j in range(stride)) + "}" for k in range(steps))
    mi_rows = ", ".join("{%d,%d,%d}" % g for g in IM)
    return ("#define SFMM_NT_%d %d  /* steps of the L2L translation */\n" % (p, steps)
            + "static __device__ const unsigned short sfmm_l2l_steps_%d[%d][%d] = {\n  %s};\n" % (p, steps, stride, body)
            + "static const int sfmm_moment_mi_%d[%d][3] = {%s};\n" % (p, len(IM), mi_rows))


def fold_of(g):
    """The component g as a combination of components with at most one z."""
    if g[2] <= 1:
        return {g: 1}
    out = {}
    for d in ((2, 0, -2), (0, 2, -2)):
        for k, v in fold_of(add(g, d)).items():
            out[k] = out.get(k, 0) - v
    return out


def kept(K, lo=0):
    return [g for g in mis(K, lo) if g[2] <= 1]


def row_mis(p):
    """Folded moments of a source row: the monopole and degrees 2..p."""
    return [(0, 0, 0)] + kept(p, 2)


def extra_mis(p):
    """F_gamma that have terms beyond those of M_gamma."""
    return [g for g in kept(p + 1, 1) if deg(g) != p]


def gen_fold(p):
    IQ = idx_of(p)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_fold_%d(const T* Q, T* q) {" % p]
    for k, r in enumerate(row_mis(p)):
        terms = [(fold_of(a).get(r, 0), IQ[a]) for a in mis(p) if deg(a) == deg(r)]
        expr = "".join((" + " if c > 0 else " - ") + ("" if abs(c) == 1 else lit(abs(c)) + " * ") + "Q[%d]" % i
                       for c, i in terms if c)
        lines.append("  q[%d] =%s;" % (k, expr[2:] if expr.startswith(" +") else expr))
    lines.append("}")
    return "\n".join(lines)


def gen_derivs_fold(K, unit):
    """D_gamma with at most one z by the McMurchie-Davidson recurrence, those
    with two (where the interaction reads them) from the Laplace equation.
    unit: in u = r/|r|, the powers of rinv multiplied in at the end (no
    overflow in FP32); else in r itself, the powers in the base values."""
    I = idx_of(K)
    stmts, have = [], {}

    def R(m, g):
        if (m, g) in have:
            return have[(m, g)]
        if deg(g) == 0:
            df = 1
            for k in range(2 * m - 1, 1, -2):
                df *= k
            val = lit(((-1) ** m) * df) if unit else "b%d" % m
            have[(m, g)] = val
            return val
        t = min((i for i in range(3) if g[i]), key=lambda i: g[i] > 1)
        a = R(m + 1, tuple(x - (i == t) for i, x in enumerate(g)))
        expr = "%s * %s" % ("xyz"[t], a)
        if g[t] > 1:
            b = R(m + 1, tuple(x - 2 * (i == t) for i, x in enumerate(g)))
            expr = "fma(%s, %s, %s)" % ("xyz"[t], a, b if g[t] == 2 else "%s * %s" % (lit(g[t] - 1), b))
        name = "R%d_%d%d%d" % (m, g[0], g[1], g[2])
        stmts.append("  const T %s = %s;" % (name, expr))
        have[(m, g)] = name
        return name

    for g in kept(K):
        R(0, g)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_%sderivs_fold_%d(T x, T y, T z, T rinv, T* D) {"
             % ("u" if unit else "", K)]
    if not unit:
        lines.append("  const T ri2 = rinv * rinv, b0 = rinv;")
        for m in range(1, K + 1):
            lines.append("  const T b%d = b%d * (ri2 * %s);" % (m, m - 1, lit(-(2 * m - 1))))
    lines += stmts
    if unit:
        lines.append("  T s = rinv;")
    for n in range(K + 1):
        for g in kept(n, n):
            lines.append("  D[%d] = %s%s;" % (I[g], have[(0, g)], " * s" if unit else ""))
        for g in mis(n, n):
            if g[2] == 2 and n >= 3:  # read as alpha + beta, both with one z
                lines.append("  D[%d] = -D[%d] - D[%d];" % (I[g], I[add(g, (2, 0, -2))], I[add(g, (0, 2, -2))]))
        if unit and n < K:
            lines.append("  s = s * rinv;")
    lines.append("}")
    return "\n".join(lines)


def gen_m2l_fold(p):
    ID = idx_of(p + 1)
    row = row_mis(p)
    lines = ["template <typename T> __device__ __forceinline__ void sfmm_m2l_fold_%d(const T* D, const T* q, T* C) {" % p]
    for k, b in enumerate(kept(p)):
        rest = [(ID[add(a, b)], i) for i, a in enumerate(row) if 2 <= deg(a) <= p - deg(b)]
        if rest:
            # the higher moments' small terms first, then the monopole
            lines.append("  { T s = D[%d] * q[%d];" % rest[0])
            for d, i in rest[1:]:
                lines.append("    s = fma(D[%d], q[%d], s);" % (d, i))
            lines.append("    C[%d] += fma(D[%d], q[0], s); }" % (k, ID[b]))
        else:
            lines.append("  C[%d] = fma(D[%d], q[0], C[%d]);" % (k, ID[b], k))
    nm = len(kept(p))
    for k, g in enumerate(extra_mis(p)):
        for i, a in enumerate(row):
            if deg(a) == p + 1 - deg(g):
                lines.append("  C[%d] = fma(D[%d], q[%d], C[%d]);" % (nm + k, ID[add(a, g)], i, nm + k))
    lines.append("}")
    return "\n".join(lines)


def gen_unfold(p):
    KM = {g: i for i, g in enumerate(kept(p))}
    KE = {g: len(KM) + i for i, g in enumerate(extra_mis(p))}
    rows = []
    for b in mis(p):
        rows.append([(KM[r], c * (-1) ** deg(b)) for r, c in fold_of(b).items()])
    for g in mis(p + 1, 1):
        row = []
        for r, c in fold_of(g).items():
            c *= (-1) ** deg(g)
            if deg(g) <= p:
                row.append((KM[r], c))
            if r in KE:
                row.append((KE[r], c))
        rows.append(row)
    nx = max(len(r) for r in rows)
    body = ",\n  ".join("{" + ", ".join("{%d, %d}" % e for e in r + [(0, 0)] * (nx - len(r))) + "}" for r in rows)
    return ("#define SFMM_NR_%d %d  /* entries of a source row */\n" % (p, len(row_mis(p)))
            + "#define SFMM_NS_%d %d  /* sums of an interaction */\n" % (p, len(KM) + len(KE))
            + "#define SFMM_NX_%d %d\nstatic __device__ const signed char sfmm_unfold_%d[%d][%d][2] = {\n  %s};\n"
            % (p, nx, p, len(rows), nx, body))


def main():
    out = [
        "// GENERATED by gen_expansion.py -- do not edit by hand.",
        "// Straight-line Cartesian expansion pieces over scaled symmetric",
        "// coefficients (multi-index alpha, divided by alpha!).  Multi-indices are",
        "// ordered by degree, then a descending, then b descending.",
        "#pragma once",
        "",
    ]
    for p in range(PMAX + 1):
        nm = len(mis(p))
        nf = len(mis(p + 1, 1))
        out.append("#define SFMM_NM_%d %d  /* potential coefficients, |beta| <= %d */" % (p, nm, p))
        out.append("#define SFMM_NF_%d %d  /* acceleration coefficients, 1 <= |gamma| <= %d */" % (p, nf, p + 1))
    out.append("")
    for K in range(PMAX + 2):
        out.append(gen_mono(K))
        out.append("")
    for K in range(1, PMAX + 2):
        out.append(gen_derivs(K))
        out.append("")
    for p in range(PMAX + 1):
        out.append(gen_m2l(p, False))
        out.append("")
        out.append(gen_m2l(p, True))
        out.append("")
        out.append(gen_l2p(p))
        out.append("")
        out.append(gen_m2m(p))
        out.append("")
        out.append(gen_tables(p))
        out.append(gen_m2m_steps(p))
        out.append(gen_fold(p))
        out.append("")
        out.append(gen_m2l_fold(p))
        out.append("")
        out.append(gen_unfold(p))
    for K in range(1, PMAX + 2):
        out.append(gen_derivs_fold(K, False))
        out.append("")
        out.append(gen_derivs_fold(K, True))
        out.append("")
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "expansion_gen.cuh")
    text = "\n".join(out) + "\n"
    old = open(path).read() if os.path.exists(path) else None
    if old != text:
        with open(path, "w") as f:
            f.write(text)
    return path


if __name__ == "__main__":
    print(main())
