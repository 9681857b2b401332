// Floating-point expansions: a value carried as an unevaluated sum of three
// floats (about 70 bits), evaluated with error-free transformations (TwoSum,
// Knuth; Fast2Sum, Dekker 1971; TwoProduct with a fused multiply-add), two
// values at a time in the packed FP32 instructions.
//
// Why: GB300's FP64 pipe takes about 80 cycles per warp instruction and SM
// quarter (measured with a chain of DADD), its FP32 pipe one.  An unsoftened
// pair takes 23 FP64 instructions (about 1380 cycles measured in isolation)
// or the 290 FP32 operations below (360 cycles).
//
// Accuracy of one pair against 113-bit arithmetic (2x10^5 random pairs,
// separations of 1e-2 to 1e-4 of the box): force 2^-62.4 rms, 2^-56 at worst,
// potential 2^-64.7 and 2^-57; the FP64 evaluation 2^-51.9 and 2^-49.9,
// 2^-53.3 and 2^-51.5.
#pragma once
#include "sfmm_common.cuh"

namespace sfmm {
namespace fexp {

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __fadd2_rn(a, neg(b)); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vmax(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ float2 vmin(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }

// s + e == a + b; |a| >= |b|, or a a multiple of a power of two that |b| does not exceed
__device__ __forceinline__ void fast2sum(float2 a, float2 b, float2& s, float2& e) {
  s = add(a, b);
  e = sub(b, sub(s, a));
}
__device__ __forceinline__ void two_sum(float2 a, float2 b, float2& s, float2& e) {
  s = add(a, b);
  const float2 t = sub(s, a);
  e = add(sub(a, sub(s, t)), sub(b, t));
}
// the same for a, b >= 0: the larger one leads (the comparison runs on another pipe)
__device__ __forceinline__ void two_sum_pos(float2 a, float2 b, float2& s, float2& e) {
  fast2sum(vmax(a, b), vmin(a, b), s, e);
}
__device__ __forceinline__ void two_prod(float2 a, float2 b, float2& p, float2& e) {
  p = mul(a, b);
  e = fma(a, b, neg(p));
}
// A += t with A far larger than t; the exact rounding error joins lo
__device__ __forceinline__ void grow(float2& A, float2 t, float2& lo) {
  const float2 s = add(A, t);
  lo = add(lo, sub(t, sub(s, A)));
  A = s;
}
__device__ __forceinline__ void shrink(float2& A, float2 t, float2& lo) {
  const float2 s = sub(A, t);
  lo = sub(lo, add(t, sub(s, A)));
  A = s;
}

// One value split into three floats: h on the grid 2^-22, m on the grid
// 2^-45 (both of at most 23 bits for |x| < 1, so that differences of two
// values' h and m are exact), l the rest (24 bits).
__device__ __forceinline__ void split_grid(double x, float& h, float& m, float& l) {
  const double c1 = 6755399441055744.0 * 0x1p-22, c2 = 6755399441055744.0 * 0x1p-45;  // 1.5 2^52 grid
  const double a = __dsub_rn(__dadd_rn(x, c1), c1);
  const double r = __dsub_rn(x, a);
  const double b = __dsub_rn(__dadd_rn(r, c2), c2);
  h = (float)a;
  m = (float)b;
  l = (float)__dsub_rn(r, b);
}
// A positive value as three floats of 24 bits.
__device__ __forceinline__ void split_plain(double x, float& h, float& m, float& l) {
  h = (float)x;
  const double r = __dsub_rn(x, (double)h);
  m = (float)r;
  l = (float)__dsub_rn(r, (double)m);
}

// Sums of one run of pairs: force (3) and potential, each in three levels.
// Levels 0 and 1 carry a bias (a power of two times 1.5, far above the sums)
// so that adding to them is exact but for a remainder that moves to the next
// level; their sums are multiples of the bias's last place.
struct PairSums {
  float2 a0[4], a1[4], a2[4];
};

// Two unsoftened pairs: target at (xh, xm, xl), sources negated at q[0..8]
// (x, y, z: h, m, l each), masses q[9..11].  off: halves to leave out (their
// sources get zero weight).  Returns the leading part of r^2 through r2.
// F -= m r^-3 d and pot -= m / r are accumulated with positive sign (the
// caller negates).
__device__ __forceinline__ float2 separation(const float2 (&x)[9], const float2* q, float2 (&D0)[3], float2 (&D1)[3],
                                             float2 (&D2)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // h and m differences are exact multiples of their grids, and an m
    // difference is at most one step of the h grid: Fast2Sum applies
    const float2 a = add(x[3 * c], q[3 * c]), b = add(x[3 * c + 1], q[3 * c + 1]), l = add(x[3 * c + 2], q[3 * c + 2]);
    float2 e;
    fast2sum(a, b, D0[c], e);
    fast2sum(e, l, D1[c], D2[c]);
  }
  return fma(D0[0], D0[0], fma(D0[1], D0[1], mul(D0[2], D0[2])));
}

__device__ __forceinline__ void unsoftened(const float2 (&D0)[3], const float2 (&D1)[3], const float2 (&D2)[3],
                                           float2 m0, float2 m1, float2 m2, bool offx, bool offy, PairSums& S) {
  // r^2 = R + U + W (24 bits, order 2^-24, order 2^-48)
  float2 p[3], e1[3], q1[3], W;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    two_prod(D0[c], D0[c], p[c], e1[c]);
    const float2 T = add(D0[c], D0[c]);
    float2 f;
    two_prod(T, D1[c], q1[c], f);
    const float2 s = fma(D1[c], D1[c], fma(T, D2[c], f));
    W = c ? add(W, s) : s;
  }
  float2 A, a1, R, a2;
  two_sum_pos(p[0], p[1], A, a1);
  two_sum_pos(A, p[2], R, a2);
  const float2 V0 = mul(R, dup(0x1p-19f));
  float2 V = V0;
  grow(V, a1, W);
  grow(V, a2, W);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    grow(V, e1[c], W);
    grow(V, q1[c], W);
  }
  const float2 U = sub(V, V0);
  // y ~ 1/r, q = y^2, and the remainder e = 1 - r^2 q = E0 + E1, |e| < 2^-20
  float2 y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(R.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(R.y));
  if (offx) y.x = 0.0f;
  if (offy) y.y = 0.0f;
  float2 q0, qe, P, Pe, h1, h1e, h2, h2e;
  two_prod(y, y, q0, qe);
  two_prod(R, q0, P, Pe);
  two_prod(R, qe, h1, h1e);
  two_prod(U, q0, h2, h2e);
  float2 E1 = neg(fma(U, qe, add(fma(W, q0, h1e), h2e)));
  const float2 C = dup(0x1.8p-18f);
  float2 X = add(C, sub(dup(1.0f), P));  // exact: 1 - P has few bits
  shrink(X, Pe, E1);
  shrink(X, h1, E1);
  shrink(X, h2, E1);
  const float2 E0 = sub(X, C);
  // 1/r = y (1 + d1), 1/r^3 = y^3 (1 + d3), d = leading + remainder
  const float2 ee = mul(E0, E0);
  const float2 d30 = mul(dup(1.5f), E0),
               d31 = fma(dup(1.5f), E1, mul(ee, fma(dup(35.0f / 16.0f), E0, dup(15.0f / 8.0f))));
  const float2 d10 = mul(dup(0.5f), E0),
               d11 = fma(dup(0.5f), E1, mul(ee, fma(dup(5.0f / 16.0f), E0, dup(3.0f / 8.0f))));
  // w = m y
  float2 w0, we, t1, t1e, w1, w2;
  two_prod(m0, y, w0, we);
  two_prod(m1, y, t1, t1e);
  two_sum(we, t1, w1, w2);
  w2 = fma(m2, y, add(w2, t1e));
  // s = w q (1 + d3) = s0 + s1 + s2
  float2 s0, ve, g1, g1e, g2, g2e, x3, x3e;
  two_prod(w0, q0, s0, ve);
  two_prod(w0, qe, g1, g1e);
  two_prod(w1, q0, g2, g2e);
  two_prod(s0, d30, x3, x3e);
  float2 s2 = add(add(g1e, g2e), x3e);
  s2 = fma(w1, qe, s2);
  s2 = fma(w2, q0, s2);
  s2 = fma(s0, d31, s2);
  const float2 B0 = mul(s0, dup(0x1p-17f));
  float2 B = B0;
  grow(B, ve, s2);
  grow(B, g1, s2);
  grow(B, g2, s2);
  const float2 v1 = sub(B, B0);  // (before d3: its product with d3 is of order 2^-46)
  s2 = fma(v1, d30, s2);
  grow(B, x3, s2);
  const float2 s1 = sub(B, B0);
  // force s d, potential w (1 + d1)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float2 t0, t0e, u1, u1e, u2, u2e;
    two_prod(s0, D0[c], t0, t0e);
    two_prod(s0, D1[c], u1, u1e);
    two_prod(s1, D0[c], u2, u2e);
    float2 o = add(fma(s0, D2[c], u1e), u2e);
    o = fma(s1, D1[c], o);
    o = fma(s2, D0[c], o);
    const float2 n = add(S.a0[c], t0);
    const float2 l = sub(t0, sub(n, S.a0[c]));
    S.a0[c] = n;
    grow(S.a1[c], l, o);
    grow(S.a1[c], t0e, o);
    grow(S.a1[c], u1, o);
    grow(S.a1[c], u2, o);
    S.a2[c] = add(S.a2[c], o);
  }
  {
    float2 x1, x1e;
    two_prod(w0, d10, x1, x1e);
    float2 o = add(w2, x1e);
    o = fma(w0, d11, o);
    o = fma(w1, d10, o);
    const float2 n = add(S.a0[3], w0);
    const float2 l = sub(w0, sub(n, S.a0[3]));
    S.a0[3] = n;
    grow(S.a1[3], l, o);
    grow(S.a1[3], w1, o);
    grow(S.a1[3], x1, o);
    S.a2[3] = add(S.a2[3], o);
  }
}

}  // namespace fexp
}  // namespace sfmm
