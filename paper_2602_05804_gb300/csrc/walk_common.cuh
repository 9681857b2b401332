// Device pieces shared by the two walk kernels (walk.cu: one warp per leaf,
// replaying Algorithm 1 for the leaf's branch; walk_shared.cu: one warp per
// node, each node's pairs evaluated once): the acceptance test of Sect. 3,
// the node-node expansion (Eq. dmkdeffmm) of one pair, the warp
// reduce-scatter of coefficients and the generated expansion dispatch.
#pragma once
#include <type_traits>

#include "expansion_gen.cuh"
#include "sfmm_internal.cuh"

namespace sfmm {

#define WALK_WARPS 4
#define WALK_NT (WALK_WARPS * 32)
#define WALK_MQ 64

enum { MODE_COMPUTE = 0, MODE_COUNT = 1, MODE_WRITE = 2 };

struct WalkArgs {
  int nleaves;
  const int* leaf_node;
  const int* nfirst;
  const int* ncount;
  const int* nright;
  const float4* geo_hi;
  const float4* geo_lo;
  const double* ncx;
  const double* ncy;
  const double* ncz;
  const double* nsize;
  const double* nhmax;
  const float* Qf;
  const double* Qd;
  int nqs;  // row stride of Qf
  const float* row32;   // source rows of the shared walk, by form (row_len)
  const double* row64;
  const float4* prel;
  const double* px;
  const double* py;
  const double* pz;
  int* ring;
  int ring_cap;  // power of two
  int* leaf_counter;
  int* arena;
  unsigned long long* arena_counter;
  long long arena_cap;
  long long* p2p_off;
  int* p2p_cnt;
  float4* far32;
  double* far64;
  int* status;
  unsigned long long* stat;  // m2l, m2l_unique, p2p_leaves, p2p_pairs, fallbacks
  double theta;
  float theta_f;
  float theta2_f;
  const int* psys;            // system of each particle (null: one system)
  const int* sys_root;        // root node of each system
  int* m2l_cnt;               // MODE_COUNT
  const long long* m2l_off;   // MODE_WRITE
  int* dump_level;
  int* dump_src;
};

template <int P> struct Exp;
#define SFMM_EXP(PP, PP1)                                                                                      \
  template <> struct Exp<PP> {                                                                                 \
    static constexpr int NM = SFMM_NM_##PP, NF = SFMM_NF_##PP, NC = NM + NF;                                   \
    static constexpr int NQ = ncoef(PP), NMONO1 = ncoef(PP + 1);                                               \
    template <typename T> __device__ static void derivs(T x, T y, T z, T ri, T* D) { sfmm_derivs_##PP1(x, y, z, ri, D); } \
    template <typename T> __device__ static void m2l(const T* D, const T* Q, T* C) { sfmm_m2l_##PP(D, Q, C); }  \
    template <typename T> __device__ static void m2l_nodip(const T* D, const T* Q, T* C) { sfmm_m2l_##PP##_nodip(D, Q, C); } \
    template <typename T, typename U> __device__ static void l2p(const T* am, const U* C, T* o) { sfmm_l2p_##PP(am, C, o); } \
    template <typename T> __device__ static void mono(T x, T y, T z, T* o) { sfmm_mono_##PP(x, y, z, o); }     \
    template <typename T> __device__ static void mono1(T x, T y, T z, T* o) { sfmm_mono_##PP1(x, y, z, o); }   \
    static constexpr int NT = SFMM_NT_##PP, TS = (NC + 31) / 32 * 32;  /* L2L: steps, stride */                \
    __device__ static const unsigned short* table() { return &sfmm_l2l_steps_##PP[0][0]; }                    \
    /* independent components (at most one z): source rows, sums, their unfolding */                           \
    static constexpr int NR = SFMM_NR_##PP, NS = SFMM_NS_##PP, NX = SFMM_NX_##PP;                              \
    template <typename T> __device__ static void fold(const T* Q, T* q) { sfmm_fold_##PP(Q, q); }              \
    template <typename T> __device__ static void derivs_fold(T x, T y, T z, T ri, T* D) { sfmm_derivs_fold_##PP1(x, y, z, ri, D); } \
    template <typename T> __device__ static void uderivs_fold(T x, T y, T z, T ri, T* D) { sfmm_uderivs_fold_##PP1(x, y, z, ri, D); } \
    template <typename T> __device__ static void m2l_fold(const T* D, const T* q, T* C) { sfmm_m2l_fold_##PP(D, q, C); } \
    __device__ static const signed char* unfold() { return &sfmm_unfold_##PP[0][0][0]; }                      \
  };
SFMM_EXP(0, 1)
SFMM_EXP(1, 2)
SFMM_EXP(2, 3)
SFMM_EXP(3, 4)
SFMM_EXP(4, 5)
#undef SFMM_EXP

// Source rows of the shared walk (k_walk_prepare), one per node.  FP32 form:
// the folded moments about the node's centre, padded to float4.  FP64 form:
// {centre (3), offset d to the centre of mass (3), folded moments about centre
// + d}: the stored centre is the centre of mass to rounding, the rest of it is
// the dipole.  With d = Q_1 / Q_0 carried beside the centre, and centre + d the
// expansion centre of targets as well as sources (r, and with it every pair
// force, antisymmetric), the dipole's 27 terms (p = 2) become six additions.
template <int P, bool F32> __host__ __device__ constexpr int row_len() {
  return F32 ? (Exp<P>::NR + 3) & ~3 : (6 + Exp<P>::NR + 1) & ~1;
}

// A node's expansion centre as centre + d: FP64 form of the shared walk (d = 0
// where there are no rows).
template <int P>
__device__ __forceinline__ void node_offset(const WalkArgs& a, int v, double (&d)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = a.row64 ? a.row64[(size_t)v * row_len<P, false>() + 3 + c] : 0.0;
}

// Sum of the translated terms of coefficient j (App. A.2): h the monomials of
// the shift, T the source coefficients.  9 steps at p = 2 and 34 at p = 4,
// where a walk over every source took 29 and 90.
template <int P, typename R>
__device__ __forceinline__ R shift_sum(int j, const R* h, const R* T, const unsigned short* s_tab) {
  R corr = R(0);
#pragma unroll 9
  for (int k = 0; k < Exp<P>::NT; ++k) {
    const int e = s_tab[k * Exp<P>::TS + j];
    if (e != 0xffff) corr = fma(h[e >> 8], T[e & 255], corr);
  }
  return corr;
}

// Reduce-scatter over the warp: on entry every lane holds v[0..32); on exit
// v[0] on lane l is the warp sum of entry l.
template <typename T>
__device__ __forceinline__ T reduce_scatter32(T (&v)[32], int lane) {
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int o = 16 >> step;
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int c = 0; c < o; ++c) {
      T send = upper ? v[c] : v[c + o];
      T keep = upper ? v[c + o] : v[c];
      v[c] = keep + __shfl_xor_sync(SFMM_FULL, send, o);
    }
  }
  return v[0];
}

// The same for N sums, 32 to a block: s[b] on lane l is the warp sum of entry
// 32 b + l (a last block of fewer entries: entry 32 b + l mod the power of two
// that holds them).
template <int N, typename T>
__device__ __forceinline__ void reduce_sums(const T (&C)[N], T* s, int lane) {
#pragma unroll
  for (int b = 0; b < (N + 31) / 32; ++b) {
    const int left = N - 32 * b;
    const int w = left >= 32 ? 32 : left > 16 ? 32 : left > 8 ? 16 : left > 4 ? 8 : left > 2 ? 4 : left;
    T v[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) v[t] = t < left ? C[32 * b + t < N ? 32 * b + t : 0] : T(0);
#pragma unroll
    for (int step = 0; step < 5; ++step) {
      const int o = 16 >> step;
      if (o < w) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int c = 0; c < o; ++c) {
          const T send = upper ? v[c] : v[c + o];
          const T keep = upper ? v[c + o] : v[c];
          v[c] = keep + __shfl_xor_sync(SFMM_FULL, send, o);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      if (o >= w) v[0] += __shfl_xor_sync(SFMM_FULL, v[0], o);
    s[b] = v[0];
  }
}

// Acceptance test of Sect. 3: accept iff (l_t + l_s) < theta d and not
// d < l_t + l_s + R_kern max(h_t, h_s).
// on: whether the lane holds a pair to test (else false).  Branch-free but for
// the float64 path: the walk is half decisions, and with early returns it took
// 14.65 ms instead of 13.79 on the 1.6e7 cloud, 0.89 instead of 0.79 at 1e5
// particles and order 4.
__device__ __forceinline__ bool decide(const float4& hiA, const float4& loA, const float4& hiB, const float4& loB,
                                       int A, int B, const WalkArgs& a, int& nfb, float& dx, float& dy, float& dz,
                                       bool on) {
  dx = df_diff(hiB.x, loB.x, hiA.x, loA.x);
  dy = df_diff(hiB.y, loB.y, hiA.y, loA.y);
  dz = df_diff(hiB.z, loB.z, hiA.z, loA.z);
  // squared form (all terms non-negative): l^2 < theta^2 d^2 and d^2 >= (l + 2h)^2;
  // the float32 error is below 1.5e-6 relative, the tie band 1e-5
  const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const float ls = hiA.w + hiB.w;
  const float hm = fmaxf(loA.w, loB.w);
  const float td2 = a.theta2_f * d2, ls2 = ls * ls;
  const float m1 = td2 - ls2, t1 = 1e-5f * (td2 + ls2);
  const float rhs = fmaf(2.0f, hm, ls);
  const float rhs2 = rhs * rhs;
  const float m2 = d2 - rhs2, t2 = 1e-5f * (d2 + rhs2);
  const bool ok = (d2 >= 1e-30f) & (d2 <= 1e30f);
  const bool no = (m1 < -t1) | (m2 < -t2);
  bool acc = (m1 > t1) & (m2 > t2);
  if (on & (!ok | !(no | acc))) {
    ++nfb;
    const double ddx = dsub(a.ncx[B], a.ncx[A]);
    const double ddy = dsub(a.ncy[B], a.ncy[A]);
    const double ddz = dsub(a.ncz[B], a.ncz[A]);
    const double dd = __dsqrt_rn(dadd(dadd(dmul(ddx, ddx), dmul(ddy, ddy)), dmul(ddz, ddz)));
    const double lsd = dadd(a.nsize[A], a.nsize[B]);
    const double hmd = fmax(a.nhmax[A], a.nhmax[B]);
    const bool mac = lsd < dmul(a.theta, dd);
    const bool soft = dd < dadd(lsd, dmul(SFMM_RKERN, hmd));
    acc = mac && !soft;
  }
  return on & acc;
}

// One node-node interaction (target centre A, source node s) accumulated
// into the lane's coefficients.  In the FP32 form r = s_B - s_A comes from
// the acceptance test (the same double-float difference).
template <int P, bool F32>
__device__ __forceinline__ void m2l_eval(int s, const float4& hiA, const float4& loA, double cAx, double cAy,
                                         double cAz, const WalkArgs& a,
                                         typename std::conditional<F32, float, double>::type* C,
                                         const float4& r) {
  using E = Exp<P>;
  if (s < 0) return;
  if constexpr (F32) {
    const float rx = r.x, ry = r.y, rz = r.z;
    const float ri = rsqrtf(fmaf(rx, rx, fmaf(ry, ry, rz * rz)));
    float D[E::NMONO1];
    E::derivs(rx * ri, ry * ri, rz * ri, ri, D);
    constexpr int NQ4 = (E::NQ + 3) / 4;
    float Q[NQ4 * 4];
    const float4* q4 = reinterpret_cast<const float4*>(a.Qf + (size_t)s * a.nqs);
#pragma unroll
    for (int t = 0; t < NQ4; ++t) {
      float4 v = __ldg(q4 + t);
      Q[4 * t] = v.x;
      Q[4 * t + 1] = v.y;
      Q[4 * t + 2] = v.z;
      Q[4 * t + 3] = v.w;
    }
    // moments are about the centre of mass: the dipole vanishes to rounding
    E::m2l_nodip(D, Q, C);
  } else {
    const double rx = a.ncx[s] - cAx, ry = a.ncy[s] - cAy, rz = a.ncz[s] - cAz;
    const double ri = rsqrt(fma(rx, rx, fma(ry, ry, rz * rz)));
    double D[E::NMONO1];
    E::derivs(rx * ri, ry * ri, rz * ri, ri, D);
    double Q[E::NQ];
    const double* q = a.Qd + (size_t)s * E::NQ;
#pragma unroll
    for (int t = 0; t < E::NQ; ++t) Q[t] = __ldg(q + t);
    E::m2l(D, Q, C);
  }
}

// One interaction on the independent components (see gen_expansion.py) added
// to the lane's sums: 41 FP64 instructions against 121 at p = 2 for the
// contraction, 35 against 52 for the derivatives.  FP32 form: r = s_B - s_A
// from the acceptance test.  FP64 form: from the rows; the derivatives take
// powers of 1/r itself while they stay in range, else r scaled by a power of
// two.
template <int P, bool F32>
__device__ __forceinline__ void m2l_fold(int s, double cAx, double cAy, double cAz, const double (&dA)[3],
                                         const WalkArgs& a, typename std::conditional<F32, float, double>::type* C,
                                         const float4& r) {
  using E = Exp<P>;
  if (s < 0) return;
  constexpr int RL = row_len<P, F32>();
  if constexpr (F32) {
    float q[RL];
    const float4* q4 = reinterpret_cast<const float4*>(a.row32) + (size_t)s * (RL / 4);
#pragma unroll
    for (int t = 0; t < RL / 4; ++t) {
      const float4 v = __ldg(q4 + t);
      q[4 * t] = v.x;
      q[4 * t + 1] = v.y;
      q[4 * t + 2] = v.z;
      q[4 * t + 3] = v.w;
    }
    const float ri = rsqrtf(fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z)));
    float D[E::NMONO1];
    E::uderivs_fold(r.x * ri, r.y * ri, r.z * ri, ri, D);
    E::m2l_fold(D, q, C);
  } else {
    double q[RL];
    const double2* q2 = reinterpret_cast<const double2*>(a.row64) + (size_t)s * (RL / 2);
#pragma unroll
    for (int t = 0; t < RL / 2; ++t) {
      const double2 v = __ldg(q2 + t);
      q[2 * t] = v.x;
      q[2 * t + 1] = v.y;
    }
    double rx = (q[0] - cAx) + (q[3] - dA[0]), ry = (q[1] - cAy) + (q[4] - dA[1]), rz = (q[2] - cAz) + (q[5] - dA[2]);
    double r2 = fma(rx, rx, fma(ry, ry, rz * rz));
    double D[E::NMONO1];
    if (r2 >= 0x1p-110 && r2 <= 0x1p110) {
      E::derivs_fold(rx, ry, rz, rsqrt_refined(r2), D);
    } else {
      // D(r) = k^(|gamma|+1) D(k r), k a power of two that brings r near 1
      const int e = ilogb(fmax(fmax(fabs(rx), fabs(ry)), fabs(rz)));
      const double k = ldexp(1.0, -e);
      rx *= k;
      ry *= k;
      rz *= k;
      r2 = fma(rx, rx, fma(ry, ry, rz * rz));
      E::derivs_fold(rx, ry, rz, rsqrt(r2), D);
      double w = k;
#pragma unroll
      for (int n = 0, t = 0; n <= P + 1; ++n) {
#pragma unroll
        for (; t < ncoef(n); ++t) D[t] *= w;
        w *= k;
      }
    }
    E::m2l_fold(D, q + 6, C);
  }
}

// Sums of one node (reduce_sums) to its coefficient vector, entry lane + 32 b
// in lev[b]: each is a sum of a few of them.  sx: scratch of 32 (NS blocks).
template <int P, typename R>
__device__ __forceinline__ void unfold_sums(const R* sums, R* lev, R* sx, const signed char* s_unf, int lane) {
  using E = Exp<P>;
  constexpr int NB = (E::NS + 31) / 32, NCS = (E::NC + 31) / 32;
#pragma unroll
  for (int b = 0; b < NB; ++b) sx[32 * b + lane] = sums[b];
  __syncwarp();
#pragma unroll
  for (int b = 0; b < NCS; ++b) {
    const int j = lane + 32 * b;
    R v = R(0);
    if (j < E::NC) {
      const signed char* u = s_unf + j * 2 * E::NX;
#pragma unroll
      for (int t = 0; t < E::NX; ++t) {
        const int f = u[2 * t + 1];
        if (f != 0) v = fma(R(f), sx[u[2 * t]], v);
      }
    }
    lev[b] = v;
  }
  __syncwarp();
}

// Sign (-1)^|gamma| of entry t of a derivative vector (entries are ordered by
// degree: ncoef(k) of them have degree <= k).
__host__ __device__ constexpr int deriv_degree(int t) {
  int k = 0;
  while (ncoef(k) <= t) ++k;
  return k;
}

// One-sided symmetric interaction (Sect. 5, after Dehnen 2002): D_gamma(r) is
// evaluated once for the pair; the target's coefficients from the source's
// moments are added to C as in m2l_eval, and the source's coefficients from
// the target's moments QA, with D_gamma(-r) = (-1)^|gamma| D_gamma(r), are
// added to the source's received sums EB (FP64 atomics).
template <int P, bool F32>
__device__ __forceinline__ void m2l_eval_sym(int s, double cAx, double cAy, double cAz, const WalkArgs& a,
                                             typename std::conditional<F32, float, double>::type* C,
                                             const float4& r,
                                             const typename std::conditional<F32, float, double>::type* QA,
                                             double* EB) {
  using E = Exp<P>;
  using R = typename std::conditional<F32, float, double>::type;
  if (s < 0) return;
  R D[E::NMONO1];
  R Q[F32 ? ((E::NQ + 3) / 4) * 4 : E::NQ];
  if constexpr (F32) {
    const float ri = rsqrtf(fmaf(r.x, r.x, fmaf(r.y, r.y, r.z * r.z)));
    E::derivs(r.x * ri, r.y * ri, r.z * ri, ri, D);
    const float4* q4 = reinterpret_cast<const float4*>(a.Qf + (size_t)s * a.nqs);
#pragma unroll
    for (int t = 0; t < (E::NQ + 3) / 4; ++t) {
      const float4 v = __ldg(q4 + t);
      Q[4 * t] = v.x;
      Q[4 * t + 1] = v.y;
      Q[4 * t + 2] = v.z;
      Q[4 * t + 3] = v.w;
    }
    E::m2l_nodip(D, Q, C);
  } else {
    const double rx = a.ncx[s] - cAx, ry = a.ncy[s] - cAy, rz = a.ncz[s] - cAz;
    const double ri = rsqrt(fma(rx, rx, fma(ry, ry, rz * rz)));
    E::derivs(rx * ri, ry * ri, rz * ri, ri, D);
    const double* q = a.Qd + (size_t)s * E::NQ;
#pragma unroll
    for (int t = 0; t < E::NQ; ++t) Q[t] = __ldg(q + t);
    E::m2l(D, Q, C);
  }
#pragma unroll
  for (int t = 0; t < E::NMONO1; ++t)
    if (deriv_degree(t) & 1) D[t] = -D[t];
  R Cp[E::NC];
#pragma unroll
  for (int t = 0; t < E::NC; ++t) Cp[t] = R(0);
  if constexpr (F32) E::m2l_nodip(D, QA, Cp);
  else E::m2l(D, QA, Cp);
#pragma unroll
  for (int t = 0; t < E::NC; ++t) atomicAdd(EB + t, (double)Cp[t]);
}

// The same with r computed here from the node records (FP32 form).
template <int P, bool F32>
__device__ __forceinline__ void m2l_eval(int s, const float4& hiA, const float4& loA, double cAx, double cAy,
                                         double cAz, const WalkArgs& a,
                                         typename std::conditional<F32, float, double>::type* C) {
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (F32 && s >= 0) {
    const float4 hB = a.geo_hi[s], lB = a.geo_lo[s];
    r.x = df_diff(hB.x, lB.x, hiA.x, loA.x);
    r.y = df_diff(hB.y, lB.y, hiA.y, loA.y);
    r.z = df_diff(hB.z, lB.z, hiA.z, loA.z);
  }
  m2l_eval<P, F32>(s, hiA, loA, cAx, cAy, cAz, a, C, r);
}

// Acceptance test without the separation output.
__device__ __forceinline__ bool decide(const float4& hiA, const float4& loA, const float4& hiB, const float4& loB,
                                       int A, int B, const WalkArgs& a, int& nfb) {
  float dx, dy, dz;
  return decide(hiA, loA, hiB, loB, A, B, a, nfb, dx, dy, dz, true);
}

}  // namespace sfmm
