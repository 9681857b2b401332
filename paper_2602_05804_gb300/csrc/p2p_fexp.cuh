// Near field of the FP64 form on the FP32 pipe: unsoftened pairs as
// floating-point expansions (fexp.cuh), pairs inside a softening kernel in
// FP64.  Included by p2p.cu.
//
// Why: the FP64 pipe bounds the plain FP64 near field (87 % busy, 1.4e9 pairs
// at 1e6 particles).  Here the 95 % of pairs outside every kernel run on the
// FP32 pipe, and the FP64 pipe only evaluates the softened pairs, 32 at a time
// with every lane busy, while other warps of the SM quarter run expansions.
// Measured, before and now: 66.6 and 17.5 ms for the 1.38e9 pairs of a Plummer
// sphere of 10^6 (FMA pipe 64 % busy, FP64 40 %; 16 warps per SM by shared
// memory and 128 registers, of which 140 bytes are spilled: 19.0 ms with twenty,
// 18.7 with twelve), 5.87 and 1.75 ms
// for 10^5 with leaves of 8, 0.77 and 0.23 ms for 10^4 (the last two with the
// finer list chunks).
//
// Per particle: coordinates scaled by a power of two to |x| < 1 and split into
// three floats (exactly for |x| >= 2^-18, else to 2^-71), masses scaled by a
// power of two to below the total and split likewise, (2h)^2 rounded up.
// A leaf whose smallest 2h is below 2^-18 of that scale, a source mass below
// 2^-80 of the total, or a scale outside 2^+-300 go to k_p2p_fp64: its
// FP64 arithmetic has no such limits.

// Powers of two of a system: positions by 2^-kx, masses by 2^-km.
struct SysScale {
  int kx, km;
  bool ok;
};

struct FexpArgs {
  const int* psys;      // system of a sorted particle (NULL: one system)
  const int* sys_root;
  const double* nsize;
  const double* nmass;
  float4* rec0;         // {x, y, z (grid 2^-22), m (24 bits)}
  float4* rec1;         // {x, y, z (grid 2^-45), m (next 24)}
  float4* rec2;         // {x, y, z (rest), m (rest)}
  float2* rech;         // {(2h)^2 rounded up, 2h rounded down}, scaled
  double2* hinv;        // {1 / h, 1 / h^3}
  int* fb;              // [0] work items left to k_p2p_fp64, [1] its item counter, [4 ..] the items
};

__device__ __forceinline__ SysScale sys_scale(const P2PArgs& a, const FexpArgs& f, int sorted) {
  const int root = f.sys_root[f.psys ? f.psys[sorted] : 0];
  const double b = (fmax(fmax(fabs(a.ncx[root]), fabs(a.ncy[root])), fabs(a.ncz[root])) + f.nsize[root]) * 1.000000001;
  SysScale s;
  s.kx = b > 0.0 ? ilogb(b) + 1 : 0;
  s.km = ilogb(f.nmass[root]) + 1;
  s.ok = abs(s.kx) < 300 && abs(s.km) < 300;
  return s;
}

__global__ void __launch_bounds__(256) k_fexp_records(const P2PArgs a, const FexpArgs f, int n) {
  if (blockIdx.x == 0 && threadIdx.x < 4) f.fb[threadIdx.x] = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double hi = 1.0 / a.ph[i];
    f.hinv[i] = make_double2(hi, hi * hi * hi);
    const SysScale s = sys_scale(a, f, i);
    if (!s.ok) continue;  // (not read: every leaf of the system goes to k_p2p_fp64)
    const double sx = __hiloint2double((1023 - s.kx) << 20, 0), sm = __hiloint2double((1023 - s.km) << 20, 0);
    float4 r0, r1, r2;
    fexp::split_grid(a.px[i] * sx, r0.x, r1.x, r2.x);
    fexp::split_grid(a.py[i] * sx, r0.y, r1.y, r2.y);
    fexp::split_grid(a.pz[i] * sx, r0.z, r1.z, r2.z);
    fexp::split_plain(a.pm[i] * sm, r0.w, r1.w, r2.w);
    const double h2 = 2.0 * a.ph[i] * sx;
    f.rec0[i] = r0;
    f.rec1[i] = r1;
    f.rec2[i] = r2;
    f.rech[i] = make_float2(__double2float_ru(h2 * h2) * (1.0f + 0x1p-19f), __double2float_rd(h2));
  }
}

// M4 kernel of one particle in FP64: g and phi of a unit mass at r = q h,
// added to g, phi.  The piece is chosen by its coefficients (an FP64
// instruction takes the time of many selects) and by integer comparison.
__device__ __forceinline__ void m4_add(double r, double ri, double ri3, double2 hinv, double& g, double& phi) {
  const double q = r * hinv.x;
  const int qh = __double2hiint(q);
  const bool in1 = qh < 0x3ff00000, out = qh >= 0x40000000;  // q < 1, q >= 2
  const double g0 = in1 ? 4.0 / 3.0 : 8.0 / 3.0, g1 = in1 ? 0.0 : -3.0, g2 = in1 ? -1.2 : 1.2,
               g3 = in1 ? 0.5 : -1.0 / 6.0;
  const double p0 = in1 ? -1.4 : -1.6, p2 = in1 ? 2.0 / 3.0 : 4.0 / 3.0, p3 = in1 ? 0.0 : -1.0,
               p4 = in1 ? -0.3 : 0.3, p5 = in1 ? 0.1 : -1.0 / 30.0;
  // outside 2h the polynomials take no part: 1/r^3 and -1/r; inside h 1/r^3
  // takes none (selected, not multiplied by zero: it overflows where r < 2e-103)
  const double hv = out ? 0.0 : hinv.x, hv3 = out ? 0.0 : hinv.y, qq = out ? 0.0 : q;
  const double cg = out ? 1.0 : -1.0 / 15.0, cp = in1 ? 0.0 : (out ? -1.0 : 1.0 / 15.0);
  const double r3 = in1 ? 0.0 : ri3;
  const double gp = ::fma(qq, ::fma(qq, ::fma(qq, g3, g2), g1), g0);
  const double pp = ::fma(qq * qq, ::fma(qq, ::fma(qq, ::fma(qq, p5, p4), p3), p2), p0);
  g = ::fma(hv3, gp, ::fma(cg, r3, g));
  phi = ::fma(hv, pp, ::fma(cp, ri, phi));
}

#define FX_WARPS 4
#define FX_NT (FX_WARPS * 32)
#define FX_SB 128  // staged sources per flush
#define FX_SQ 96   // queued softened pairs: below 32 carried over and at most 64 of one step

__device__ __forceinline__ float bias_of(float bound) {
  return __int_as_float(((__float_as_int(bound * 1.001f) & 0x7f800000) + (2 << 23)) | 0x400000);
}

// One warp per work item (a leaf, or a chunk of a long list).  Sources are
// staged up to 128 at a time; the (target, source pair) combinations of a
// flush are cut into 32 equal runs, one per lane, target-major, so that every
// lane is busy for any leaf size; a run spans at most two targets.
__global__ void __launch_bounds__(FX_NT, 4) k_p2p_fexp(const P2PArgs a, const FexpArgs f) {
  using namespace fexp;
  // sources of a flush in pairs, negated coordinates: 12 float2 per pair
  __shared__ __align__(16) float2 s_src[FX_WARPS][(FX_SB / 2 + 1) * 12];
  __shared__ float s_h2[FX_WARPS][FX_SB + 2];
  __shared__ int s_idx[FX_WARPS][FX_SB + 2];
  __shared__ double s_acc[FX_WARPS][64][4];
  __shared__ __align__(16) float s_part[FX_WARPS][12][32];  // run sums; softened results (32 x 4 doubles)
  __shared__ int s_qj[FX_WARPS][FX_SQ];  // queued softened pairs: source particle, target in the leaf
  __shared__ unsigned char s_qt[FX_WARPS][FX_SQ];
  __shared__ unsigned s_gm[FX_WARPS][32];  // a batch's targets: lanes holding their results, target in the leaf
  __shared__ unsigned char s_gt[FX_WARPS][32];
  __shared__ float2 s_bias[FX_WARPS][32];  // per target of a group: level-0 bias of force and potential

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = lanemask_lt();
  float2* const src = s_src[warp];
  const int nextra = (int)a.d_split[0];
  const int nitems = nextra + (int)a.counts[1];
  unsigned long long pairs = 0;
  while (true) {
    int item = 0;
    if (lane == 0) item = atomicAdd(a.leaf_counter, 1);
    item = __shfl_sync(SFMM_FULL, item, 0);
    if (item >= nitems) break;
    int leaf, chunk = 0;
    if (item < nextra) {
      const int2 x = a.extra[item];
      leaf = x.x;
      chunk = x.y;
    } else {
      leaf = item - nextra;
    }
    const int pslot = a.split ? a.split[leaf] : -1;
    const int L = a.leaf_node[leaf];
    const int fL = a.nfirst[L], nL = a.ncount[L];
    const SysScale sc = sys_scale(a, f, fL);
    float hmin = INFINITY, hmax = 0.0f;  // the targets' 2h
    if (sc.ok)
      for (int t = lane; t < nL; t += 32) {
        const float h2 = f.rech[fL + t].y;
        hmin = fminf(hmin, h2);
        hmax = fmaxf(hmax, h2);
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      hmin = fminf(hmin, __shfl_xor_sync(SFMM_FULL, hmin, o));
      hmax = fmaxf(hmax, __shfl_xor_sync(SFMM_FULL, hmax, o));
    }
    if (!sc.ok || !(hmin >= 0x1p-18f)) {
      if (lane == 0) f.fb[4 + atomicAdd(&f.fb[0], 1)] = item;
      continue;
    }
    // the leaf's centre and size in scaled floats
    const double sx = __hiloint2double((1023 - sc.kx) << 20, 0);
    const float cx = (float)(a.ncx[L] * sx), cy = (float)(a.ncy[L] * sx), cz = (float)(a.ncz[L] * sx);
    const float lL = (float)(f.nsize[L] * sx) * 1.0001f + 0x1p-21f;  // (the rounded centre is within 2^-23)
    for (int t = lane; t < nL * 4; t += 32) (&s_acc[warp][0][0])[t] = 0.0;
    __syncwarp();

    long long off = a.p2p_off[leaf];
    int cnt = a.p2p_cnt[leaf];
    if (pslot >= 0) {
      const int per = (int)*a.chunk_now;
      off += (long long)chunk * per;
      cnt = min(per, cnt - chunk * per);
    }
    int ns = 0;                // staged sources
    int e = 0;                 // next list entry to load
    int tot = 0, pdone = 0;    // particles of the loaded entries / staged so far
    int cum = 0, fS = 0;       // this lane's entry: first particle in the stream, first particle index
    int qn = 0;                // queued softened pairs
    bool tiny = false;
    unsigned long long mypairs = 0;
    // bounds of the staged sources' unsoftened forces and potentials on any
    // target: above, and below from the sources outside every kernel
    float bf = 0.0f, bp = 0.0f, low = 0.0f;

    // queued softened pairs, the last cnt entries, one per lane
    auto soft_batch = [&](int base, int nb) {
      double4_16a* const res = reinterpret_cast<double4_16a*>(&s_part[warp][0][0]);
      const int t = lane < nb ? (int)s_qt[warp][base + lane] : 64 + lane;
      double4_16a v = make_double4_16a(0.0, 0.0, 0.0, 0.0);
      if (lane < nb) {
        const int i = fL + t, j = s_qj[warp][base + lane];
        const double dx = a.px[i] - a.px[j], dy = a.py[i] - a.py[j], dz = a.pz[i] - a.pz[j];
        const double r2 = ::fma(dx, dx, ::fma(dy, dy, dz * dz));
        // (coincident particles: no force, the kernel's central potential)
        const double ri = (r2 >= 0x1p-120 && r2 <= 0x1p120) ? rsqrt_refined(r2) : (r2 > 0.0 ? rsqrt(r2) : 0.0);
        const double r = r2 * ri, ri3 = ri * ri * ri;
        double g = 0.0, phi = 0.0;
        m4_add(r, ri, ri3, f.hinv[i], g, phi);
        m4_add(r, ri, ri3, f.hinv[j], g, phi);
        const double mj = a.pm[j], mh = __hiloint2double(__double2hiint(mj) - 0x100000, __double2loint(mj));
        const double mg = -mh * g;
        v = make_double4_16a(mg * dx, mg * dy, mg * dz, mh * phi);
      }
      // each target's results in lane order, one (target, component) per lane:
      // 8 targets at a time
      const unsigned same = __match_any_sync(SFMM_FULL, t);
      res[lane] = v;
      const unsigned lead = __ballot_sync(SFMM_FULL, lane < nb && lane == __ffs(same) - 1);
      if (lead >> lane & 1u) {
        const int g = __popc(lead & lt);
        s_gm[warp][g] = same;
        s_gt[warp][g] = (unsigned char)t;
      }
      __syncwarp();
      const double* const rd = reinterpret_cast<const double*>(res) + (lane & 3);
      for (int g = lane >> 2; g < __popc(lead); g += 8) {
        unsigned m = s_gm[warp][g];
        double w = rd[4 * (__ffs(m) - 1)];
        m &= m - 1;
        while (m) {
          w += rd[4 * (__ffs(m) - 1)];
          m &= m - 1;
        }
        s_acc[warp][s_gt[warp][g]][lane & 3] += w;
      }
      __syncwarp();
    };

    while (true) {
      const bool stream_left = (pdone < tot) || (e < cnt);
      if (stream_left && pdone == tot) {
        // next 32 list entries, one per lane: prefix sum of their particle counts
        const int k = e + lane;
        int nS = 0;
        if (k < cnt) {
          const int S = a.arena[off + k];
          fS = a.nfirst[S];
          nS = a.ncount[S];
          mypairs += (unsigned long long)nL * nS - (S == L ? nL : 0);
        }
        int incl = nS;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(SFMM_FULL, incl, o);
          if (lane >= o) incl += y;
        }
        cum = (nS > 0) ? incl - nS : INT_MAX;  // padding entries start nowhere
        tot = __shfl_sync(SFMM_FULL, incl, 31);
        pdone = 0;
        e += 32;
      }
      if (stream_left) {
        // stage one window of up to 32 particles of the stream (as k_p2p_f32)
        const int p = pdone + lane;
        const bool valid = p < tot;
        const bool pre = cum < pdone;
        const int rs = cum - pdone;
        const unsigned starts = __reduce_or_sync(SFMM_FULL, (!pre && rs < 32) ? (1u << rs) : 0u);
        const int before = __popc(__ballot_sync(SFMM_FULL, pre));
        const int l = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        const int d_l = __shfl_sync(SFMM_FULL, fS - cum, l);
        if (valid) {
          const int i = d_l + p, q = ns + lane;
          const float4 r0 = f.rec0[i], r1 = f.rec1[i], r2 = f.rec2[i];
          const float2 hh = f.rech[i];
          float* const d = reinterpret_cast<float*>(src + 12 * (q >> 1)) + (q & 1);
          d[0] = -r0.x; d[2] = -r1.x; d[4] = -r2.x;
          d[6] = -r0.y; d[8] = -r1.y; d[10] = -r2.y;
          d[12] = -r0.z; d[14] = -r1.z; d[16] = -r2.z;
          d[18] = r0.w; d[20] = r1.w; d[22] = r2.w;
          s_h2[warp][q] = hh.x;
          s_idx[warp][q] = i;
          tiny |= r0.w < 0x1p-80f;
          // no unsoftened pair of this source is closer than dmin
          const float ux = r0.x - cx, uy = r0.y - cy, uz = r0.z - cz;
          const float dist = sqrtf(ux * ux + uy * uy + uz * uz);
          const float dmin = dist * 0.9999f - 0x1p-21f - lL;
          const float di = 1.0f / fmaxf(dmin, fmaxf(hh.y, hmin) * 0.999f);
          const float mi = r0.w * di;
          bp += mi;
          bf += mi * di;
          const float dmax = dist + lL;
          if (dmin > 1.0001f * fmaxf(hh.y, hmax)) low += r0.w / (dmax * dmax);
        }
        const int add_n = min(32, tot - pdone);
        ns += add_n;
        pdone += add_n;
      }
      const bool last = !((pdone < tot) || (e < cnt));
      if (!(ns > FX_SB - 32 || last)) continue;
      if (__any_sync(SFMM_FULL, tiny)) break;
      if (lane == 0 && (ns & 1)) {
        // odd count: the last pair's second source has no mass and never counts
        float* const d = reinterpret_cast<float*>(src + 12 * (ns >> 1)) + 1;
#pragma unroll
        for (int c = 0; c < 12; ++c) d[2 * c] = 0.0f;
        s_h2[warp][ns] = INFINITY;
        s_idx[warp][ns] = -1;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        bf += __shfl_xor_sync(SFMM_FULL, bf, o);
        bp += __shfl_xor_sync(SFMM_FULL, bp, o);
        low += __shfl_xor_sync(SFMM_FULL, low, o);
      }
      const bool loose = !(bf <= 32.0f * low);
      const float2 bound = make_float2(bf, bp);
      bf = bp = low = 0.0f;
      __syncwarp();
      const int np = (ns + 1) >> 1;
      for (int g0 = 0; g0 < nL && ns > 0; g0 += 32) {
        const int ng = min(32, nL - g0);
        const int P = ng * np;
        const int b0 = (lane * P) >> 5, b1 = ((lane + 1) * P) >> 5;
        const int trips = (P + 31) >> 5;
        // Biases: 1.5 x the power of two 2 to 4 times a bound of the target's
        // sum of absolute terms.  The last level resolves 2^-58 of the bias,
        // so the bound has to be near the sum: the one over all targets where
        // the sources outside every kernel alone reach 1/32 of it, else the
        // target's own sum in FP32 (7 % of a flush; small h, a heavy particle
        // among light ones)
        if (!loose) {
          s_bias[warp][lane] = make_float2(bias_of(bound.x), bias_of(bound.y));
        } else {
          for (int t = 0; t < ng; ++t) {
            const int i = fL + g0 + t;
            const float4 r0 = f.rec0[i], r1 = f.rec1[i];
            const float h2t = f.rech[i].x;
            float af = 0.0f, ap = 0.0f;
            for (int q = lane; q < ns; q += 32) {
              const float* const d = reinterpret_cast<const float*>(src + 12 * (q >> 1)) + (q & 1);
              const float ux = (r0.x + d[0]) + (r1.x + d[2]), uy = (r0.y + d[6]) + (r1.y + d[8]),
                          uz = (r0.z + d[12]) + (r1.z + d[14]);
              const float rr = ux * ux + uy * uy + uz * uz;
              if (rr >= 0.999f * fmaxf(h2t, s_h2[warp][q])) {
                const float y = rsqrtf(rr);
                ap += d[18] * y;
                af += d[18] * y * y;
              }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
              af += __shfl_xor_sync(SFMM_FULL, af, o);
              ap += __shfl_xor_sync(SFMM_FULL, ap, o);
            }
            if (lane == t) s_bias[warp][t] = make_float2(bias_of(af), bias_of(ap));
          }
        }
        __syncwarp();
        PairSums S;
        float first[12];   // the run's first target's sums, once it moved on
        float sf = 0.0f, sp = 0.0f;
        auto clear = [&]() {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            S.a0[c] = dup(c < 3 ? sf : sp);
            S.a1[c] = dup((c < 3 ? sf : sp) * 0x1p-15f);
            S.a2[c] = dup(0.0f);
          }
        };
#pragma unroll
        for (int c = 0; c < 12; ++c) first[c] = 0.0f;
        // both halves' sums without the bias (exact: multiples of the bias's last place)
        auto take = [&](float (&v)[12]) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float b = c < 3 ? sf : sp, b1_ = b * 0x1p-15f;
            v[3 * c] = (S.a0[c].x - b) + (S.a0[c].y - b);
            v[3 * c + 1] = (S.a1[c].x - b1_) + (S.a1[c].y - b1_);
            v[3 * c + 2] = S.a2[c].x + S.a2[c].y;
          }
        };
        bool moved = false;
        int t = 0, j = 0;
        if (b0 < b1) {
          t = b0 / np;
          j = b0 - t * np;
        }
        float2 x[9];
        float h2i = 0.0f;
        auto target = [&](int tt) {
          const int i = fL + g0 + tt;
          const float4 r0 = f.rec0[i], r1 = f.rec1[i], r2 = f.rec2[i];
          x[0] = dup(r0.x); x[1] = dup(r1.x); x[2] = dup(r2.x);
          x[3] = dup(r0.y); x[4] = dup(r1.y); x[5] = dup(r2.y);
          x[6] = dup(r0.z); x[7] = dup(r1.z); x[8] = dup(r2.z);
          h2i = f.rech[i].x;
          sf = s_bias[warp][tt].x;
          sp = s_bias[warp][tt].y;
          clear();
        };
        target(t);
        for (int k = 0; k < trips; ++k) {
          bool inx = false, iny = false;
          if (b0 + k < b1) {
            if (j == np) {
              take(first);
              moved = true;
              ++t;
              j = 0;
              target(t);
            }
            float2 q[12];
            const float4* const qp = reinterpret_cast<const float4*>(src + 12 * j);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              const float4 w = qp[c];
              q[2 * c] = make_float2(w.x, w.y);
              q[2 * c + 1] = make_float2(w.z, w.w);
            }
            float2 D0[3], D1[3], D2[3];
            const float2 rr = separation(x, q, D0, D1, D2);
            // inside a kernel (or on its edge): FP64, below
            inx = rr.x < fmaxf(h2i, s_h2[warp][2 * j]);
            iny = rr.y < fmaxf(h2i, s_h2[warp][2 * j + 1]);
            unsoftened(D0, D1, D2, q[9], q[10], q[11], inx, iny, S);
            if (inx || iny) {
              const int i = fL + g0 + t;
              const int jx = s_idx[warp][2 * j], jy = s_idx[warp][2 * j + 1];
              inx = inx && jx != i;
              iny = iny && jy != i && jy >= 0;
            }
          }
          const unsigned bx = __ballot_sync(SFMM_FULL, inx), by = __ballot_sync(SFMM_FULL, iny);
          if (bx | by) {
            if (inx) {
              const int w = qn + __popc(bx & lt);
              s_qj[warp][w] = s_idx[warp][2 * j];
              s_qt[warp][w] = (unsigned char)(g0 + t);
            }
            if (iny) {
              const int w = qn + __popc(bx) + __popc(by & lt);
              s_qj[warp][w] = s_idx[warp][2 * j + 1];
              s_qt[warp][w] = (unsigned char)(g0 + t);
            }
            qn += __popc(bx) + __popc(by);
            __syncwarp();
            while (qn >= 32) {
              soft_batch(qn - 32, 32);
              qn -= 32;
            }
          }
          ++j;
        }
        // lanes covering target t: from the one holding unit t np (which may
        // have started in target t - 1: then its second part) to the one
        // holding unit (t + 1) np - 1; level sums are exact, then to double
        float now[12];
        take(now);
        int l0 = 0, l1 = -1;
        bool second = false;
        if (lane < ng) {
          l0 = (32 * lane * np + 31) / P;
          l1 = (32 * ((lane + 1) * np - 1) + 31) / P;
          second = ((l0 * P) >> 5) < lane * np;
        }
        float sum[12];
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 12; ++c) s_part[warp][c][lane] = moved ? now[c] : 0.0f;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 12; ++c) sum[c] = second ? s_part[warp][c][l0] : 0.0f;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 12; ++c) s_part[warp][c][lane] = moved ? first[c] : now[c];
        __syncwarp();
        for (int l = second ? l0 + 1 : l0; l <= l1; ++l) {
#pragma unroll
          for (int c = 0; c < 12; ++c) sum[c] += s_part[warp][c][l];
        }
        if (lane < ng) {
          const double fs = __hiloint2double((1023 + sc.km - 2 * sc.kx) << 20, 0),
                       ps = __hiloint2double((1023 + sc.km - sc.kx) << 20, 0);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const double v = ((double)sum[3 * c + 2] + (double)sum[3 * c + 1]) + (double)sum[3 * c];
            s_acc[warp][g0 + lane][c] = ::fma(v, c < 3 ? -fs : -ps, s_acc[warp][g0 + lane][c]);
          }
        }
        __syncwarp();
      }
      ns = 0;
      if (last) break;
    }
    if (qn > 0) soft_batch(0, qn);
    if (__any_sync(SFMM_FULL, tiny)) {
      if (lane == 0) f.fb[4 + atomicAdd(&f.fb[0], 1)] = item;
      __syncwarp();
      continue;
    }
    pairs += mypairs;
    for (int t = lane; t < nL; t += 32) {
      const double v[4] = {s_acc[warp][t][0], s_acc[warp][t][1], s_acc[warp][t][2], s_acc[warp][t][3]};
      if (pslot < 0) {
        p2p_finish<false>(a, fL + t, v);
      } else {
        double* pp = static_cast<double*>(a.part) + ((size_t)(pslot + chunk) * a.lmax + t) * 4;
#pragma unroll
        for (int c = 0; c < 4; ++c) pp[c] = v[c];
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(SFMM_FULL, pairs, o);
  if (lane == 0 && pairs) atomicAdd(a.pair_counter, pairs);
}
