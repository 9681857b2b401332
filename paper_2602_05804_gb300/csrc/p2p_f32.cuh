// Near field of the FP32 form.  Included by p2p.cu.
//
// One warp per work item (a target leaf, or a chunk of a long list).  Sources:
// the particles of the leaf's neighbour list, streamed 32 at a time over
// consecutive list entries (every lane busy), moved to the target leaf's frame
// and split once per source into those that may lie inside the kernel of some
// target (|x_j - s_L| < l_L + 2 max(h_max,L, h_j), with a small safety factor:
// the candidates, 24 % of the pairs on a Plummer sphere) and those that cannot.
// Both are staged in pairs and evaluated unsoftened, two sources per lane step
// in the packed FP32 instructions; a candidate pair inside a kernel (4 % of
// all pairs) is left out there and marked in the lane's bit masks.  Each lane
// then evaluates its own marked pairs with both kernels.  Where one lane has
// far more marks than the others, the marks of all lanes are dealt one per
// lane instead, in lane order (the k-th lane finds the owner of the k-th mark
// and the mark in its masks), and the owners add their results in order.
//
// Bound: instruction issue.  With the M4 kernels evaluated in place for every
// candidate, the whole warp ran them for almost every step, because some lane
// nearly always is inside a kernel: the candidates took 122 issue cycles per
// 32 pairs where the unsoftened sources take 23.  Measured, in place and now:
// 2.25 and 1.87 ms for the 1.38e9 pairs of a Plummer sphere of 10^6 (0.82 of the
// issue slots, 25 of 32 lanes), 7.58 and 6.43 ms at theta 0.3, 34.5 and 28.5 ms
// for a clustered cloud of 1.6e7.  Without the dealt marks (less code) leaves of
// 16 gain 1 % and leaves of 24 and more lose 2 to 5 %.
#define P2P_RES 64  // marked pairs evaluated before their owners collect
// Own marks take as many steps as the fullest lane has, dealt ones a 32nd of all
// marks at about four times a step.  Own marks where the fullest lane holds at
// most 1/12 of all (10^6 particles: 1.87 ms; 1/4 1.89, 1/8 1.88, 1/16 1.90, own
// marks always 1.89, dealt always 1.98).
#define P2P_OWN 12
// Where 2h of every target is beyond three times the leaf's size, about half of
// the candidates lie inside a kernel and all of them are evaluated with both
// kernels at once, without the unsoftened pass (uniform set of 3 10^5 with h of
// 2, 3, 4, 6, 12 mean spacings, this line, never, and always the dealt marks:
// 1.00 1.01 1.24, 2.29 2.49 3.46, 4.17 4.83 7.45, 10.3 12.7 22.0, 51.7 68.1 137
// ms; the line at 2: 1.03 for the first, at 4: 2.41 for the second.  By the
// largest 2h a leaf at a binary's surface, with one wide kernel among narrow
// ones, would take this path: leaves of 48, theta 0.4: 1.85 instead of 1.76 ms).
#define P2P_DENSE 3.0f
struct P2PWarp {
  float4 far[P2P_SB];   // pairs, negated: [q/2] {x0, x1, y0, y1}, [SB/2 + q/2] {z0, z1, m0, m1}
  float4 near[P2P_SB];  // candidates, the same
  float4 res[P2P_RES];  // softened results of a window of marked pairs; phase sums at the end of a leaf
  float4 tgt[32];       // targets {x, y, z, 1/h}
  float nh2[P2P_SB];    // candidates: (2h)^2, 1/h, index in the target leaf (-1 outside it)
  float nhinv[P2P_SB];
  short nloc[P2P_SB];
};

// Position of the r-th set bit of m (r below the number of set bits).
__device__ __forceinline__ int nth_bit(unsigned m, int r) {
  int pos = 0;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    const int c = __popc(m & ((1u << w) - 1u));
    if (r >= c) {
      r -= c;
      pos += w;
      m >>= w;
    }
  }
  return pos;
}

// Four blocks per SM: 64 registers, 55 KB of shared memory per block (three:
// 2.18 against 2.03 ms at 10^6).
__global__ void __launch_bounds__(P2P_NT, 4) k_p2p_f32(const P2PArgs a) {
  constexpr int SB = P2P_SB;
  extern __shared__ __align__(16) unsigned char p2p_smem[];
  const int lane = threadIdx.x & 31;
  P2PWarp& w = reinterpret_cast<P2PWarp*>(p2p_smem)[threadIdx.x >> 5];
  const unsigned lt = lanemask_lt();
  const int nextra = (int)a.d_split[0];
  const int nitems = nextra + (int)a.counts[1];
  unsigned long long pairs = 0;  // this lane's share of the pair evaluations
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
    const float4 hiL = a.geo_hi[L], loL = a.geo_lo[L];
    const float lL = hiL.w * 1.0001f;
    const float hL = loL.w * 1.0001f;
    // lane -> (target slot, phase); more than 32 targets: a second slot, 32 on
    const int nph = (nL <= 16) ? (32 / nL) : 1;
    const int ntl = (nL <= 32) ? nL : 32;
    const int ph = lane / ntl;
    const bool lane_on = ph < nph;
    const int t0 = lane % ntl;
    // target lane + 32 slot of the leaf to shared memory, this lane's own to registers
    auto load_targets = [&](int slot, float& x, float& y, float& z, float& h2) {
      const int t = lane + 32 * slot;
      if (t < nL) {
        const float4 p = a.prel[fL + t];
        const float4 hr = a.phh[fL + t];
        w.tgt[lane] = make_float4(p.x, p.y, p.z, hr.x);
      }
      x = y = z = h2 = 0.0f;
      if (lane_on && t0 + 32 * slot < nL) {
        const float4 p = a.prel[fL + t0 + 32 * slot];
        x = p.x;
        y = p.y;
        z = p.z;
        h2 = a.phh[fL + t0 + 32 * slot].y;
      }
    };
    float xi, yi, zi, h2i;
    load_targets(0, xi, yi, zi, h2i);
    // least (2h)^2 of the (first 32) targets, as bits
    const unsigned h2m = __reduce_min_sync(SFMM_FULL, __float_as_uint(lane_on && t0 < nL ? h2i : INFINITY));
    const bool dense = __uint_as_float(h2m) > (P2P_DENSE * P2P_DENSE) * (lL * lL);
    float ax = 0.0f, ay = 0.0f, az = 0.0f, pt = 0.0f;      // current slot
    float bx = 0.0f, by = 0.0f, bz = 0.0f, bp = 0.0f;      // the other one

    long long off = a.p2p_off[leaf];
    int cnt = a.p2p_cnt[leaf];
    if (pslot >= 0) {
      const int per = (int)*a.chunk_now;
      off += (long long)chunk * per;
      cnt = min(per, cnt - chunk * per);
    }
    int nfar = 0, nnear = 0;
    int e = 0;                 // next list entry to load
    int tot = 0, pdone = 0;    // particles of the loaded entries / staged so far
    int cum = 0, fS = 0;       // this lane's entry: first particle in the stream, first particle index
    float ox = 0.0f, oy = 0.0f, oz = 0.0f;
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
          pairs += (unsigned long long)nL * nS - (S == L ? nL : 0);
          const float4 hS = a.geo_hi[S], lS = a.geo_lo[S];
          ox = df_diff(hS.x, lS.x, hiL.x, loL.x);
          oy = df_diff(hS.y, lS.y, hiL.y, loL.y);
          oz = df_diff(hS.z, lS.z, hiL.z, loL.z);
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
        // stage one window of up to 32 particles of the stream
        const int p = pdone + lane;
        const bool valid = p < tot;
        // the entry holding position p: entries starting before the window
        // plus those starting inside it at or before p (every entry holds at
        // least one particle; the padding entries past the list hold none)
        const bool pre = cum < pdone;
        const int rs = cum - pdone;  // (no overflow: padding lanes test as neither)
        const unsigned starts = __reduce_or_sync(SFMM_FULL, (!pre && rs < 32) ? (1u << rs) : 0u);
        const int before = __popc(__ballot_sync(SFMM_FULL, pre));
        const int l = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        const int d_l = __shfl_sync(SFMM_FULL, fS - cum, l);  // particle index minus stream position
        const float ox_l = __shfl_sync(SFMM_FULL, ox, l), oy_l = __shfl_sync(SFMM_FULL, oy, l),
                    oz_l = __shfl_sync(SFMM_FULL, oz, l);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f), hr = v;  // v: position and mass negated
        int i = 0;
        if (valid) {
          i = d_l + p;
          const float4 q = a.prel[i];
          v = make_float4(-q.x - ox_l, -q.y - oy_l, -q.z - oz_l, -q.w);
          hr = a.phh[i];  // {1/h, (2h)^2, 2h rounded up}
        }
        // reach = l_L + 2 max(h_L, h_j) (l_L and h_L carry a 1.0001 margin)
        const float reach = lL + fmaxf(2.0f * hL, hr.z);
        const bool near = valid && (fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z)) < reach * reach);
        const unsigned bn = __ballot_sync(SFMM_FULL, near), bf = __ballot_sync(SFMM_FULL, valid && !near);
        if (valid) {
          const int q = near ? nnear + __popc(bn & lt) : nfar + __popc(bf & lt);
          float4* const base = near ? w.near : w.far;
          float* const xy = reinterpret_cast<float*>(base + (q >> 1)) + (q & 1);
          float* const zm = xy + 4 * (SB / 2);
          xy[0] = v.x;
          xy[2] = v.y;
          zm[0] = v.z;
          zm[2] = v.w;
          if (near) {
            w.nh2[q] = hr.y;
            w.nhinv[q] = hr.x;
            w.nloc[q] = (short)((i >= fL && i < fL + nL) ? i - fL : -1);
          }
        }
        nnear += __popc(bn);
        nfar += __popc(bf);
        pdone += min(32, tot - pdone);
      }
      const bool last = !((pdone < tot) || (e < cnt));
      // the two kinds are evaluated each when its own buffer is full: the
      // candidates' marks then come in few and large groups
      const bool do_far = nfar > SB - 32 || last, do_near = nnear > SB - 32 || last;
      if (!(do_far || do_near)) continue;
      __syncwarp();
      // odd counts: the last pair's second source repeats the first with no
      // mass (far: outside every kernel, so r > 0; candidate: its mark is dropped)
      if (lane < 2) {
        const int n = lane ? nnear : nfar;
        if (n & 1) {
          float* const xy = reinterpret_cast<float*>((lane ? w.near : w.far) + (n >> 1));
          float* const zm = xy + 4 * (SB / 2);
          xy[1] = xy[0];
          xy[3] = xy[2];
          zm[1] = zm[0];
          zm[3] = 0.0f;
          if (lane) w.nh2[n] = FLT_MIN;
        }
      }
      __syncwarp();
      const int npf = do_far ? (nfar + 1) >> 1 : 0, npn = do_near ? (nnear + 1) >> 1 : 0;
#pragma unroll 1
      for (int slot = 0; slot < (nL > 32 ? 2 : 1); ++slot) {
        if (nL > 32) {
          __syncwarp();
          load_targets(slot, xi, yi, zi, h2i);
          __syncwarp();
        }
        const float2 x2 = make_float2(xi, xi), y2 = make_float2(yi, yi), z2 = make_float2(zi, zi);
        float2 fx = make_float2(0.0f, 0.0f), fy = fx, fz = fx, fp = fx;
        if (lane_on) {
          for (int pj = ph; pj < npf; pj += nph) {
            const float4 c = w.far[pj], d = w.far[SB / 2 + pj];
            pair_far2(x2, y2, z2, make_float2(c.x, c.y), make_float2(c.z, c.w), make_float2(d.x, d.y),
                      make_float2(d.z, d.w), fx, fy, fz, fp);
          }
        }
        // pair of target t and candidate j with both kernels evaluated
        auto softened = [&](int t, int j) {
          const float4 T4 = w.tgt[t];
          const float* const xy = reinterpret_cast<const float*>(w.near + (j >> 1)) + (j & 1);
          const float* const zm = xy + 4 * (SB / 2);
          const float dx = T4.x + xy[0], dy = T4.y + xy[2], dz = T4.z + zm[0];
          const bool self = w.nloc[j] == t + 32 * slot;
          const float nm = 0.5f * zm[2];  // -m/2
          const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          const float ri = (r2 > 0.0f) ? rsqrtf(r2) : 0.0f;
          // (0 for coincident particles, no number where r^2 overflows)
          const float r = fmaxf(fminf(r2 * ri, FLT_MAX), FLT_MIN), hj = w.nhinv[j];
          float gi, pi, gj, pj;
          m4_kernel<float>(r * T4.w, T4.w, ri, gi, pi);
          m4_kernel<float>(r * hj, hj, ri, gj, pj);
          const float mg = self ? 0.0f : nm * (gi + gj), mp = self ? 0.0f : -nm * (pi + pj);
          return make_float4(mg * dx, mg * dy, mg * dz, mp);
        };
        auto take = [&](const float4& v) {
          ax += v.x;
          ay += v.y;
          az += v.z;
          pt += v.w;
        };
        if (dense && do_near && lane_on)
          for (int j = ph; j < nnear; j += nph) take(softened(t0, j));
        // candidates, up to 32 steps of every lane at a time
        for (int s0 = dense ? npn : 0; s0 < npn; s0 += 32 * nph) {
          const int end = min(npn, s0 + 32 * nph);
          unsigned m0 = 0u, m1 = 0u;  // marks of even / odd sources, the last step in bit 0
          int steps = 0;
          if (lane_on) {
            for (int pj = s0 + ph; pj < end; pj += nph) {
              const float4 c = w.near[pj], d = w.near[SB / 2 + pj];
              const float2 h2j = *reinterpret_cast<const float2*>(&w.nh2[2 * pj]);
              const float2 dx = __fadd2_rn(x2, make_float2(c.x, c.y)), dy = __fadd2_rn(y2, make_float2(c.z, c.w)),
                           dz = __fadd2_rn(z2, make_float2(d.x, d.y));
              const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
              const bool in0 = r2.x < fmaxf(h2i, h2j.x), in1 = r2.y < fmaxf(h2i, h2j.y);
              m0 = 2u * m0 + (in0 ? 1u : 0u);
              m1 = 2u * m1 + (in1 ? 1u : 0u);
              const float2 ri = make_float2(rsqrt_normal(in0 ? INFINITY : r2.x), rsqrt_normal(in1 ? INFINITY : r2.y));
              const float2 mr = __fmul2_rn(make_float2(d.z, d.w), ri);
              const float2 mr3 = __fmul2_rn(mr, __fmul2_rn(ri, ri));
              fx = __ffma2_rn(mr3, dx, fx);
              fy = __ffma2_rn(mr3, dy, fy);
              fz = __ffma2_rn(mr3, dz, fz);
              fp = __fadd2_rn(fp, mr);
              ++steps;
            }
            // the padding source of an odd count: the last pair of the last step
            if ((nnear & 1) && end == npn && (npn - 1 - s0) % nph == ph) m1 &= ~1u;
          }
          if (t0 + 32 * slot >= nL) m0 = m1 = 0u;
          const int c = __popc(m0) + __popc(m1);
          if (__reduce_max_sync(SFMM_FULL, c) * P2P_OWN <= __reduce_add_sync(SFMM_FULL, c)) {
            for (int k = 0; k < c; ++k) {
              const bool odd = m0 == 0u;
              const unsigned m = odd ? m1 : m0;
              const int bit = 31 - __clz(m);
              if (odd) m1 = m ^ (1u << bit);
              else m0 = m ^ (1u << bit);
              take(softened(t0, 2 * (s0 + ph + (steps - 1 - bit) * nph) + (odd ? 1 : 0)));
            }
            continue;
          }
          int incl = c;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(SFMM_FULL, incl, o);
            if (lane >= o) incl += y;
          }
          const int T = __shfl_sync(SFMM_FULL, incl, 31);
          const int own0 = incl - c;
          for (int r0 = 0; r0 < T; r0 += P2P_RES) {
            const int r1 = min(r0 + P2P_RES, T), mine = min(incl, r1);
            for (int kb = r0; kb < r1; kb += 32) {
              const int k = kb + lane;
              // the owner: the first lane whose inclusive count exceeds k
              int o = 0;
#pragma unroll
              for (int b = 16; b > 0; b >>= 1)
                if (__shfl_sync(SFMM_FULL, incl, o + b - 1) <= k) o += b;
              const unsigned om0 = __shfl_sync(SFMM_FULL, m0, o), om1 = __shfl_sync(SFMM_FULL, m1, o);
              const int rank = k - __shfl_sync(SFMM_FULL, own0, o);
              const int osteps = __shfl_sync(SFMM_FULL, steps, o), oph = __shfl_sync(SFMM_FULL, ph, o),
                        t = __shfl_sync(SFMM_FULL, t0, o);
              if (k < r1) {
                const int c0 = __popc(om0);
                const bool odd = rank >= c0;
                const int bit = nth_bit(odd ? om1 : om0, odd ? rank - c0 : rank);
                w.res[k - r0] = softened(t, 2 * (s0 + oph + (osteps - 1 - bit) * nph) + (odd ? 1 : 0));
              }
            }
            __syncwarp();
            for (int k = max(own0, r0); k < mine; ++k) take(w.res[k - r0]);
            __syncwarp();
          }
        }
        ax += fx.x + fx.y;
        ay += fy.x + fy.y;
        az += fz.x + fz.y;
        pt += fp.x + fp.y;
        if (nL > 32) {
          float s = ax; ax = bx; bx = s;
          s = ay; ay = by; by = s;
          s = az; az = bz; bz = s;
          s = pt; pt = bp; bp = s;
        }
      }
      __syncwarp();
      if (do_far) nfar = 0;
      if (do_near) nnear = 0;
      if (last) break;
    }

    // combine the phases of each target, add the far field, write out
    for (int slot = 0; slot < (nL > 32 ? 2 : 1); ++slot) {
      const int t = lane + 32 * slot;
      const bool on = lane_on && t0 + 32 * slot < nL;
      w.res[lane] = on ? (slot ? make_float4(bx, by, bz, bp) : make_float4(ax, ay, az, pt))
                       : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      __syncwarp();
      if (lane < ntl && t < nL) {
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int q = 0; q < nph; ++q) {
          const float4 s = w.res[q * ntl + lane];
          v[0] += s.x;
          v[1] += s.y;
          v[2] += s.z;
          v[3] += s.w;
        }
        if (pslot < 0) {
          p2p_finish<true>(a, fL + t, v);
        } else {
          float4* const pp = static_cast<float4*>(a.part) + (size_t)(pslot + chunk) * a.lmax + t;
          *pp = make_float4(v[0], v[1], v[2], v[3]);
        }
      }
      __syncwarp();
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(SFMM_FULL, pairs, o);
  if (lane == 0 && pairs) atomicAdd(a.pair_counter, pairs);
}
