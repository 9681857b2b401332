// Momentum and energy sums of a gravity call, over the particles and per
// system (the solver's diagnostics: total momentum, which Newton's third law
// and the symmetric expansions keep at rounding level, and the potential
// energy W = 1/2 sum m Phi).
#include <algorithm>

#include "sfmm_internal.cuh"

namespace sfmm {

// Momentum and energy sums over the particles: sum m a (3), sum |m a| (over
// components), sum m Phi, in FP64 in a fixed order (reruns are bitwise
// identical); the momentum components, whose terms cancel to ~1e-18 of
// sum |m a|, as Neumaier-compensated sums.  Every block takes a contiguous range of
// sorted positions (thread t: positions lo + t, lo + t + RED_NT, ...), merges
// its threads' sums in a fixed tree and writes one partial (s and c: 10
// doubles); one warp per sum merges the partials.  Accelerations and potentials are
// read in caller order through the permutation.  A separate pass costs fewer
// FP64 instructions per particle than sums formed in the near-field kernel,
// whose warps hold a leaf of ~11 particles.
#define RED_NT 256
#define RED_BLOCKS 304

// Tree over the threads' sums: one (pair of threads, sum) per thread and
// trip, so that the narrow FP64 pipe runs full warps (a thread merging all
// five sums of its pair took 12 us for a set of 1000 particles).  used: threads
// that hold a sum (the tree of a system of ten particles needs no 256 of them).
__device__ __forceinline__ void block_merge(csum (&s)[5], double (&sh)[10][RED_NT], int used = RED_NT) {
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    sh[c][threadIdx.x] = s[c].s;
    sh[5 + c][threadIdx.x] = s[c].c;
  }
  __syncthreads();
  int top = RED_NT / 2;
  while (top > 0 && top >= used) top >>= 1;
  for (int w = top; w > 0; w >>= 1) {
    for (int q = threadIdx.x; q < 5 * w; q += RED_NT) {
      const int c = q / w, t = q - c * w;
      csum a{sh[c][t], sh[5 + c][t]};
      cs_merge(a, sh[c][t + w], sh[5 + c][t + w]);
      sh[c][t] = a.s;
      sh[5 + c][t] = a.c;
    }
    __syncthreads();
  }
}

// Compensated sums of sorted positions [lo, hi) into s (this thread's share).
__device__ __forceinline__ void particle_sums(int64_t lo, int64_t hi, const double* __restrict__ pm,
                                              const int* __restrict__ perm, const double* __restrict__ acc,
                                              const double* __restrict__ pot, csum (&s)[5]) {
  for (int64_t i = lo + threadIdx.x; i < hi; i += RED_NT) {
    const double m = pm[i];
    const int o = perm[i];
    const double ax = m * acc[3 * (size_t)o], ay = m * acc[3 * (size_t)o + 1], az = m * acc[3 * (size_t)o + 2];
    cs_add(s[0], ax);
    cs_add(s[1], ay);
    cs_add(s[2], az);
    // sums of same-sign terms cannot cancel: plain additions are accurate to
    // a few eps of the result there, and cost a seventh of a compensated one
    s[3].s = __dadd_rn(s[3].s, __dadd_rn(__dadd_rn(fabs(ax), fabs(ay)), fabs(az)));
    s[4].s = __dadd_rn(s[4].s, m * pot[o]);
  }
}

__global__ void __launch_bounds__(RED_NT) k_reduce_particles(int64_t n, const double* __restrict__ pm,
                                                             const int* __restrict__ perm,
                                                             const double* __restrict__ acc,
                                                             const double* __restrict__ pot,
                                                             double* __restrict__ part) {
  __shared__ double sh[10][RED_NT];
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * per, hi = min(n, lo + per);
  csum s[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
  particle_sums(lo, hi, pm, perm, acc, pot, s);
  block_merge(s, sh);
  if (threadIdx.x < 10) part[10 * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

// One warp per sum (block c: sum c): lane l merges partials lo + l, lo + l +
// 32, ... in order, then the lanes merge in a fixed tree (lane 0 holds it).
__device__ __forceinline__ csum merge_parts(int lo, int hi, const double* __restrict__ part) {
  const int c = blockIdx.x, lane = threadIdx.x;
  csum s{0.0, 0.0};
  for (int q = lo + lane; q < hi; q += 32) cs_merge(s, part[10 * q + c], part[10 * q + 5 + c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double bs = __shfl_down_sync(SFMM_FULL, s.s, o), bc = __shfl_down_sync(SFMM_FULL, s.c, o);
    if (lane < o) cs_merge(s, bs, bc);
  }
  return s;
}
__global__ void k_reduce_final(int nparts, const double* __restrict__ part, double* __restrict__ out) {
  const csum s = merge_parts(0, nparts, part);
  if (threadIdx.x == 0) out[blockIdx.x] = __dadd_rn(s.s, s.c);
}
// Many partials: RED_GROUP of them to one first (60,000 systems left five warps
// 1900 FP64 additions one after another).
#define RED_GROUP 1024
__global__ void k_reduce_group(int nparts, const double* __restrict__ part, double* __restrict__ out) {
  const int lo = blockIdx.y * RED_GROUP;
  const csum s = merge_parts(lo, min(nparts, lo + RED_GROUP), part);
  if (threadIdx.x == 0) {
    out[10 * (size_t)blockIdx.y + blockIdx.x] = s.s;
    out[10 * (size_t)blockIdx.y + 5 + blockIdx.x] = s.c;
  }
}

// Batches: a block per slice (batch_slice) of a system's sorted positions
// (systems are contiguous in the sorted order).
__global__ void __launch_bounds__(RED_NT) k_reduce_slices(int nsys, const int* __restrict__ sys_off, int shift,
                                                          const double* __restrict__ pm,
                                                          const int* __restrict__ perm,
                                                          const double* __restrict__ acc,
                                                          const double* __restrict__ pot, double* __restrict__ part) {
  __shared__ double sh[10][RED_NT];
  const BatchSlice b = batch_slice(sys_off, nsys, shift, blockIdx.x);
  csum s[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
  particle_sums(b.lo, b.hi, pm, perm, acc, pot, s);
  block_merge(s, sh, (int)min((int64_t)RED_NT, b.hi - b.lo));
  if (threadIdx.x < 10) part[10 * (size_t)blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

// One thread per (system, sum): the slices merged in order, as the system's
// partial (for the sums over all systems) and as its value.
__global__ void k_reduce_sys(int nsys, const int* __restrict__ sys_off, int shift, const double* __restrict__ part,
                             double* __restrict__ sys_part, double* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 5 * nsys) return;
  const int sys = t / 5, c = t - 5 * sys;
  csum s{0.0, 0.0};
  for (int k = slice_base(sys_off, shift, sys); k < slice_base(sys_off, shift, sys + 1); ++k) {
    const double* q = part + 10 * (size_t)k;
    cs_merge(s, q[c], q[5 + c]);
  }
  sys_part[10 * (size_t)sys + c] = s.s;
  sys_part[10 * (size_t)sys + 5 + c] = s.c;
  const double v = __dadd_rn(s.s, s.c);
  out[t] = (c == 4) ? 0.5 * v : v;
}

// Sums over all particles (device pointer in *out_dev) and, for batches, per
// system, in slices of at most 8192 particles (of 1/64 of the largest system,
// where that is more: one thread per system and sum adds its slices).  One block
// per system took 1.45 ms for 256 systems of up to 10^5 particles, beside a
// second pass for the totals; as many slices for every system as the largest
// needs took 70 ms for one of 5 10^5 among 60,000 of ten (0.4 ms now).
int run_reduce(sfmm_ctx* c, double** out_dev) {
  int rc;
  const bool batch = c->nsys > 1;
  const int shift = slice_shift(c, 13, 64);
  const size_t slices = batch ? (size_t)(c->n >> shift) + c->nsys : 0;
  const int blocks = (int)std::min<int64_t>(RED_BLOCKS, (c->n + RED_NT - 1) / RED_NT);
  const int groups = c->nsys > RED_GROUP ? (c->nsys + RED_GROUP - 1) / RED_GROUP : 0;
  const size_t nparts = batch ? slices + c->nsys + groups : (size_t)blocks;
  if ((rc = c->red_part.ensure(sizeof(double) * 10 * (nparts + 1)))) return rc;
  double* part = c->red_part.as<double>();
  double* out = part + 10 * nparts;
  if (batch) {
    if ((rc = c->sys_sums.ensure(sizeof(double) * 5 * (size_t)c->nsys))) return rc;
    double* sys_part = part + 10 * slices;
    const int* off = c->sys_off.as<int>();
    k_reduce_slices<<<(unsigned)slices, RED_NT, 0, c->stream>>>(c->nsys, off, shift, c->pm.as<double>(),
                                                                c->perm.as<int>(), c->red_acc, c->red_pot, part);
    ++c->nlaunch;
    k_reduce_sys<<<(5 * c->nsys + 127) / 128, 128, 0, c->stream>>>(c->nsys, off, shift, part, sys_part,
                                                                   c->sys_sums.as<double>());
    ++c->nlaunch;
    if (groups) {
      double* grouped = sys_part + 10 * (size_t)c->nsys;
      k_reduce_group<<<dim3(5, groups), 32, 0, c->stream>>>(c->nsys, sys_part, grouped);
      ++c->nlaunch;
      k_reduce_final<<<5, 32, 0, c->stream>>>(groups, grouped, out);
    } else {
      k_reduce_final<<<5, 32, 0, c->stream>>>(c->nsys, sys_part, out);
    }
  } else {
    k_reduce_particles<<<blocks, RED_NT, 0, c->stream>>>(c->n, c->pm.as<double>(), c->perm.as<int>(), c->red_acc,
                                                        c->red_pot, part);
    ++c->nlaunch;
    k_reduce_final<<<5, 32, 0, c->stream>>>(blocks, part, out);
  }
  ++c->nlaunch;
  *out_dev = out;
  SFMM_CUDA_TRY(cudaGetLastError());
  return SFMM_OK;
}

}  // namespace sfmm
