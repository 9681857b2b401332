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
// five sums of its pair took 12 us for a set of 1000 particles).
__device__ __forceinline__ void block_merge(csum (&s)[5], double (&sh)[10][RED_NT]) {
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    sh[c][threadIdx.x] = s[c].s;
    sh[5 + c][threadIdx.x] = s[c].c;
  }
  __syncthreads();
  for (int w = RED_NT / 2; w > 0; w >>= 1) {
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

// One warp per sum (block c: sum c), on five SMs: lane l merges partials l,
// l + 32, ... in order, then the lanes merge in a fixed tree.
__global__ void k_reduce_final(int nparts, const double* __restrict__ part, double* __restrict__ out) {
  const int c = blockIdx.x, lane = threadIdx.x;
  csum s{0.0, 0.0};
  for (int q = lane; q < nparts; q += 32) cs_merge(s, part[10 * q + c], part[10 * q + 5 + c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double bs = __shfl_down_sync(SFMM_FULL, s.s, o), bc = __shfl_down_sync(SFMM_FULL, s.c, o);
    if (lane < o) cs_merge(s, bs, bc);
  }
  if (lane == 0) out[c] = __dadd_rn(s.s, s.c);
}

// Batches: block (k, system) takes the k-th of gridDim.x equal slices of the
// system's sorted positions (systems are contiguous in the sorted order).
__global__ void __launch_bounds__(RED_NT) k_reduce_slices(const int* __restrict__ sys_off,
                                                          const double* __restrict__ pm,
                                                          const int* __restrict__ perm,
                                                          const double* __restrict__ acc,
                                                          const double* __restrict__ pot, double* __restrict__ part) {
  __shared__ double sh[10][RED_NT];
  const int sys = blockIdx.y;
  const int64_t b = sys_off[sys], cnt = sys_off[sys + 1] - b;
  csum s[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
  particle_sums(b + cnt * blockIdx.x / gridDim.x, b + cnt * (blockIdx.x + 1) / gridDim.x, pm, perm, acc, pot, s);
  block_merge(s, sh);
  if (threadIdx.x < 10) part[10 * ((size_t)sys * gridDim.x + blockIdx.x) + threadIdx.x] = sh[threadIdx.x][0];
}

// One thread per (system, sum): the slices merged in order, as the system's
// partial (for the sums over all systems) and as its value.
__global__ void k_reduce_sys(int nsys, int slices, const double* __restrict__ part, double* __restrict__ sys_part,
                             double* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 5 * nsys) return;
  const int sys = t / 5, c = t - 5 * sys;
  csum s{0.0, 0.0};
  for (int k = 0; k < slices; ++k) {
    const double* q = part + 10 * ((size_t)sys * slices + k);
    cs_merge(s, q[c], q[5 + c]);
  }
  sys_part[10 * (size_t)sys + c] = s.s;
  sys_part[10 * (size_t)sys + 5 + c] = s.c;
  const double v = __dadd_rn(s.s, s.c);
  out[t] = (c == 4) ? 0.5 * v : v;
}

// Sums over all particles (device pointer in *out_dev) and, for batches, per
// system.  Slices of at most 8192 particles: one block per system took 1.45 ms
// for 256 systems of up to 10^5 particles, beside a second pass for the totals.
int run_reduce(sfmm_ctx* c, double** out_dev) {
  int rc;
  const bool batch = c->nsys > 1;
  int64_t largest = 0;
  for (int k = 0; k < c->nsys; ++k) largest = std::max(largest, c->h_sys_off[k + 1] - c->h_sys_off[k]);
  const int slices = (int)std::min<int64_t>(64, (largest + 8191) / 8192);
  const int blocks = (int)std::min<int64_t>(RED_BLOCKS, (c->n + RED_NT - 1) / RED_NT);
  const size_t nparts = batch ? (size_t)c->nsys * (slices + 1) : (size_t)blocks;
  if ((rc = c->red_part.ensure(sizeof(double) * 10 * (nparts + 1)))) return rc;
  double* part = c->red_part.as<double>();
  double* out = part + 10 * nparts;
  if (batch) {
    if ((rc = c->sys_sums.ensure(sizeof(double) * 5 * (size_t)c->nsys))) return rc;
    double* sys_part = part + 10 * (size_t)c->nsys * slices;
    for (int s0 = 0; s0 < c->nsys; s0 += 65535) {  // (the grid's y limit)
      const int ns = std::min(65535, c->nsys - s0);
      k_reduce_slices<<<dim3(slices, ns), RED_NT, 0, c->stream>>>(
          c->sys_off.as<int>() + s0, c->pm.as<double>(), c->perm.as<int>(), c->red_acc, c->red_pot,
          part + 10 * (size_t)s0 * slices);
      ++c->nlaunch;
    }
    k_reduce_sys<<<(5 * c->nsys + 127) / 128, 128, 0, c->stream>>>(c->nsys, slices, part, sys_part,
                                                                   c->sys_sums.as<double>());
    ++c->nlaunch;
    k_reduce_final<<<5, 32, 0, c->stream>>>(c->nsys, sys_part, out);
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
