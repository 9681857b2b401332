// C ABI of the SFMM gravity solver: contexts, argument checks, the build and
// gravity pipelines, exports for tests, error reporting.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <new>
#include <vector>

#include "sfmm_internal.cuh"

#define SFMM_VERSION "sfmm-gb300 0.1"

int sfmm_internal_cuda_fail(cudaError_t e, const char*, const char*, int) {
  return (e == cudaErrorMemoryAllocation) ? SFMM_ENOMEM : SFMM_ECUDA;
}

int DevBuf::ensure(size_t need) {
  if (need == 0) need = 16;
  if (need <= bytes) return SFMM_OK;
  if (p) cudaFree(p);
  p = nullptr;
  bytes = 0;
  size_t grow = need + need / 8;
  if (cudaMalloc(&p, grow) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
    return SFMM_ENOMEM;
  }
  bytes = grow;
  return SFMM_OK;
}

void DevBuf::release() {
  if (p) cudaFree(p);
  p = nullptr;
  bytes = 0;
}

namespace sfmm {

int set_error(sfmm_ctx* c, int code, const char* msg) {
  if (c) c->last_error = msg ? msg : sfmm_strerror(code);
  return code;
}

// Read (and clear) the device status word: one stream synchronisation.
// With `counts`, the build's node and leaf counts come back in the same
// synchronisation (into c->nnodes, c->nleaves).
int sync_status(sfmm_ctx* c, int* bits, bool counts) {
  cudaError_t e = cudaMemcpyAsync(c->h_status, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess && counts)
    e = cudaMemcpyAsync(c->h_status + 1, c->d_counts, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) {
    c->last_error = cudaGetErrorString(e);
    return (e == cudaErrorMemoryAllocation) ? SFMM_ENOMEM : SFMM_ECUDA;
  }
  *bits = *c->h_status;
  if (counts) {
    c->nnodes = c->h_status[1];
    c->nleaves = c->h_status[2];
  }
  if (*bits) {
    e = cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream);
    if (e != cudaSuccess) return SFMM_ECUDA;
  }
  return SFMM_OK;
}

int run_walk_dump_write(sfmm_ctx* c, double theta, const long long* d_off, int* d_level, int* d_src);

}  // namespace sfmm

using namespace sfmm;

namespace {

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    cudaGetDevice(&cur);
    if (prev >= 0 && cur != prev) cudaSetDevice(prev);
  }
};

float elapsed(cudaEvent_t a, cudaEvent_t b) {
  float ms = 0.f;
  if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) {
    cudaGetLastError();
    return 0.f;
  }
  return ms;
}

int check_ctx(const sfmm_ctx* c) { return c ? SFMM_OK : SFMM_EINVAL; }

}  // namespace

extern "C" {

const char* sfmm_version(void) { return SFMM_VERSION; }

const char* sfmm_strerror(int code) {
  switch (code) {
    case SFMM_OK: return "ok";
    case SFMM_EINVAL: return "invalid argument";
    case SFMM_ENOMEM: return "device allocation failed";
    case SFMM_ECUDA: return "CUDA runtime error";
    case SFMM_ESTATE: return "call out of order (no tree built)";
    case SFMM_ESTACK: return "tree branch deeper than the walk supports";
    case SFMM_ECAPACITY: return "work buffer capacity exceeded";
    case SFMM_ENONFINITE: return "non-finite or non-positive input";
    case SFMM_ENOTIMPL: return "not implemented";
    default: return "unknown error";
  }
}

const char* sfmm_last_error(const sfmm_ctx* c) { return c ? c->last_error.c_str() : "no context"; }

int sfmm_create(sfmm_ctx** out, int device, int precision, void* stream) {
  if (!out) return SFMM_EINVAL;
  *out = nullptr;
  if (precision != SFMM_FP64 && precision != SFMM_FP32) return SFMM_EINVAL;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return SFMM_ECUDA;
  }
  if (device < 0 || device >= ndev) return SFMM_EINVAL;
  DeviceGuard g(device);
  sfmm_ctx* c = new (std::nothrow) sfmm_ctx();
  if (!c) return SFMM_ENOMEM;
  c->device = device;
  c->precision = precision;
  if (stream) {
    c->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete c;
      return SFMM_ECUDA;
    }
    c->owns_stream = true;
  }
  bool ok = cudaMalloc(&c->d_status, sizeof(int)) == cudaSuccess &&
            cudaMallocHost(&c->h_status, 4 * sizeof(int)) == cudaSuccess &&
            cudaMallocHost(&c->h_scalars, 64 * sizeof(double)) == cudaSuccess &&
            cudaMemset(c->d_status, 0, sizeof(int)) == cudaSuccess;
  for (int i = 0; ok && i < 8; ++i) ok = cudaEventCreate(&c->ev[i]) == cudaSuccess;
  if (ok) ok = cudaEventCreateWithFlags(&c->ev_stage, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    sfmm_destroy(c);
    return SFMM_ECUDA;
  }
  *out = c;
  return SFMM_OK;
}

}  // extern "C"

namespace sfmm {

// Every device buffer of a context.
std::vector<DevBuf*> ctx_buffers(sfmm_ctx* c) {
  return {&c->in_pos, &c->in_mass, &c->in_h, &c->out_acc, &c->out_pot, &c->keys_a, &c->keys_b,
                    &c->idx_a, &c->idx_b, &c->sort_counts, &c->scan_tmp, &c->bbox_part, &c->k_left,
                    &c->k_right, &c->k_first, &c->k_last, &c->par_int, &c->par_leaf, &c->chain,
                    &c->pre_int, &c->pre_leaf, &c->misc, &c->px, &c->py, &c->pz, &c->pm, &c->ph,
                    &c->perm, &c->pnode, &c->prel, &c->phh, &c->nfirst, &c->ncount, &c->nright,
                    &c->nparent, &c->ndepth, &c->ncx, &c->ncy, &c->ncz, &c->nsize, &c->nhmax, &c->nmass,
                    &c->l2bits, &c->flags, &c->geo_hi, &c->geo_lo, &c->leaf_node, &c->isleaf, &c->Qd,
                    &c->Qf, &c->ring, &c->far, &c->arena, &c->p2p_off, &c->p2p_cnt, &c->counters,
                    &c->red_part, &c->dump, &c->nlu, &c->level_nodes, &c->level_off, &c->level_cur,
                    &c->cf_arena, &c->cf_off, &c->cf_cnt, &c->Tnode, &c->leaf_order, &c->sys_off,
                    &c->sys_lsz, &c->psys, &c->sys_root, &c->wparent, &c->sys_sums,
                    &c->p2p_extra, &c->p2p_split, &c->p2p_slist, &c->p2p_part, &c->lf_acc, &c->lf_part,
                    &c->kd_ord, &c->kd_node, &c->kd_act, &c->kd_work, &c->kd_chunk, &c->kd_part, &c->kd_split,
                    &c->sym_own, &c->sym_recv, &c->wqueue, &c->sort_aux, &c->n_extv, &c->n_exti, &c->size_cand,
                    &c->fx_rec, &c->fx_items, &c->src_rows};
}

// Addresses and sizes of a context's buffers, folded into one number: a
// captured graph holds the addresses it was captured with.
unsigned long long buffers_fingerprint(sfmm_ctx* c) {
  unsigned long long f = 1469598103934665603ull;
  for (DevBuf* b : ctx_buffers(c)) {
    f = (f ^ (unsigned long long)(uintptr_t)b->p) * 1099511628211ull;
    f = (f ^ (unsigned long long)b->bytes) * 1099511628211ull;
  }
  return f;
}

}  // namespace sfmm

extern "C" {

void sfmm_destroy(sfmm_ctx* c) {
  if (!c) return;
  DeviceGuard g(c->device);
  if (c->stream) cudaStreamSynchronize(c->stream);
  for (DevBuf* b : ctx_buffers(c)) b->release();
  for (int i = 0; i < 8; ++i)
    if (c->ev[i]) cudaEventDestroy(c->ev[i]);
  if (c->ev_stage) cudaEventDestroy(c->ev_stage);
  if (c->d_status) cudaFree(c->d_status);
  if (c->h_status) cudaFreeHost(c->h_status);
  if (c->h_scalars) cudaFreeHost(c->h_scalars);
  if (c->h_level_pin) cudaFreeHost(c->h_level_pin);
  if (c->h_sys_pin) cudaFreeHost(c->h_sys_pin);
  if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
  if (c->owns_stream && c->stream) cudaStreamDestroy(c->stream);
  tune_table_free(c);
  delete c;
}

int sfmm_set_stream(sfmm_ctx* c, void* stream) {
  if (check_ctx(c)) return SFMM_EINVAL;
  DeviceGuard g(c->device);
  if (c->owns_stream && c->stream) {
    cudaStreamSynchronize(c->stream);
    cudaStreamDestroy(c->stream);
    c->stream = nullptr;
    c->owns_stream = false;
  }
  if (stream) {
    c->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) != cudaSuccess) return SFMM_ECUDA;
    c->owns_stream = true;
  }
  return SFMM_OK;
}

int sfmm_set_option(sfmm_ctx* c, const char* key, double v) {
  if (check_ctx(c) || !key) return SFMM_EINVAL;
  c->graph_valid = false;
  if (!std::isfinite(v)) return set_error(c, SFMM_EINVAL, "option value must be finite");
  if (!strcmp(key, "G")) {
    c->G = v;
  } else if (!strcmp(key, "self_potential")) {
    c->self_potential = (v != 0.0);
  } else if (!strcmp(key, "ring_capacity")) {
    int cap = (int)v;
    if (cap < 256 || cap > (1 << 24) || (cap & (cap - 1))) return set_error(c, SFMM_EINVAL, "ring_capacity: power of two in [256, 2^24]");
    c->ring_capacity = cap;
  } else if (!strcmp(key, "list_capacity")) {
    if (v < 0) return set_error(c, SFMM_EINVAL, "list_capacity must be >= 0");
    c->list_capacity = (int64_t)v;
  } else if (!strcmp(key, "walk")) {
    if (v != 0.0 && v != 1.0 && v != 2.0)
      return set_error(c, SFMM_EINVAL, "walk: 0 (per-leaf replay), 1 (per-node shared pairs), 2 (one-sided symmetric pairs)");
    c->walk_mode = (int)v;
  } else if (!strcmp(key, "schedule")) {
    if (v != 0.0 && v != 1.0 && v != 2.0 && v != 3.0)
      return set_error(c, SFMM_EINVAL,
                       "schedule: 0 (automatic), 1 (one launch per depth), 2 (queue of nodes), 3 (queue of sibling pairs)");
    c->schedule = (int)v;
  } else if (!strcmp(key, "p2p_chunk")) {
    if (v != std::floor(v) || v < 32 || v > 65536)
      return set_error(c, SFMM_EINVAL, "p2p_chunk: integer in [32, 65536]");
    c->p2p_chunk = (int)v;
  } else if (!strcmp(key, "p2p_blocks")) {
    if (v != std::floor(v) || v < 0 || v > 64) return set_error(c, SFMM_EINVAL, "p2p_blocks: integer in [0, 64]");
    c->p2p_blocks = (int)v;
  } else if (!strcmp(key, "autotune_theta")) {
    if (!(v >= 0.0 && v < 1.0)) return set_error(c, SFMM_EINVAL, "autotune_theta must be in [0, 1)");
    c->tune_theta = v;
  } else if (!strcmp(key, "autotune_order")) {
    if (v != std::floor(v) || v < 0 || v > SFMM_PMAX) return set_error(c, SFMM_EINVAL, "autotune_order must be in [0, 4]");
    c->tune_order = (int)v;
  } else if (!strcmp(key, "tree")) {
    if (v != 0.0 && v != 1.0) return set_error(c, SFMM_EINVAL, "tree: 0 (Morton radix tree) or 1 (centre-of-mass kd tree)");
    c->tree_kind = (int)v;
  } else if (!strcmp(key, "profile")) {
    c->profile = (v != 0.0);
  } else {
    return set_error(c, SFMM_EINVAL, "unknown option key");
  }
  return SFMM_OK;
}

}  // extern "C"

namespace {

// Build for nsys >= 1 systems packed back to back (h_sys_off / h_sys_lsz set).
int build_common(sfmm_ctx* c, const double* pos, const double* mass, const double* h) {
  c->built = false;
  c->graph_valid = false;
  c->moments_order = -1;
  int rc;
  if ((rc = c->sys_off.ensure(sizeof(int) * ((size_t)c->nsys + 1))) ||
      (rc = c->sys_lsz.ensure(sizeof(int) * (size_t)c->nsys)))
    return set_error(c, rc, "allocation failed");
  {
    // system offsets and leaf sizes through a pinned staging buffer: the
    // copies run in stream order without a wait here; the buffer is reused
    // once the previous build's copies have run (an event marks them)
    SFMM_CUDA_TRY(cudaEventSynchronize(c->ev_stage));
    const size_t need = (size_t)c->nsys + 1 + (size_t)c->nsys;
    if (need > c->h_sys_pin_cap) {
      if (c->h_sys_pin) cudaFreeHost(c->h_sys_pin);
      c->h_sys_pin = nullptr;
      c->h_sys_pin_cap = 0;
      if (cudaMallocHost(&c->h_sys_pin, sizeof(int) * need) != cudaSuccess) {
        c->h_sys_pin = nullptr;
        return set_error(c, SFMM_ENOMEM, "pinned allocation failed");
      }
      c->h_sys_pin_cap = need;
    }
    int* off32 = c->h_sys_pin;
    int* lsz = c->h_sys_pin + c->nsys + 1;
    for (int s = 0; s <= c->nsys; ++s) off32[s] = (int)c->h_sys_off[s];
    for (int s = 0; s < c->nsys; ++s) lsz[s] = c->h_sys_lsz[s];
    SFMM_CUDA_TRY(cudaMemcpyAsync(c->sys_off.p, off32, sizeof(int) * ((size_t)c->nsys + 1), cudaMemcpyHostToDevice,
                                  c->stream));
    SFMM_CUDA_TRY(cudaMemcpyAsync(c->sys_lsz.p, lsz, sizeof(int) * (size_t)c->nsys, cudaMemcpyHostToDevice,
                                  c->stream));
    SFMM_CUDA_TRY(cudaEventRecord(c->ev_stage, c->stream));
  }
  if (c->profile) cudaEventRecord(c->ev[0], c->stream);
  rc = build_tree(c, pos, mass, h);
  if (rc) return set_error(c, rc, "tree build failed");
  if (c->profile) cudaEventRecord(c->ev[1], c->stream);
  int bits = 0;
  if ((rc = sync_status(c, &bits, true))) return rc;
  if (bits & (SFMM_ST_NONFINITE | SFMM_ST_NONPOSITIVE))
    return set_error(c, SFMM_ENONFINITE, "non-finite position/mass/h or non-positive mass/h");
  if (bits) return set_error(c, SFMM_ECUDA, "internal consistency check of the tree failed");
  c->built = true;
  c->stats = sfmm_stats{};
  c->stats.n = c->n;
  c->stats.nnodes = c->nnodes;
  c->stats.nleaves = c->nleaves;
  if (c->profile) c->stats.ms_build = elapsed(c->ev[0], c->ev[1]);
  return SFMM_OK;
}

}  // namespace

extern "C" {

int sfmm_build(sfmm_ctx* c, int64_t n, const double* pos, const double* mass, const double* h, int leaf_size) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (n < 1 || n > ((int64_t)1 << 31) - 2) return set_error(c, SFMM_EINVAL, "n must be in [1, 2^31 - 2]");
  if (!pos || !mass || !h) return set_error(c, SFMM_EINVAL, "NULL input pointer");
  if (leaf_size < 1 || leaf_size > 64) return set_error(c, SFMM_EINVAL, "leaf_size must be in [1, 64]");
  DeviceGuard g(c->device);
  c->n = n;
  c->leaf_size = leaf_size;
  c->nsys = 1;
  c->h_sys_off.assign({0, n});
  c->h_sys_lsz.assign({leaf_size});
  return build_common(c, pos, mass, h);
}

int sfmm_build_batch(sfmm_ctx* c, int nsys, const int64_t* offsets, const double* pos, const double* mass,
                     const double* h, const int* leaf_size) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (nsys < 1 || nsys > 65536 || !offsets) return set_error(c, SFMM_EINVAL, "nsys must be in [1, 65536]");
  if (!pos || !mass || !h) return set_error(c, SFMM_EINVAL, "NULL input pointer");
  if (offsets[0] != 0) return set_error(c, SFMM_EINVAL, "offsets[0] must be 0");
  if (c->tree_kind != 0) return set_error(c, SFMM_ENOTIMPL, "batched builds use the Morton tree (option tree = 0)");
  for (int s = 0; s < nsys; ++s)
    if (offsets[s + 1] <= offsets[s]) return set_error(c, SFMM_EINVAL, "every system needs at least one particle");
  const int64_t n = offsets[nsys];
  if (n > ((int64_t)1 << 31) - 2) return set_error(c, SFMM_EINVAL, "total n must be <= 2^31 - 2");
  std::vector<int> lsz(nsys, 16);
  if (leaf_size)
    for (int s = 0; s < nsys; ++s) {
      if (leaf_size[s] < 1 || leaf_size[s] > 64) return set_error(c, SFMM_EINVAL, "leaf sizes must be in [1, 64]");
      lsz[s] = leaf_size[s];
    }
  DeviceGuard g(c->device);
  if (!leaf_size) {
    // autotuned: table entries, trials for groups without one
    c->built = false;
    int rc = tuned_leaf_sizes(c, nsys, offsets, pos, mass, h, c->tune_theta, c->tune_order, lsz);
    if (rc) return set_error(c, rc, c->last_error.empty() ? "autotune failed" : c->last_error.c_str());
  }
  c->n = n;
  c->leaf_size = *std::max_element(lsz.begin(), lsz.end());
  c->nsys = nsys;
  c->h_sys_off.assign(offsets, offsets + nsys + 1);
  c->h_sys_lsz = lsz;
  int rc = build_common(c, pos, mass, h);
  // autotuned builds also take the batch's cached launch knobs, if any
  if (rc == SFMM_OK && !leaf_size) rc = tuned_knobs(c, c->tune_theta, c->tune_order, nullptr, false);
  return rc;
}

int sfmm_autotune_cache(sfmm_ctx* c, const char* path) {
  if (check_ctx(c)) return SFMM_EINVAL;
  return tune_set_cache(c, path);
}

int sfmm_autotune_batch(sfmm_ctx* c, int nsys, const int64_t* offsets, const double* pos, const double* mass,
                        const double* h, double theta, int order, int* leaf_size_out) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!(theta >= 0.0 && theta < 1.0)) return set_error(c, SFMM_EINVAL, "theta must be in [0, 1)");
  if (order < 0 || order > SFMM_PMAX) return set_error(c, SFMM_EINVAL, "order must be in [0, 4]");
  c->tune_theta = theta;
  c->tune_order = order;
  int rc = sfmm_build_batch(c, nsys, offsets, pos, mass, h, nullptr);
  if (rc) return rc;
  DeviceGuard g(c->device);
  if ((rc = c->out_acc.ensure(sizeof(double) * 3 * (size_t)c->n))) return set_error(c, rc, "allocation failed");
  if ((rc = tuned_knobs(c, theta, order, c->out_acc.as<double>(), true)))
    return set_error(c, rc, c->last_error.empty() ? "autotune failed" : c->last_error.c_str());
  if (leaf_size_out) std::copy(c->h_sys_lsz.begin(), c->h_sys_lsz.end(), leaf_size_out);
  return SFMM_OK;
}

int sfmm_gravity(sfmm_ctx* c, double theta, int order, double* acc, double* pot) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!c->built) return set_error(c, SFMM_ESTATE, "sfmm_gravity before sfmm_build");
  if (!(theta >= 0.0 && theta < 1.0)) return set_error(c, SFMM_EINVAL, "theta must be in [0, 1)");
  if (order < 0 || order > SFMM_PMAX) return set_error(c, SFMM_EINVAL, "order must be in [0, 4]");
  if (!acc) return set_error(c, SFMM_EINVAL, "NULL acc");
  DeviceGuard g(c->device);
  int rc;
  cudaStream_t st = c->stream;
  if (c->profile) cudaEventRecord(c->ev[2], st);
  c->pref_order = order;  // later builds compute these moments on the way up
  if (c->moments_order != order) {
    if ((rc = compute_moments(c, order))) return set_error(c, rc, "moment pass failed");
  }
  // walk, near field and sums are issued without a host wait; one
  // synchronisation at the end reads the status word, the sums and the
  // walk's counters.  A walk buffer that ran out sets a status bit: grow it
  // and run again (the partial results are overwritten)
  unsigned long long* hs = reinterpret_cast<unsigned long long*>(c->h_scalars + 32);
  for (int attempt = 0;; ++attempt) {
    if (c->profile) cudaEventRecord(c->ev[3], st);
    if ((rc = (c->walk_mode >= 1) ? run_walk_shared(c, theta, order) : run_walk(c, theta, order, false, 0, 0)))
      return rc;
    if (c->profile) cudaEventRecord(c->ev[4], st);
    if ((rc = run_p2p(c, acc, pot))) return set_error(c, rc, "near-field pass failed");
    if (c->profile) cudaEventRecord(c->ev[5], st);
    double* red = nullptr;
    if ((rc = run_reduce(c, &red))) return set_error(c, rc, "reduction failed");
    if (c->profile) cudaEventRecord(c->ev[6], st);
    cudaError_t e = cudaMemcpyAsync(c->h_scalars + 16, red, 5 * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)  // walk counters (statistics, buffer needs) and pair evaluations
      e = cudaMemcpyAsync(hs, c->counters.p, 20 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return set_error(c, SFMM_ECUDA, cudaGetErrorString(e));
    int bits = 0;
    if ((rc = sync_status(c, &bits))) return rc;
    if (bits & SFMM_ST_DEPTH) return set_error(c, SFMM_ESTACK, "tree deeper than supported");
    if (c->walk_mode >= 1 && (bits & (SFMM_ST_RING | SFMM_ST_ARENA | SFMM_ST_CHILDLIST)) &&
        !(bits & ~(SFMM_ST_RING | SFMM_ST_ARENA | SFMM_ST_CHILDLIST | SFMM_ST_INTERNAL))) {
      // (an overflowing walk can leave the long-list split inconsistent:
      // SFMM_ST_INTERNAL then comes with a capacity bit and goes with it)
      if (attempt == SFMM_WALK_ATTEMPTS - 1)
        return set_error(c, SFMM_ECAPACITY, "walk buffers too small after the last regrow");
      walk_shared_regrow(c, bits, hs);
      continue;
    }
    if (bits & SFMM_ST_INTERNAL) return set_error(c, SFMM_ECUDA, "walk: internal consistency check failed");
    if (bits) return set_error(c, SFMM_ECUDA, "device status error after the near-field pass");
    break;
  }
  if (c->walk_mode >= 1) {
    c->stats.m2l = (int64_t)hs[0];
    c->stats.m2l_unique = (int64_t)hs[1];
    c->stats.p2p_leaves = (int64_t)hs[2];
    c->stats.mac_fallbacks = (int64_t)hs[4];
  }
  const double* r = c->h_scalars + 16;
  c->stats.momentum[0] = r[0];
  c->stats.momentum[1] = r[1];
  c->stats.momentum[2] = r[2];
  c->stats.abs_momentum = r[3];
  c->stats.W = 0.5 * r[4];
  c->stats.p2p_pairs = (int64_t)hs[3];
  if (c->profile) {
    c->stats.ms_moments = elapsed(c->ev[2], c->ev[3]);
    c->stats.ms_walk = elapsed(c->ev[3], c->ev[4]);
    c->stats.ms_p2p = elapsed(c->ev[4], c->ev[5]);
    c->stats.ms_reduce = elapsed(c->ev[5], c->ev[6]);
    c->stats.ms_gravity = elapsed(c->ev[2], c->ev[6]);
  }
  return SFMM_OK;
}

int sfmm_gravity_batch(sfmm_ctx* c, double theta, int order, double* acc, double* pot) {
  return sfmm_gravity(c, theta, order, acc, pot);
}

int sfmm_batch_sums(const sfmm_ctx* cc, int nsys, double* out) {
  sfmm_ctx* c = const_cast<sfmm_ctx*>(cc);
  if (check_ctx(c) || !out) return SFMM_EINVAL;
  if (!c->built) return SFMM_ESTATE;
  if (nsys != c->nsys) return set_error(c, SFMM_EINVAL, "nsys differs from the built batch");
  DeviceGuard g(c->device);
  SFMM_CUDA_TRY(cudaStreamSynchronize(c->stream));
  if (c->nsys == 1) {
    out[0] = c->stats.momentum[0];
    out[1] = c->stats.momentum[1];
    out[2] = c->stats.momentum[2];
    out[3] = c->stats.abs_momentum;
    out[4] = c->stats.W;
    return SFMM_OK;
  }
  if (!c->sys_sums.p) return SFMM_ESTATE;
  SFMM_CUDA_TRY(cudaMemcpy(out, c->sys_sums.p, sizeof(double) * 5 * (size_t)nsys, cudaMemcpyDeviceToHost));
  return SFMM_OK;
}

}  // extern "C"

namespace {

// One step, build and gravity, issued on the context's stream with no host
// wait: what sfmm_solve_graph captures.  It ends with the copies the host
// reads after a replay: sums, walk counters, status word, node and leaf
// counts (pinned buffers).
int issue_step(sfmm_ctx* c, const double* pos, const double* mass, const double* h, double theta, int order,
               double* acc, double* pot) {
  cudaStream_t st = c->stream;
  int rc;
  SFMM_CUDA_TRY(cudaMemsetAsync(c->d_status, 0, sizeof(int), st));
  if ((rc = build_tree(c, pos, mass, h))) return rc;
  if ((rc = run_walk_shared(c, theta, order))) return rc;
  if ((rc = run_p2p(c, acc, pot))) return rc;
  double* red = nullptr;
  if ((rc = run_reduce(c, &red))) return rc;
  SFMM_CUDA_TRY(cudaMemcpyAsync(c->h_scalars + 16, red, 5 * sizeof(double), cudaMemcpyDeviceToHost, st));
  SFMM_CUDA_TRY(cudaMemcpyAsync(c->h_scalars + 32, c->counters.p, 20 * sizeof(unsigned long long),
                                cudaMemcpyDeviceToHost, st));
  SFMM_CUDA_TRY(cudaMemcpyAsync(c->h_status, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  SFMM_CUDA_TRY(cudaMemcpyAsync(c->h_status + 1, c->d_counts, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
  return SFMM_OK;
}

// Captures issue_step into c->graph_exec.  False (and no graph) if the
// capture failed or a device buffer moved while it ran.
bool capture_step(sfmm_ctx* c, const double* pos, const double* mass, const double* h, double theta, int order,
                  double* acc, double* pot) {
  const unsigned long long mark = buffers_fingerprint(c);
  const int prof = c->profile;
  c->profile = 0;
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    c->profile = prof;
    return false;
  }
  const int rc = issue_step(c, pos, mass, h, theta, order, acc, pot);
  const cudaError_t e = cudaStreamEndCapture(c->stream, &g);
  c->profile = prof;
  bool ok = rc == SFMM_OK && e == cudaSuccess && g && buffers_fingerprint(c) == mark;
  cudaGraphExec_t ex = nullptr;
  if (ok) ok = cudaGraphInstantiate(&ex, g, 0) == cudaSuccess;
  if (g) cudaGraphDestroy(g);
  if (!ok) {
    cudaGetLastError();
    if (ex) cudaGraphExecDestroy(ex);
    return false;
  }
  if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
  c->graph_exec = ex;
  c->g_mark = mark;
  return true;
}

// Counts, sums and statistics of a replayed step, from the copies it made.
void replay_stats(sfmm_ctx* c, int order) {
  c->nnodes = c->h_status[1];
  c->nleaves = c->h_status[2];
  c->built = true;
  c->levels_ready = false;
  c->moments_order = order;
  c->pref_order = order;
  const unsigned long long* hs = reinterpret_cast<const unsigned long long*>(c->h_scalars + 32);
  const double* r = c->h_scalars + 16;
  c->stats = sfmm_stats{};
  c->stats.n = c->n;
  c->stats.nnodes = c->nnodes;
  c->stats.nleaves = c->nleaves;
  c->stats.m2l = (int64_t)hs[0];
  c->stats.m2l_unique = (int64_t)hs[1];
  c->stats.p2p_leaves = (int64_t)hs[2];
  c->stats.p2p_pairs = (int64_t)hs[3];
  c->stats.mac_fallbacks = (int64_t)hs[4];
  c->stats.momentum[0] = r[0];
  c->stats.momentum[1] = r[1];
  c->stats.momentum[2] = r[2];
  c->stats.abs_momentum = r[3];
  c->stats.W = 0.5 * r[4];
}

}  // namespace

extern "C" {

int sfmm_solve_graph(sfmm_ctx* c, int nsys, const int64_t* offsets, const double* pos, const double* mass,
                     const double* h, const int* leaf_size, double theta, int order, double* acc, double* pot) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (nsys < 1 || nsys > 65536 || !offsets) return set_error(c, SFMM_EINVAL, "nsys must be in [1, 65536]");
  if (!pos || !mass || !h || !acc) return set_error(c, SFMM_EINVAL, "NULL pointer");
  if (!(theta >= 0.0 && theta < 1.0)) return set_error(c, SFMM_EINVAL, "theta must be in [0, 1)");
  if (order < 0 || order > SFMM_PMAX) return set_error(c, SFMM_EINVAL, "order must be in [0, 4]");
  if (c->tree_kind != 0 || c->walk_mode != 1)
    return set_error(c, SFMM_ENOTIMPL, "captured steps run the Morton tree and the shared walk (walk 1)");
  if (offsets[nsys] < 2) return set_error(c, SFMM_EINVAL, "a captured step needs at least two particles");
  DeviceGuard g(c->device);
  std::vector<int64_t> off(offsets, offsets + nsys + 1);
  std::vector<int> lsz;
  if (leaf_size) lsz.assign(leaf_size, leaf_size + nsys);
  const void* ptr[5] = {pos, mass, h, acc, pot};
  bool same = c->graph_exec && c->graph_valid && buffers_fingerprint(c) == c->g_mark && c->g_off == off &&
              c->g_auto_leaf == !leaf_size && c->g_lsz == lsz && c->g_theta == theta && c->g_order == order;
  for (int k = 0; same && k < 5; ++k) same = c->g_ptr[k] == ptr[k];
  if (same) {
    cudaError_t e = cudaGraphLaunch(c->graph_exec, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return set_error(c, SFMM_ECUDA, cudaGetErrorString(e));
    const int bits = c->h_status[0];
    if (bits == 0) {
      replay_stats(c, order);
      ++c->graph_replays;
      c->nlaunch += c->g_launches;
      return SFMM_OK;
    }
    // a walk buffer ran out, or the inputs are bad: the ordinary path below
    // regrows and reruns, or reports the inputs
    if (bits & (SFMM_ST_RING | SFMM_ST_ARENA | SFMM_ST_CHILDLIST))
      walk_shared_regrow(c, bits, reinterpret_cast<const unsigned long long*>(c->h_scalars + 32));
    SFMM_CUDA_TRY(cudaMemsetAsync(c->d_status, 0, sizeof(int), c->stream));
    c->graph_valid = false;
  }
  // the ordinary build and gravity with buffers sized for any tree of these
  // particles, then the capture that the next calls replay
  c->graph_mode = true;
  int rc = sfmm_build_batch(c, nsys, offsets, pos, mass, h, leaf_size);
  if (rc == SFMM_OK) rc = sfmm_gravity(c, theta, order, acc, pot);
  if (rc == SFMM_OK) {
    const int64_t l0 = c->nlaunch;
    const sfmm_stats keep = c->stats;
    if (capture_step(c, pos, mass, h, theta, order, acc, pot)) {
      c->graph_valid = true;
      c->g_off = off;
      c->g_lsz = lsz;
      c->g_auto_leaf = !leaf_size;
      c->g_theta = theta;
      c->g_order = order;
      for (int k = 0; k < 5; ++k) c->g_ptr[k] = ptr[k];
      c->g_launches = c->nlaunch - l0;
    }
    c->nlaunch = l0;  // captured, not run
    c->stats = keep;
  }
  c->graph_mode = false;
  return rc;
}

}  // extern "C"

namespace {

// Copies between host and device memory by a kernel when the host side is
// device-accessible (pinned or registered): on GB300 the GPU reads and
// writes host memory over the chip-to-chip link faster than a copy engine
// moves it.  Otherwise (pageable memory) a stream copy.
__global__ void k_copy_f64(const double2* __restrict__ src, double2* __restrict__ dst, int64_t n2,
                           const double* __restrict__ src_tail, double* __restrict__ dst_tail, int tail) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
  if (tail && blockIdx.x == 0 && threadIdx.x == 0) *dst_tail = *src_tail;
}

const double* device_view(const void* p) {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) return static_cast<const double*>(p);
  if (at.type == cudaMemoryTypeHost && at.devicePointer) return static_cast<const double*>(at.devicePointer);
  return nullptr;
}

int copy_f64(sfmm_ctx* c, double* dst, const double* src, int64_t count, cudaMemcpyKind kind) {
  const double* hs = (kind == cudaMemcpyHostToDevice) ? device_view(src) : nullptr;
  double* hd = (kind == cudaMemcpyDeviceToHost) ? const_cast<double*>(device_view(dst)) : nullptr;
  const double* s = (kind == cudaMemcpyHostToDevice) ? hs : src;
  double* d = (kind == cudaMemcpyDeviceToHost) ? hd : dst;
  const bool aligned = ((reinterpret_cast<uintptr_t>(s) | reinterpret_cast<uintptr_t>(d)) & 15u) == 0;
  if (s && d && aligned) {
    const int64_t n2 = count / 2;
    const int blocks = (int)std::min<int64_t>((n2 + 255) / 256, 8 * (int64_t)num_sms(c->device));
    k_copy_f64<<<std::max(blocks, 1), 256, 0, c->stream>>>(reinterpret_cast<const double2*>(s),
                                                           reinterpret_cast<double2*>(d), n2, s + count - 1,
                                                           d + count - 1, (int)(count & 1));
    ++c->nlaunch;
    SFMM_CUDA_TRY(cudaGetLastError());
    return SFMM_OK;
  }
  SFMM_CUDA_TRY(cudaMemcpyAsync(dst, src, sizeof(double) * count, kind, c->stream));
  return SFMM_OK;
}

}  // namespace

extern "C" {

int sfmm_solve_host(sfmm_ctx* c, int64_t n, const double* pos, const double* mass, const double* h, int leaf_size,
                    double theta, int order, double* acc, double* pot) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!pos || !mass || !h || !acc) return set_error(c, SFMM_EINVAL, "NULL pointer");
  if (n < 1 || n > ((int64_t)1 << 31) - 2) return set_error(c, SFMM_EINVAL, "n must be in [1, 2^31 - 2]");
  if (!(theta >= 0.0 && theta < 1.0)) return set_error(c, SFMM_EINVAL, "theta must be in [0, 1)");
  if (order < 0 || order > SFMM_PMAX) return set_error(c, SFMM_EINVAL, "order must be in [0, 4]");
  if (leaf_size < 1 || leaf_size > 64) return set_error(c, SFMM_EINVAL, "leaf_size must be in [1, 64]");
  DeviceGuard g(c->device);
  int rc;
  if ((rc = c->in_pos.ensure(sizeof(double) * 3 * (size_t)n)) || (rc = c->in_mass.ensure(sizeof(double) * n)) ||
      (rc = c->in_h.ensure(sizeof(double) * n)) || (rc = c->out_acc.ensure(sizeof(double) * 3 * (size_t)n)) ||
      (rc = c->out_pot.ensure(sizeof(double) * n)))
    return set_error(c, rc, "staging allocation failed");
  cudaStream_t st = c->stream;
  if ((rc = copy_f64(c, c->in_pos.as<double>(), pos, 3 * n, cudaMemcpyHostToDevice)) ||
      (rc = copy_f64(c, c->in_mass.as<double>(), mass, n, cudaMemcpyHostToDevice)) ||
      (rc = copy_f64(c, c->in_h.as<double>(), h, n, cudaMemcpyHostToDevice)))
    return rc;
  if (c->tree_kind == 0 && c->walk_mode == 1 && n >= 2) {
    // build + gravity as the captured step (one host wait; bitwise the
    // results of the separate calls): the staging buffers keep their
    // addresses, so repeated calls of one shape replay one graph
    const int64_t off[2] = {0, n};
    const int lsz[1] = {leaf_size};
    if ((rc = sfmm_solve_graph(c, 1, off, c->in_pos.as<double>(), c->in_mass.as<double>(), c->in_h.as<double>(), lsz,
                               theta, order, c->out_acc.as<double>(), pot ? c->out_pot.as<double>() : nullptr)))
      return rc;
  } else {
    if ((rc = sfmm_build(c, n, c->in_pos.as<double>(), c->in_mass.as<double>(), c->in_h.as<double>(), leaf_size)))
      return rc;
    if ((rc = sfmm_gravity(c, theta, order, c->out_acc.as<double>(), pot ? c->out_pot.as<double>() : nullptr)))
      return rc;
  }
  if ((rc = copy_f64(c, acc, c->out_acc.as<double>(), 3 * n, cudaMemcpyDeviceToHost))) return rc;
  if (pot && (rc = copy_f64(c, pot, c->out_pot.as<double>(), n, cudaMemcpyDeviceToHost))) return rc;
  SFMM_CUDA_TRY(cudaStreamSynchronize(st));
  return SFMM_OK;
}

int sfmm_get_stats(const sfmm_ctx* c, sfmm_stats* out) {
  if (check_ctx(c) || !out) return SFMM_EINVAL;
  *out = c->stats;
  out->kernel_launches = c->nlaunch;
  out->graph_replays = c->graph_replays;
  return SFMM_OK;
}

int sfmm_tree_size(const sfmm_ctx* c, int64_t* nnodes, int64_t* nleaves) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!c->built) return SFMM_ESTATE;
  if (nnodes) *nnodes = c->nnodes;
  if (nleaves) *nleaves = c->nleaves;
  return SFMM_OK;
}

int sfmm_tree_export(const sfmm_ctx* cc, int64_t* perm, uint64_t* keys, int32_t* first, int32_t* count,
                     int32_t* right, int32_t* parent, int32_t* depth, double* centre, double* size, double* hmax,
                     double* mass, int32_t* leaves) {
  sfmm_ctx* c = const_cast<sfmm_ctx*>(cc);
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!c->built) return SFMM_ESTATE;
  DeviceGuard g(c->device);
  const size_t n = (size_t)c->n, nn = (size_t)c->nnodes;
  cudaStream_t st = c->stream;
  int rc;
  if (depth && (rc = compute_depth(c))) return rc;
  SFMM_CUDA_TRY(cudaStreamSynchronize(st));
  if (perm) {
    std::vector<int32_t> tmp(n);
    SFMM_CUDA_TRY(cudaMemcpy(tmp.data(), c->perm.p, n * sizeof(int32_t), cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < n; ++i) perm[i] = tmp[i];
  }
  if (keys) SFMM_CUDA_TRY(cudaMemcpy(keys, c->keys_a.p, n * sizeof(uint64_t), cudaMemcpyDeviceToHost));
  if (first) SFMM_CUDA_TRY(cudaMemcpy(first, c->nfirst.p, nn * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (count) SFMM_CUDA_TRY(cudaMemcpy(count, c->ncount.p, nn * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (right) SFMM_CUDA_TRY(cudaMemcpy(right, c->nright.p, nn * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (parent) SFMM_CUDA_TRY(cudaMemcpy(parent, c->nparent.p, nn * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (depth) SFMM_CUDA_TRY(cudaMemcpy(depth, c->ndepth.p, nn * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (centre) {
    std::vector<double> x(nn), y(nn), z(nn);
    SFMM_CUDA_TRY(cudaMemcpy(x.data(), c->ncx.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
    SFMM_CUDA_TRY(cudaMemcpy(y.data(), c->ncy.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
    SFMM_CUDA_TRY(cudaMemcpy(z.data(), c->ncz.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
    for (size_t v = 0; v < nn; ++v) {
      centre[3 * v] = x[v];
      centre[3 * v + 1] = y[v];
      centre[3 * v + 2] = z[v];
    }
  }
  if (size) SFMM_CUDA_TRY(cudaMemcpy(size, c->nsize.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
  if (hmax) SFMM_CUDA_TRY(cudaMemcpy(hmax, c->nhmax.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
  if (mass) SFMM_CUDA_TRY(cudaMemcpy(mass, c->nmass.p, nn * sizeof(double), cudaMemcpyDeviceToHost));
  if (leaves) SFMM_CUDA_TRY(cudaMemcpy(leaves, c->leaf_node.p, (size_t)c->nleaves * sizeof(int32_t), cudaMemcpyDeviceToHost));
  return SFMM_OK;
}

int sfmm_moments_export(sfmm_ctx* c, int order, double* Q, int32_t* mi) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!c->built) return SFMM_ESTATE;
  if (order < 0 || order > SFMM_PMAX) return SFMM_EINVAL;
  DeviceGuard g(c->device);
  int rc;
  if ((c->moments_order != order || !c->moments_fp64) && (rc = compute_moments(c, order))) return rc;
  const int nq = ncoef(order);
  SFMM_CUDA_TRY(cudaStreamSynchronize(c->stream));
  if (Q) SFMM_CUDA_TRY(cudaMemcpy(Q, c->Qd.p, sizeof(double) * (size_t)c->nnodes * nq, cudaMemcpyDeviceToHost));
  if (mi) {
    int k = 0;
    for (int n = 0; n <= order; ++n)
      for (int a = n; a >= 0; --a)
        for (int b = n - a; b >= 0; --b) {
          mi[3 * k] = a;
          mi[3 * k + 1] = b;
          mi[3 * k + 2] = n - a - b;
          ++k;
        }
  }
  return SFMM_OK;
}

int sfmm_lists(sfmm_ctx* c, double theta, int64_t* m2l_off, int32_t* m2l_level, int32_t* m2l_src, int64_t cap_m2l,
               int64_t* p2p_off, int32_t* p2p_src, int64_t cap_p2p) {
  if (check_ctx(c)) return SFMM_EINVAL;
  if (!c->built) return SFMM_ESTATE;
  if (!(theta >= 0.0 && theta < 1.0)) return set_error(c, SFMM_EINVAL, "theta must be in [0, 1)");
  if (!m2l_off || !p2p_off) return set_error(c, SFMM_EINVAL, "NULL offsets");
  DeviceGuard g(c->device);
  const int nl = c->nleaves;
  int rc;
  if ((rc = run_walk(c, theta, 0, true, 0, 0))) return rc;
  std::vector<int> cnt(nl), pcnt(nl);
  std::vector<long long> poff(nl);
  SFMM_CUDA_TRY(cudaMemcpy(cnt.data(), c->dump.p, sizeof(int) * nl, cudaMemcpyDeviceToHost));
  m2l_off[0] = 0;
  for (int q = 0; q < nl; ++q) m2l_off[q + 1] = m2l_off[q] + cnt[q];
  const int64_t tot = m2l_off[nl];
  if (m2l_level && m2l_src) {
    if (cap_m2l < tot) return set_error(c, SFMM_ECAPACITY, "m2l capacity too small");
    DevBuf off, lev, src;
    if ((rc = off.ensure(sizeof(long long) * (nl + 1))) || (rc = lev.ensure(sizeof(int) * (size_t)(tot + 1))) ||
        (rc = src.ensure(sizeof(int) * (size_t)(tot + 1))))
      return rc;
    std::vector<long long> offh(nl + 1);
    for (int q = 0; q <= nl; ++q) offh[q] = m2l_off[q];
    cudaMemcpy(off.p, offh.data(), sizeof(long long) * (nl + 1), cudaMemcpyHostToDevice);
    rc = run_walk_dump_write(c, theta, off.as<long long>(), lev.as<int>(), src.as<int>());
    if (rc == SFMM_OK) {
      cudaMemcpy(m2l_level, lev.p, sizeof(int) * (size_t)tot, cudaMemcpyDeviceToHost);
      cudaMemcpy(m2l_src, src.p, sizeof(int) * (size_t)tot, cudaMemcpyDeviceToHost);
    }
    off.release();
    lev.release();
    src.release();
    if (rc) return rc;
  }
  SFMM_CUDA_TRY(cudaMemcpy(pcnt.data(), c->p2p_cnt.p, sizeof(int) * nl, cudaMemcpyDeviceToHost));
  SFMM_CUDA_TRY(cudaMemcpy(poff.data(), c->p2p_off.p, sizeof(long long) * nl, cudaMemcpyDeviceToHost));
  p2p_off[0] = 0;
  for (int q = 0; q < nl; ++q) p2p_off[q + 1] = p2p_off[q] + pcnt[q];
  if (p2p_src) {
    if (cap_p2p < p2p_off[nl]) return set_error(c, SFMM_ECAPACITY, "p2p capacity too small");
    for (int q = 0; q < nl; ++q)
      if (pcnt[q])
        SFMM_CUDA_TRY(cudaMemcpy(p2p_src + p2p_off[q], c->arena.as<int>() + poff[q], sizeof(int) * pcnt[q],
                                 cudaMemcpyDeviceToHost));
  }
  return SFMM_OK;
}

}  // extern "C"
