// Kernels shared by both windows: the final per-template reduction, the standalone
// marginalisation, and a batch's input and index phases.
#include <math.h>

#include "fmap_batch.cuh"
#include "fmap_front.cuh"

namespace fmap {

// ---------------------------------------------------------------------------
// Final reduction in two levels, accumulated in FP64: level 1 merges groups of
// kRedGroup tile partials per template (many blocks), level 2 merges the
// groups of one template (one block).  Each level fixes the order of its
// additions (per-thread strided loop, then a fixed tree), so the result is
// deterministic.
// ---------------------------------------------------------------------------
constexpr int kRedThreads = 256;
constexpr int kRedGroup = 2048;

struct __align__(32) Partial64 {
  double sum;      // sum of exp(F - max2F/2) over the group's valid cells
  float max2F;
  int32_t arg;
  long long nvalid;
  long long pad;
};

// Block-wide (max, count) then (sum, min arg at max) over items get(b),
// b in [0, n).  Returns the block's merged partial in thread 0.
template <typename Get>
__device__ __forceinline__ Partial64 block_merge(int64_t n, Get get) {
  __shared__ float s_max[kRedThreads];
  __shared__ long long s_cnt[kRedThreads];
  __shared__ double s_sum[kRedThreads];
  __shared__ int32_t s_arg[kRedThreads];
  const int tid = threadIdx.x;
  float mx = -1.0f;
  long long cnt = 0;
  for (int64_t b = tid; b < n; b += kRedThreads) {
    const Partial64 q = get(b);
    if (q.nvalid > 0) {
      mx = fmaxf(mx, q.max2F);
      cnt += q.nvalid;
    }
  }
  s_max[tid] = mx;
  s_cnt[tid] = cnt;
  __syncthreads();
  for (int w = kRedThreads / 2; w > 0; w >>= 1) {
    if (tid < w) {
      s_max[tid] = fmaxf(s_max[tid], s_max[tid + w]);
      s_cnt[tid] += s_cnt[tid + w];
    }
    __syncthreads();
  }
  const float M = s_max[0];
  const long long N = s_cnt[0];
  __syncthreads();
  double sum = 0.0;
  int32_t arg = kNoArg;
  if (N > 0) {
    for (int64_t b = tid; b < n; b += kRedThreads) {
      const Partial64 q = get(b);
      if (q.nvalid > 0) {
        // Rescale factor exp((max2F - M) / 2) <= 1 in FP32 (relative error
        // ~1e-7, the order of the FP32 tile sums themselves), accumulated in
        // FP64; factors below 2^-126 flush to 0.
        float f;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((q.max2F - M) * 0.72134752044448170368f));
        sum += q.sum * (double)f;
        if (q.max2F == M && q.arg < arg) arg = q.arg;
      }
    }
  }
  s_sum[tid] = sum;
  s_arg[tid] = arg;
  __syncthreads();
  for (int w = kRedThreads / 2; w > 0; w >>= 1) {
    if (tid < w) {
      s_sum[tid] += s_sum[tid + w];
      s_arg[tid] = min(s_arg[tid], s_arg[tid + w]);
    }
    __syncthreads();
  }
  Partial64 r;
  r.sum = s_sum[0];
  r.max2F = M;
  r.arg = s_arg[0];
  r.nvalid = N;
  r.pad = 0;
  return r;
}

__device__ __forceinline__ Partial64 widen(const Partial& q) {
  Partial64 r;
  r.sum = (double)q.sum;
  r.max2F = q.max2F;
  r.arg = q.arg;
  r.nvalid = q.nvalid;
  r.pad = 0;
  return r;
}

// Level 1: block (g, t) merges slots [g*kRedGroup, (g+1)*kRedGroup) of the
// concatenation [main tiles 0..n_tiles) ++ [fix-up slots in use, from fix0] (n_flag
// of them marked among `entries`; null: none).
__device__ __forceinline__ void reduce_groups_body(const Partial* __restrict__ parts, int64_t n_tiles, int64_t fix0,
                const int32_t* __restrict__ n_flag, int64_t entries,
                int64_t stride, int64_t n_groups, Partial64* __restrict__ groups,
    const uint3 bid, const dim3 gdim) {
  const int64_t n_fix = n_flag ? fix_slots_used(min((int64_t)*n_flag, entries)) : 0;
  const Partial* pp = parts + (int64_t)bid.y * stride;
  const int64_t n_all = n_tiles + n_fix;
  const int64_t lo = (int64_t)bid.x * kRedGroup;
  const int64_t n = max((int64_t)0, min((int64_t)kRedGroup, n_all - lo));
  const Partial64 r = block_merge(n, [&](int64_t b) {
    const int64_t k = lo + b;
    return widen(k < n_tiles ? pp[k] : pp[fix0 + (k - n_tiles)]);
  });
  if (threadIdx.x == 0) groups[(int64_t)bid.y * n_groups + bid.x] = r;
}

__global__ void __launch_bounds__(kRedThreads)
k_reduce_groups(const Partial* __restrict__ parts, int64_t n_tiles, int64_t fix0,
                const int32_t* __restrict__ n_flag, int64_t entries, int64_t stride,
                int64_t n_groups, Partial64* __restrict__ groups) {
  reduce_groups_body(parts, n_tiles, fix0, n_flag, entries, stride, n_groups, groups, blockIdx, gridDim);
}

// Level 2: one block per template over its groups; writes the summary.
__device__ __forceinline__ void reduce_final_body(const Partial64* __restrict__ groups, int64_t n_groups, int32_t n_tau,
               double log_prior, fmap_summary* __restrict__ out, const uint3 bid, const dim3 gdim) {
  const Partial64* gp = groups + (int64_t)bid.x * n_groups;
  const Partial64 r = block_merge(n_groups, [&](int64_t b) { return gp[b]; });
  if (threadIdx.x == 0) {
    fmap_summary o;
    o.flags = 0;
    o.n_valid = r.nvalid;
    if (r.nvalid == 0) {
      o.max2F = 0.0f;
      o.m = -1;
      o.n = -1;
      o.logB = nan("");
    } else {
      o.max2F = r.max2F;
      o.m = r.arg / n_tau;
      o.n = r.arg % n_tau;
      o.logB = 0.5 * (double)r.max2F + log(r.sum) - log((double)r.nvalid) + log_prior;
    }
    out[bid.x] = o;
  }
}

__global__ void __launch_bounds__(kRedThreads)
k_reduce_final(const Partial64* __restrict__ groups, int64_t n_groups, int32_t n_tau,
               double log_prior, fmap_summary* __restrict__ out) {
  reduce_final_body(groups, n_groups, n_tau, log_prior, out, blockIdx, gridDim);
}

int64_t reduce_groups_of(int64_t slots) { return std::max<int64_t>(1, (slots + kRedGroup - 1) / kRedGroup); }

static cudaError_t reduce_into(const Partial* parts, int64_t n_tiles, int64_t fix0,
                               const int32_t* n_flag, int64_t entries, int64_t stride, int32_t T, int32_t n_tau, double log_prior,
                               Partial64* groups, fmap_summary* d_summary, cudaStream_t s) {
  const int64_t n_groups = reduce_groups_of(n_tiles + (n_flag ? kFixSlots : 0));
  k_reduce_groups<<<dim3((unsigned)n_groups, (unsigned)T), kRedThreads, 0, s>>>(
      parts, n_tiles, fix0, n_flag, entries, stride, n_groups, groups);
  k_reduce_final<<<T, kRedThreads, 0, s>>>(groups, n_groups, n_tau > 0 ? n_tau : 1, log_prior,
                                           d_summary);
  return cudaGetLastError();
}

cudaError_t launch_final_reduce(fmap_plan_s* p, int64_t n_tiles, const fmap_atoms* a,
                                fmap_summary* d_summary, cudaStream_t s) {
  if (!d_summary || p->n_templates == 0) return cudaSuccess;
  const int64_t entries = (int64_t)p->grid.n_t0 * p->grid.n_tau *
                          (a && !a->shared_antenna ? p->n_templates : 1);
  const bool fix = a && entries > 0;
  p->launches += 2;
  return reduce_into(p->ws.partials, n_tiles, p->n_tiles, fix ? p->ws.n_flag : nullptr, entries,
                     p->part_stride, p->n_templates, p->grid.n_tau, p->log_prior,
                     (Partial64*)p->ws.groups, d_summary, s);
}

// ---------------------------------------------------------------------------
// Standalone marginalisation of a given map: 2048 cells per tile.
// ---------------------------------------------------------------------------
constexpr int kMargThreads = 256;
constexpr int kMargPer = 8;

int64_t marg_tiles(const fmap_grid& g) {
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  return (cells + kMargThreads * kMargPer - 1) / (kMargThreads * kMargPer);
}

__global__ void __launch_bounds__(kMargThreads)
k_marg_partials(const float* __restrict__ map, const uint8_t* __restrict__ valid, int64_t cells,
                int64_t stride, Partial* __restrict__ parts) {
  __shared__ Partial scratch[kMargThreads / 32];
  const int64_t tile = blockIdx.x;
  const int64_t tmpl = blockIdx.y;
  const float* mp = map + tmpl * cells;
  const uint8_t* vp = valid ? valid + tmpl * cells : nullptr;
  Partial acc = partial_empty();
  const int64_t base = tile * (kMargThreads * kMargPer);
#pragma unroll
  for (int k = 0; k < kMargPer; ++k) {
    const int64_t c = base + k * kMargThreads + threadIdx.x;
    if (c < cells) {
      const bool ok = vp ? (vp[c] != 0) : true;
      partial_add(acc, mp[c], (int32_t)c, ok);
    }
  }
  acc = partial_block_reduce<kMargThreads / 32>(acc, scratch);
  if (threadIdx.x == 0) parts[tmpl * stride + tile] = acc;
}

cudaError_t launch_marginalise_into(const fmap_grid& g, int32_t n_templates, const float* d_2F,
                                    const uint8_t* d_valid, Partial* parts, double log_prior,
                                    fmap_summary* d_summary, cudaStream_t s) {
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  const int64_t tiles = marg_tiles(g);
  if (n_templates == 0) return cudaSuccess;
  if (tiles > 0) {
    dim3 grid((unsigned)tiles, (unsigned)n_templates);
    k_marg_partials<<<grid, kMargThreads, 0, s>>>(d_2F, d_valid, cells, tiles, parts);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // the group results of the first level follow the tile partials
  Partial64* groups = (Partial64*)(parts + (int64_t)n_templates * tiles);
  groups = (Partial64*)(((uintptr_t)groups + 31) & ~(uintptr_t)31);
  return reduce_into(parts, tiles, 0, nullptr, 0, tiles, n_templates, g.n_tau, log_prior, groups,
                     d_summary, s);
}

cudaError_t launch_marginalise(fmap_plan_s* p, const float* d_2F, const uint8_t* d_valid,
                               fmap_summary* d_summary, cudaStream_t s) {
  const int64_t cells = (int64_t)p->grid.n_t0 * p->grid.n_tau;
  const int64_t tiles = marg_tiles(p->grid);
  if (tiles > 0 && p->n_templates > 0) {
    dim3 grid((unsigned)tiles, (unsigned)p->n_templates);
    k_marg_partials<<<grid, kMargThreads, 0, s>>>(d_2F, d_valid, cells, p->part_stride,
                                                  p->ws.partials);
    p->launches += 1;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return launch_final_reduce(p, tiles, nullptr, d_summary, s);
}


// ---- persistent multi-instance dispatchers (uneven batches) ----
__global__ void __launch_bounds__(256) kb_prep(const BItem* __restrict__ items, BUnits u) {
  // units [0, ru): relative times; then the marked-entry bitmask is cleared
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int64_t ru = it.n_sft > 0 ? (it.n_alloc + 255) / 256 : 0;
    if (k < ru) {
      prep_body(it.t, it.n_sft, it.n_alloc, it.rel_t, it.t_base, it.dev_err, it.antenna,
                (int64_t)3 * it.n_sft * it.n_ant, it.fafb, (int64_t)4 * it.n_sft * it.T, it.irr, it.level,
                make_uint3((unsigned)k, 0, 0), dim3((unsigned)ru));
    } else {
      const int64_t w0 = (k - ru) * kBitsPerUnit;
      const int64_t w1 = min(flag_words(it.flag_entries), w0 + kBitsPerUnit);
      for (int64_t w = w0 + threadIdx.x; w < w1; w += blockDim.x) it.flag_bits[w] = 0u;
    }
  });
}
static_assert(kIdxRowsPerUnit == kIdxGroup, "a batch index unit is one row group");
__global__ void __launch_bounds__(kIdxThreads) kb_index(const BItem* __restrict__ items, BUnits u) {
  __shared__ IndexSmem sm;
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int32_t m0 = (int32_t)k * kIdxRowsPerUnit;
    index_body(RelStored{it.rel_t}, it.n_sft > 0 ? *it.t_base : 0, it.n_sft, it.g, it.ax, it.i0,
               it.jend, m0, min(kIdxRowsPerUnit, it.g.n_t0 - m0), sm);
  });
}
__global__ void __launch_bounds__(kRedThreads) kb_red_groups(const BItem* __restrict__ items,
                                                             BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    reduce_groups_body(it.partials, it.tiles_used, it.n_tiles, it.cells > 0 ? it.n_flag : nullptr,
                       it.flag_entries, it.part_stride, it.red_groups,
                       (Partial64*)it.red_buf,
                       make_uint3((unsigned)(k % it.red_groups), (unsigned)(k / it.red_groups), 0),
                       dim3((unsigned)it.red_groups, (unsigned)it.T));
  });
}
__global__ void __launch_bounds__(kRedThreads) kb_red_final(const BItem* __restrict__ items,
                                                            BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    reduce_final_body((const Partial64*)it.red_buf, it.red_groups, it.g.n_tau > 0 ? it.g.n_tau : 1,
                      it.log_prior, it.summary, make_uint3((unsigned)k, 0, 0),
                      dim3((unsigned)it.T));
  });
}
const void* batch_kernel_common(int phase) {
  switch (phase) {
    case BP_PREP: return (const void*)kb_prep;
    case BP_INDEX: return (const void*)kb_index;
    case BP_RED_GROUPS: return (const void*)kb_red_groups;
    case BP_RED_FINAL: return (const void*)kb_red_final;
  }
  return nullptr;
}

}  // namespace fmap
