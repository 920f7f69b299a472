// Ill-conditioned cells.
//
// 2F depends on the component of (Fa, Fb) along the weak eigenvector of the
// 2x2 antenna matrix; for a window of a few SFTs of one detector the matrix is
// nearly singular (A B / D up to ~1e7), and any sum rounded to FP32 loses
// ~eps_32 sqrt(AB/D) of relative accuracy in 2F.  The per-cell coefficient
// step marks cells with AB/D > kCondThreshold (Coef.valid = 2); these are
// rare (well below 1% of the cells of the workloads) and always short
// windows in practice.  The fast kernels leave them out, and this file:
//   1. compacts the marked cells into a list in a deterministic order: the
//      coefficient kernels set one bit per marked entry; each unit of the bitmask
//      counts the bits before it and writes its own in order (long bitmasks:
//      per-unit counts, one exclusive scan, ordered writes);
//   2. recomputes each listed cell for every template from the definition
//      over its window (Sec. 2: windowed sums, Eq. F_FaFb) in float-float
//      arithmetic (a value is an unevaluated pair of FP32 numbers, ~2^-47
//      relative per operation; GB300 runs FP64 at 1/64 of the FP32 rate),
//      with D = A B - C^2 and the numerator of 2F formed in float-float too,
//      writes its 2F and adds it to per-block reduction partials kept in
//      their own slots, merged by the final reduction.
#include <math.h>

#include "fmap_batch.cuh"
#include "fmap_device.cuh"

namespace fmap {

constexpr int kFlagBlock = 1024;
constexpr int kFixThreads = 128;
static_assert(kFixPerSlot == kFixThreads, "one entry per thread in a slot");
constexpr int kFixBlocks = 32;   // slots in flight of a template group

// Per unit of kFlagUnit entries: the number of entries marked in the
// bitmask (valid == 2), from the unit's kFlagUnit / 32 words.
constexpr int kFlagWords = kFlagUnit / 32;
static_assert(kFlagWords <= kFlagBlock, "one word per thread");
__device__ __forceinline__ void flag_count_body(const uint32_t* __restrict__ bits, int64_t n_entries, int32_t* __restrict__ blockcnt,
    const uint3 bid, const dim3 gdim) {
  __shared__ int32_t warp_cnt[kFlagBlock / 32];
  const int tid = threadIdx.x;
  const unsigned c = tid < kFlagWords ? (unsigned)__popc(bits[(int64_t)bid.x * kFlagWords + tid]) : 0u;
  const unsigned wsum = __reduce_add_sync(0xffffffffu, c);
  if ((tid & 31) == 0) warp_cnt[tid >> 5] = (int32_t)wsum;
  __syncthreads();
  if (tid < 32) {
    const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)warp_cnt[tid]);
    if (tid == 0) blockcnt[bid.x] = (int32_t)t;
  }
}

__global__ void __launch_bounds__(kFlagBlock)
k_flag_count(const uint32_t* __restrict__ bits, int64_t n_entries, int32_t* __restrict__ blockcnt) {
  flag_count_body(bits, n_entries, blockcnt, blockIdx, gridDim);
}

// Exclusive scan of the block counts (one block); total into *n_flag.
__device__ __forceinline__ void flag_scan_body(int32_t* __restrict__ blockcnt, int64_t n_blocks, int32_t* __restrict__ n_flag,
    const uint3 bid, const dim3 gdim) {
  __shared__ int32_t warp_sum[32];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t base = 0; base < n_blocks; base += 1024) {
    const int64_t i = base + threadIdx.x;
    const int32_t v = i < n_blocks ? blockcnt[i] : 0;
    int32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      int32_t w = warp_sum[lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, w, d);
        if (lane >= d) w += y;
      }
      warp_sum[lane] = w;  // inclusive
    }
    __syncthreads();
    const int32_t excl = carry + (warp > 0 ? warp_sum[warp - 1] : 0) + x - v;
    if (i < n_blocks) blockcnt[i] = excl;
    __syncthreads();
    if (threadIdx.x == 0) carry += warp_sum[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) *n_flag = carry;
}

__global__ void __launch_bounds__(1024)
k_flag_scan(int32_t* __restrict__ blockcnt, int64_t n_blocks, int32_t* __restrict__ n_flag) {
  flag_scan_body(blockcnt, n_blocks, n_flag, blockIdx, gridDim);
}

// Ordered writes of the marked entries of one unit: each of the unit's words
// (one per thread) places its set bits after the set bits of the words before
// it (an exclusive scan of the words' counts over the block).
// Returns the unit's count (to the last thread of the block).
__device__ __forceinline__ int32_t flag_write_body(const uint32_t* bits, int64_t n_entries,
             int64_t base, int64_t* list,
    const uint3 bid) {
  __shared__ int32_t warp_cnt[kFlagBlock / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t w = (int64_t)bid.x * kFlagWords + tid;
  uint32_t word = tid < kFlagWords ? bits[w] : 0u;
  const int32_t c = __popc(word);
  int32_t x = c;   // inclusive scan within the warp
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_cnt[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int32_t v = warp_cnt[lane];
    int32_t y = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t z = __shfl_up_sync(0xffffffffu, y, d);
      if (lane >= d) y += z;
    }
    warp_cnt[lane] = y - v;   // exclusive over warps
  }
  __syncthreads();
  int64_t off = base + warp_cnt[warp] + (x - c);
  const int32_t total = warp_cnt[warp] + x;
  while (word) {
    const int b = __ffs(word) - 1;
    word &= word - 1;
    const int64_t e = w * 32 + b;
    if (e < n_entries && off < n_entries) list[off] = e;   // the list holds at most n_entries
    ++off;
  }
  return total;
}

// The whole compaction in one launch for short bitmasks: every block counts the
// marked entries before its unit (the words are in L2; at most kFlagOnce units),
// writes its own, and the last one records the total.  Three dependent launches
// took 6.5 us and their gaps for 31 or 122 units alike.
constexpr int64_t kFlagOnce = 128;
__global__ void __launch_bounds__(kFlagBlock)
k_flag_list(const uint32_t* bits, int64_t n_entries, int64_t* list, int32_t* n_flag) {
  stream_order();
  __shared__ int32_t part[kFlagBlock / 32];
  __shared__ int32_t s_base;
  const int tid = threadIdx.x;
  int32_t c = 0;
  const uint4* w = reinterpret_cast<const uint4*>(bits);
  const int32_t n4 = (int32_t)blockIdx.x * (kFlagWords / 4);
#pragma unroll 4
  for (int32_t i = tid; i < n4; i += kFlagBlock) {
    const uint4 v = w[i];
    c += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
  }
  c = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)c);
  if ((tid & 31) == 0) part[tid >> 5] = c;
  __syncthreads();
  if (tid < 32) {
    const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)part[tid]);
    if (tid == 0) s_base = (int32_t)t;
  }
  __syncthreads();
  const int32_t own = flag_write_body(bits, n_entries, s_base, list, blockIdx);
  if (blockIdx.x + 1 == gridDim.x && tid == kFlagBlock - 1) *n_flag = s_base + own;
}

__global__ void __launch_bounds__(kFlagBlock)
k_flag_write(const uint32_t* __restrict__ bits, int64_t n_entries,
             const int32_t* __restrict__ blockoff, int64_t* __restrict__ list) {
  flag_write_body(bits, n_entries, blockoff[blockIdx.x], list, blockIdx);
}

// 2F of a cell from its seven float-float sums (Eq. F_FaFb times two): A, B, C
// and the four data sums of a template.
// D = A B - C^2 and the numerator B |Fa|^2 + A |Fb|^2 - 2 C Re(Fa Fb*) are
// formed in float-float, so their cancellations cost ~2^-46 A B / D of
// relative accuracy (< 1e-6 at the A B / D ~ 1e7 of the worst cells), then
// divided in FP32.
__device__ __forceinline__ float fix_two_f(const FF* a, FF D, const FF* s) {
  const FF fa2 = ff_add(ff_mul(s[0], s[0]), ff_mul(s[1], s[1]));
  const FF fb2 = ff_add(ff_mul(s[2], s[2]), ff_mul(s[3], s[3]));
  const FF fab = ff_add(ff_mul(s[0], s[2]), ff_mul(s[1], s[3]));
  const FF c2 = {2.0f * a[2].h, 2.0f * a[2].l};
  const FF num = ff_sub(ff_add(ff_mul(a[1], fa2), ff_mul(a[0], fb2)), ff_mul(c2, fab));
  return 2.0f * (num.h / D.h);
}

// Float-float recomputation of listed entries.  Entry = cell (shared antenna:
// every template) or template * cells + cell (per-template antenna: that
// template).  Slot b (fix_slot_range) for the templates [y G, y G + G): one
// thread per entry sums its own window (the windows of ill-conditioned cells
// are a few SFTs long), the weights and the antenna sums once for the G
// templates, then a fixed-order block reduction per template.  The list is
// sorted by cell, so neighbouring threads read neighbouring atoms; one thread
// per template and a block per entry read a line per lane instead (590 us of the
// 1024-template exponential workload, 890 us of the rectangular one).
template <int G>
__device__ __forceinline__ void fixup_cells_body(const int64_t* list, int64_t n,
        int32_t shared_antenna,
        const int32_t* __restrict__ rel_t, const int64_t* __restrict__ t_base, int32_t n_sft,
        const fmap_grid& g, const int64_t* __restrict__ ax, const float2* __restrict__ wtab, int32_t n_tab, const int32_t* __restrict__ i0tab, const int32_t* __restrict__ jend,
        const float* __restrict__ antenna, const float* __restrict__ fafb, int32_t n_templates,
        float* __restrict__ map, Partial* __restrict__ parts, int64_t stride, int64_t slot0,
        Coef* __restrict__ coef, const TauTab* __restrict__ tauc, int32_t b, int32_t y) {
  __shared__ Partial scratch[kFixThreads / 32];
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  int64_t lo, hi;
  fix_slot_range(b, n, &lo, &hi);
  const int32_t tq0 = y * G, n_t = min(G, n_templates - tq0);
  const int64_t tb = n_sft > 0 ? *t_base : 0;
  const float* ant = antenna + (int64_t)(shared_antenna ? 0 : tq0) * 3 * n_sft;
  const float* x = fafb + (int64_t)tq0 * 4 * n_sft;
  Partial acc[G];
#pragma unroll
  for (int q = 0; q < G; ++q) acc[q] = partial_empty();
  for (int64_t k = lo + threadIdx.x; k < hi; k += kFixThreads) {
    const int64_t entry = list[k];
    const int64_t cell = shared_antenna ? entry : entry - (int64_t)tq0 * cells;
    if (cell < 0 || cell >= cells) continue;   // (another template's)
    const int32_t m = (int32_t)cell / g.n_tau, nn = (int32_t)cell - m * g.n_tau;   // (cells < 2^31)
    const int32_t i0 = i0tab[m], j = jend[cell];
    const int64_t t0rel = grid_t0(g, ax, m) - tb;
    const int64_t tau = grid_tau(g, ax, nn);
    // Exponential weights along the window as products of per-gap decays,
    // the first one being the decay from t0 to the first atom: for gaps of
    // k < kPowTab whole SFTs the tau's float-float powers of the one-SFT
    // decay (~2^-48), an FP64 exp split into a float pair for other gaps;
    // relative error ~(j - i0) 2^-47.
    const bool ex = g.window == FMAP_EXP;
    const bool tb_win = g.window == FMAP_TABLE;
    const double su = tb_win ? tab_scale(n_tab, exp_cut8_of(g), tau) : 0.0;
    const TauTab* tc = ex && tauc ? tauc + nn : nullptr;
    auto decay = [&](int64_t gap) -> FF {   // (0 <= gap < 2^31 inside a window)
      const uint32_t k = (uint32_t)gap / (uint32_t)g.t_sft;
      if (tc && k < (uint32_t)kPowTab && (int64_t)k * g.t_sft == gap) {
        const float2 v = tc->pw[0][k];
        return FF{v.x, v.y};
      }
      return ff_of(exp(-(double)gap * (tc ? tc->inv_tau : 1.0 / (double)tau)));
    };
    FF sa[3], sx[G][4];
#pragma unroll
    for (int q = 0; q < 3; ++q) sa[q] = FF{0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < G; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) sx[q][c] = FF{0.0f, 0.0f};
    FF w{1.0f, 0.0f};
    if (ex && j > i0) w = decay((int64_t)rel_t[i0] - t0rel);
    for (int32_t a = i0; a < j; ++a) {
      if (ex && a > i0) w = ff_mul(w, decay(rel_t[a] - rel_t[a - 1]));
      if (tb_win) w = ff_of(tab_weight64((double)((int64_t)rel_t[a] - t0rel) * su, wtab, n_tab));
      const FF w2 = ff_mul(w, w);
#pragma unroll
      for (int c = 0; c < 3; ++c) ff_acc(sa[c], w2, ant[(int64_t)c * n_sft + a]);
#pragma unroll
      for (int q = 0; q < G; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c)   // (missing templates repeat the last)
          ff_acc(sx[q][c], w, x[(int64_t)(4 * min(q, n_t - 1) + c) * n_sft + a]);
    }
    // (at least two atoms and D > 0: the sign of a normalised pair is the sign
    // of its high part)
    const FF D = ff_sub(ff_mul(sa[0], sa[1]), ff_mul(sa[2], sa[2]));
    const bool ok = j - i0 >= 2 && D.h > 0.0f;
    // the validity decision, recorded once per entry
    if (coef && (!shared_antenna || y == 0)) coef[entry].valid = ok ? 3.0f : 0.0f;
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const float v = ok ? fix_two_f(sa, D, sx[q]) : 0.0f;
      if (map && q < n_t) map[(int64_t)(tq0 + q) * cells + cell] = v;
      partial_add(acc[q], v, (int32_t)cell, ok);
    }
  }
#pragma unroll
  for (int q = 0; q < G; ++q) {
    const Partial r = partial_block_reduce<kFixThreads / 32>(acc[q], scratch);
    if (threadIdx.x == 0 && q < n_t) parts[(int64_t)(tq0 + q) * stride + slot0 + b] = r;
  }
}

// Templates per thread: four where there are as many and they share their
// antenna rows.
static int fixup_group(int32_t n_templates, bool shared) { return shared && n_templates >= 4 ? 4 : 1; }
int64_t fixup_blocks_y(int32_t n_templates, bool shared) {
  const int g = fixup_group(n_templates, shared);
  return (n_templates + g - 1) / g;
}

// (The read-only inputs, i0tab, jend, rel_t, t_base, tauc and the atoms, are written
// ahead of the ordinary launch that the chain follows: see stream_order.)
template <int G>
__global__ void __launch_bounds__(kFixThreads)
k_fixup(const int64_t* list, const int32_t* n_flag,
        int32_t shared_antenna, const int32_t* __restrict__ rel_t,
        const int64_t* __restrict__ t_base, int32_t n_sft, const fmap_grid g, const int64_t* __restrict__ ax, const float2* __restrict__ wtab, int32_t n_tab,
        const int32_t* __restrict__ i0tab, const int32_t* __restrict__ jend,
        const float* __restrict__ antenna, const float* __restrict__ fafb,
        int32_t n_templates, float* __restrict__ map, Partial* __restrict__ parts,
        int64_t stride, int64_t slot0, Coef* __restrict__ coef,
        const TauTab* __restrict__ tauc, uint32_t* level) {
  stream_order();
  // (the data's range of levels, read by the sweeps of this call, starts anew)
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kLevelWords) level[threadIdx.x] = 0u;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  const int64_t n = min((int64_t)*n_flag, shared_antenna ? cells : cells * n_templates);
  const int32_t used = fix_slots_used(n);
  for (int32_t b = blockIdx.x; b < used; b += gridDim.x)
    fixup_cells_body<G>(list, n, shared_antenna, rel_t, t_base, n_sft, g, ax, wtab, n_tab, i0tab, jend,
                        antenna, fafb, n_templates, map, parts, stride, slot0, coef, tauc, b, blockIdx.y);
}

cudaError_t launch_flag_and_fixup(fmap_plan_s* p, const fmap_atoms* a, float* d_2F,
                                  cudaStream_t s) {
  const int64_t cells = (int64_t)p->grid.n_t0 * p->grid.n_tau;
  const int64_t n_ant = a->shared_antenna ? 1 : p->n_templates;
  const int64_t n_entries = cells * n_ant;
  if (n_entries == 0 || p->n_templates == 0) return cudaSuccess;
  const int64_t n_blocks = (n_entries + kFlagUnit - 1) / kFlagUnit;
  if (n_blocks <= kFlagOnce) {
    launch_after(p, k_flag_list, (unsigned)n_blocks, kFlagBlock, s, p->ws.flag_bits, n_entries,
                 p->ws.flag_list, p->ws.n_flag);
    p->launches += 1;
  } else {
    k_flag_count<<<(unsigned)n_blocks, kFlagBlock, 0, s>>>(p->ws.flag_bits, n_entries, p->ws.flag_blocks);
    k_flag_scan<<<1, 1024, 0, s>>>(p->ws.flag_blocks, n_blocks, p->ws.n_flag);
    k_flag_write<<<(unsigned)n_blocks, kFlagBlock, 0, s>>>(p->ws.flag_bits, n_entries, p->ws.flag_blocks,
                                                           p->ws.flag_list);
    p->launches += 3;
  }
  const bool sh = a->shared_antenna != 0;
  const int64_t y = fixup_blocks_y(p->n_templates, sh);
  // (few template groups: every slot at once; many: a few slots at a time)
  const dim3 grid((unsigned)(y <= 16 ? kFixSlots : kFixBlocks), (unsigned)y);
  auto run = [&](auto kern) {
    launch_after(p, kern, grid, kFixThreads, s, p->ws.flag_list, p->ws.n_flag, a->shared_antenna, p->ws.rel_t,
                                      p->ws.t_base, p->n_sft, p->grid, plan_axes(p), p->ws.wtab,
                                      p->n_tab, p->ws.i0, p->ws.jend, a->antenna, a->fafb,
                                      p->n_templates, d_2F, p->ws.partials, p->part_stride,
                                      p->n_tiles, p->ws.coef,
                                      p->grid.window == FMAP_EXP ? p->ws.tauc : nullptr, p->ws.level);
  };
  fixup_group(p->n_templates, sh) == 4 ? run(k_fixup<4>) : run(k_fixup<1>);
  p->launches += 1;
  return cudaGetLastError();
}


// ---- persistent multi-instance dispatchers (uneven batches) ----
__global__ void __launch_bounds__(kFlagBlock) kb_flag_count(const BItem* __restrict__ items,
                                                            BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    flag_count_body(it.flag_bits, it.flag_entries, it.flag_blocks, make_uint3((unsigned)k, 0, 0),
                    dim3(1));
  });
}
__global__ void __launch_bounds__(1024) kb_flag_scan(const BItem* __restrict__ items, BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t) {
    flag_scan_body(it.flag_blocks, (it.flag_entries + kFlagUnit - 1) / kFlagUnit, it.n_flag,
                   make_uint3(0, 0, 0), dim3(1));
  });
}
__global__ void __launch_bounds__(kFlagBlock) kb_flag_write(const BItem* __restrict__ items,
                                                            BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    flag_write_body(it.flag_bits, it.flag_entries, it.flag_blocks[k], it.flag_list,
                    make_uint3((unsigned)k, 0, 0));
  });
}
__global__ void __launch_bounds__(kFixThreads, 4) kb_fixup(const BItem* __restrict__ items,
                                                        BUnits u) {
  // unit k: slots sg, sg + kFixUnits, ... of template group y
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int64_t n = min((int64_t)*it.n_flag, it.shared ? it.cells : it.cells * it.T);
    const int32_t sg = (int32_t)(k % kFixUnits), y = (int32_t)(k / kFixUnits);
    const int32_t used = fix_slots_used(n);
    for (int32_t b = sg; b < used; b += kFixUnits) {
      if (it.shared && it.T >= 4)
        fixup_cells_body<4>(it.flag_list, n, it.shared, it.rel_t, it.t_base, it.n_sft, it.g, it.ax,
                            nullptr, 0, it.i0, it.jend, it.antenna, it.fafb, it.T, it.map,
                            it.partials, it.part_stride, it.n_tiles, it.coef,
                            it.g.window == FMAP_EXP ? it.tauc : nullptr, b, y);
      else
        fixup_cells_body<1>(it.flag_list, n, it.shared, it.rel_t, it.t_base, it.n_sft, it.g, it.ax,
                            nullptr, 0, it.i0, it.jend, it.antenna, it.fafb, it.T, it.map,
                            it.partials, it.part_stride, it.n_tiles, it.coef,
                            it.g.window == FMAP_EXP ? it.tauc : nullptr, b, y);
    }
  });
}
const void* batch_kernel_fixup(int phase) {
  switch (phase) {
    case BP_FLAG_COUNT: return (const void*)kb_flag_count;
    case BP_FLAG_SCAN: return (const void*)kb_flag_scan;
    case BP_FLAG_WRITE: return (const void*)kb_flag_write;
    case BP_FIXUP: return (const void*)kb_fixup;
  }
  return nullptr;
}

}  // namespace fmap
