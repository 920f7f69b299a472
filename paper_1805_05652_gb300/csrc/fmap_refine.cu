// Top-cell refinement of the per-template reductions.
//
// The detection statistic of a template is its maximum 2F and the cell that
// holds it, and e^F is the odds of a transient in that cell (Sec. 2, Eq.
// F_OSG), so the marginalised Bayes factor is dominated by the cells nearest
// the maximum.  After a compute call has written its fast map, reduced it
// (max, argmax, exp-sum, count) and recomputed the ill-conditioned cells,
// this stage, per template:
//   1. histograms the valid cells whose fast 2F lies within kRefWindow of the
//      fast maximum M (kRefBins bins, bin 0 at the maximum) -- reading only
//      the tiles whose fast maximum (from the reduction partials) can bound
//      one of the cells the cut will take, so the cost does not grow with
//      the map;
//   2. cuts the histogram after the last bin that keeps the cell count within
//      the plan's cap (or after the top bin, when it alone holds more, up to
//      kRefMaxCells), and collects those cells (in no fixed order: every
//      later reduction over them is order-independent -- integer sums of
//      fixed-point terms and a minimum of cell indices): from the cells the
//      histogram pass kept (those in bins up to the tile pass's bound, at
//      most kRefCandCap per template), else by a second scan of the tiles;
//   3. recomputes each collected cell from its atoms by the plain
//      definition: the windowed sums of Eq. (winrect) / (winexp) with w on
//      Fa, Fb and w^2 on A, B, C (in float-float, ~2^-44 relative), then
//      D = AB - C^2 and 2F of Eq. (F_FaFb) in FP64; the refined value
//      replaces the fast one in the map;
//   4. rebuilds the summary: max2F and the argmax (lowest index on FP64
//      ties) from the FP64 values, and the exp-sum with the collected cells'
//      fast terms replaced by their FP64 terms,
//        S' = e^{(M - M')/2} (S - sum_k e^{(f_k - M)/2}) + sum_k e^{(v_k - M')/2},
//      logB = M'/2 + ln S' - ln N' + c.
// Four launches: k_ref_head reduces the template's partials and lists the tiles,
// k_ref_scan histograms their cells, its last block of a template cutting and
// collecting, k_ref_collect does that for the templates whose kept cells
// overflowed, k_ref_cells recomputes, its last block of a template rebuilding the
// summary.  (As seven launches -- two reductions, tiles, histogram, collection,
// cells, summary -- most of a small map's call was their latencies.)
// Every cell outside the cut had a fast 2F more than the cut's distance d
// below M; when d exceeds twice the fast path's error bound, no such cell
// can hold the FP64 maximum, and the summary says so (ARGMAX_EXACT).
#include <math.h>

#include <algorithm>

#include "fmap_device.cuh"

namespace fmap {

constexpr int kRefThreads = 256;
constexpr int kScanShare = 256;   // cells of a listed tile per scanning warp

int32_t refine_cells_of(const fmap_plan_s* p) {
  if (p->refine_cells == 0 || !p->ws.tstat) return 0;
  if (p->refine_cells > 0) return std::min(p->refine_cells, kRefMaxCells);
  return p->precision == FMAP_FP64 ? 64 : 512;
}

// Relative error bound (floor 1) of a plan's fast 2F.
static double fast_tol(const fmap_plan_s* p) { return p->precision == FMAP_FP64 ? 1e-5 : 1e-3; }

// Coef.valid of cell c for template j: 1 summed by the main kernel, 3
// recomputed by the fix-up (and summed in a fix-up slot), else invalid.
__device__ __forceinline__ float ref_valid_of(const Coef* coef, int32_t shared,
                                              int64_t cells, int32_t j, int64_t c) {
  return coef[shared ? c : (int64_t)j * cells + c].valid;
}

// Bin of a fast value v against the template's maximum M: floor((M - v)
// kRefBins / kRefWindow), -1 outside the window (or not a number).
__device__ __forceinline__ int ref_bin_of(float v, float M) {
  const float d = (M - v) * ((float)kRefBins / kRefWindow);
  if (!(d < (float)kRefBins)) return -1;
  return d > 0.0f ? (int)d : 0;
}

// First bin whose cumulative count reaches `want` (kRefBins if none), by one
// warp (all lanes get it); h in shared memory.
__device__ __forceinline__ int32_t ref_first_bin(const int32_t* h, int32_t want, int lane) {
  constexpr int P = kRefBins / 32;
  int32_t own = 0;
#pragma unroll
  for (int k = 0; k < P; ++k) own += h[lane * P + k];
  int32_t cum = own;   // inclusive over lanes
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, cum, d);
    if (lane >= d) cum += y;
  }
  const unsigned reach = __ballot_sync(0xffffffffu, cum >= want);
  int32_t at = kRefBins;
  if (reach && lane == __ffs(reach) - 1) {
    int32_t c = cum - own;
    at = lane * P;
#pragma unroll
    for (int k = 0; k < P; ++k) {
      c += h[lane * P + k];
      if (c < want) ++at;   // (the lane's total reaches it: at stays below the next lane's)
    }
  }
  return (int32_t)__reduce_min_sync(0xffffffffu, (unsigned)at);
}

// The last histogram bin whose cumulative count stays within the cap, at
// most bt (the last bin whose cells all lie in scanned tiles).  When the top
// bin alone holds more than the cap (a maximum shared by many cells within
// 1/16 of 2F, e.g. windows truncated at the data's end), the top bin as a
// whole while it fits the candidate buffer; else -1 (no refinement).
__device__ __forceinline__ int32_t ref_cut_of(const int32_t* h, int32_t cap, int32_t bt, int lane) {
  const int32_t b = min(ref_first_bin(h, cap + 1, lane) - 1, min(bt, kRefBins - 1));
  return b < 0 && h[0] <= kRefMaxCells ? 0 : b;
}

// Sums over a block's warps: every lane of warp 0 gets the total.
template <int NW>
__device__ __forceinline__ double ref_block_sum(double v, double* sh, int lane, int warp) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  v = lane < NW ? sh[lane] : 0.0;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Pass 1 (one block per template): the template's reduction (maximum and count,
// then the exp-sum relative to it and the lowest index at it; the order of the
// additions is fixed, FP64 over the tiles' FP32 sums) into its statistics, and
// which tiles to scan.  The partials give
// every tile's fast maximum (a main tile's over the cells the main kernel
// summed, a fix-up slot's over its recomputed cells: disjoint sets); with bt
// the first bin in which the count of tiles (by their maxima) reaches the
// cap, at least cap distinct cells lie in bins <= bt (those maxima), so the
// cut never passes bt, and every cell in a bin <= bt lies in a tile whose
// maximum is in a bin <= bt: those tiles are listed for the cell passes,
// and bt is kept in cut[j].
constexpr int kTileThreads = 1024;
constexpr int kTileCache = 8;   // slots per thread whose maxima stay in registers

struct HeadArgs {
  const Partial* parts;
  int64_t stride, n_tiles, fix0, entries;
  const int32_t* n_flag;
  int32_t cap;
  TStat* st;
  int32_t* hist;
  int32_t* ref_n;
  int32_t* ref_ncand;
  int32_t* ref_ntile;
  int32_t* ref_tile;
  int32_t* cut;
};

__global__ void __launch_bounds__(kTileThreads) k_ref_head(const HeadArgs A) {
  stream_order();
  constexpr int NW = kTileThreads / 32;
  __shared__ int32_t h[kRefBins];
  __shared__ unsigned s_mu[NW], s_cnt[NW], s_arg[NW];
  __shared__ double s_sum[NW];
  __shared__ int32_t s_bt, s_n;
  const int32_t j = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < kRefBins) {
    h[tid] = 0;
    A.hist[(int64_t)j * kRefBins + tid] = 0;
  }
  if (tid == 0) {
    s_n = 0;
    A.ref_n[j] = 0;
    A.ref_ncand[j] = 0;
  }
  const int64_t total = A.n_tiles + fix_slots_used(min((int64_t)*A.n_flag, A.entries));
  const Partial* pp = A.parts + (int64_t)j * A.stride;
  auto slot = [&](int64_t k) {
    return *reinterpret_cast<const float4*>(pp + (k < A.n_tiles ? k : A.fix0 + (k - A.n_tiles)));
  };
  auto top_of = [](const float4& q) { return __float_as_int(q.w) > 0 ? q.x : -1.0f; };
  // maximum and count (2F >= 0: the bit patterns order like the values)
  float tops[kTileCache];
  unsigned mu = 0u, cnt = 0u;
  auto see = [&](const float4& q) {
    const int32_t nv = __float_as_int(q.w);
    if (nv > 0) {
      mu = max(mu, __float_as_uint(q.x) + 1u);
      cnt += (unsigned)nv;
    }
  };
#pragma unroll
  for (int i = 0; i < kTileCache; ++i) {
    const int64_t k = tid + (int64_t)i * kTileThreads;
    const float4 q = k < total ? slot(k) : make_float4(-1.f, 0.f, 0.f, 0.f);
    tops[i] = top_of(q);
    see(q);
  }
#pragma unroll 4
  for (int64_t k = tid + (int64_t)kTileCache * kTileThreads; k < total; k += kTileThreads) see(slot(k));
  mu = __reduce_max_sync(0xffffffffu, mu);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) {
    s_mu[warp] = mu;
    s_cnt[warp] = cnt;
  }
  __syncthreads();
  mu = __reduce_max_sync(0xffffffffu, s_mu[lane]);
  cnt = __reduce_add_sync(0xffffffffu, s_cnt[lane]);
  const float M = mu ? __uint_as_float(mu - 1u) : -1.0f;
  // exp-sum: rescale factor exp((max2F - M) / 2) <= 1 in FP32 (relative error
  // ~1e-7, the order of the FP32 tile sums themselves), accumulated in FP64;
  // factors below 2^-126 flush to 0
  double sum = 0.0;
  unsigned arg = (unsigned)kNoArg;
  if (mu) {
#pragma unroll 4
    for (int64_t k = tid; k < total; k += kTileThreads) {
      const float4 q = slot(k);
      if (__float_as_int(q.w) <= 0) continue;
      float f;
      asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((q.x - M) * 0.72134752044448170368f));
      sum += (double)q.z * (double)f;
      if (q.x == M) arg = min(arg, (unsigned)__float_as_int(q.y));
    }
  }
  arg = __reduce_min_sync(0xffffffffu, arg);
  if (lane == 0) s_arg[warp] = arg;
  sum = ref_block_sum<NW>(sum, s_sum, lane, warp);   // (a barrier: s_arg is there too)
  if (tid < 32) {
    arg = __reduce_min_sync(0xffffffffu, s_arg[lane]);
    if (tid == 0) A.st[j] = TStat{sum, M, (int32_t)arg, (long long)cnt, {0, 0}};
  }
  // tiles by the bins of their maxima: one shared-memory atomic per distinct bin
  // among a warp's lanes
  auto bin_of = [&](float top) { return top >= 0.0f ? ref_bin_of(top, M) : -1; };
  auto count = [&](int b, unsigned mask) {
    const unsigned peers = __match_any_sync(mask, b);
    if (b >= 0 && lane == __ffs(peers) - 1) atomicAdd(&h[b], __popc(peers));
  };
#pragma unroll
  for (int i = 0; i < kTileCache; ++i) count(bin_of(tops[i]), 0xffffffffu);
  for (int64_t k = tid + (int64_t)kTileCache * kTileThreads; k < total; k += kTileThreads)
    count(bin_of(top_of(slot(k))), __activemask());
  __syncthreads();
  if (warp == 0) {
    const int32_t f = ref_first_bin(h, A.cap, lane);
    if (lane == 0) s_bt = min(f, kRefBins - 1);
  }
  __syncthreads();
  const int32_t bt = s_bt;
  int32_t* list = A.ref_tile + (int64_t)j * kRefMaxTiles;
  auto put = [&](int64_t k, int b, unsigned mask) {
    const bool take = b >= 0 && b <= bt;
    const unsigned sel = __ballot_sync(mask, take);
    if (!sel) return;
    const int leader = __ffs(sel) - 1;
    int32_t base = 0;
    if (lane == leader) base = atomicAdd(&s_n, __popc(sel));
    base = __shfl_sync(mask, base, leader);
    const int32_t at = base + __popc(sel & ((1u << lane) - 1u));
    if (take && at < kRefMaxTiles) list[at] = (int32_t)k;
  };
#pragma unroll
  for (int i = 0; i < kTileCache; ++i)
    put(tid + (int64_t)i * kTileThreads, bin_of(tops[i]), 0xffffffffu);
  for (int64_t k = tid + (int64_t)kTileCache * kTileThreads; k < total; k += kTileThreads)
    put(k, bin_of(top_of(slot(k))), __activemask());
  __syncthreads();
  if (tid == 0) {
    A.ref_ntile[j] = s_n;   // (more than kRefMaxTiles: truncated)
    A.cut[j] = bt;
  }
}

// Counts a block of a template's pass as done; true (to all its threads) for
// the last one, which then sees what the others wrote.
__device__ __forceinline__ bool ref_last_block(int32_t* done, int32_t n_blocks) {
  __shared__ int32_t s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1) == n_blocks - 1;
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  return true;
}

struct ScanArgs {
  const float* map;
  const Coef* coef;
  int32_t shared;
  int32_t n_t0, n_tau;
  int64_t cells;
  TileGeom geo;
  int64_t n_tiles;
  int32_t parts;   // warps per listed tile (each takes one share of its cells)
  const int64_t* flag_list;
  const int32_t* n_flag;
  int32_t n_templates;
  TStat* st;
  const int32_t* ref_ntile;
  const int32_t* ref_tile;
  int32_t* hist;
  int32_t cap;
  int32_t* cut;   // [T] bt of the tile pass, then the cut
  int32_t* ref_n;
  int32_t* ref_cell;
  int32_t* ref_ncand;
  int32_t* ref_cand;
};

// Calls f(cell, bin, take), all 32 lanes of the warp together, for the cells of
// share `part` (of A.parts) of listed tile k: a main tile by its geometry, a fix-up
// slot by its share of the fix-up list.  take: the cell lies in a bin up to `last`
// and the tile's partial summed it (a main tile's cells of Coef.valid 1, a fix-up
// slot's of 3), so that no cell is taken twice.  Steps that take none are left
// out: only the few cells near the maximum cost more than the load of their
// value, four steps of which are in flight at once.  (With every cell's
// coefficient loaded, 64-bit divisions and a match over the lanes' bins, a share of
// 256 cells took eight dependent round trips: 25 us of a 1000 x 1000 band of 16
// templates.)
template <typename F>
__device__ __forceinline__ void ref_tile_cells(const ScanArgs& A, int32_t j, int64_t k,
                                               int32_t part, float M, int32_t last, int lane,
                                               F f) {
  const float* mp = A.map + (int64_t)j * A.cells;
  if (k < A.n_tiles) {
    constexpr int U = 4;
    const TileGeom& g = A.geo;
    const int32_t kk = (int32_t)k;   // (tiles: fewer than cells, < 2^31)
    const int32_t tr = g.col_major ? kk % g.ntr : kk / g.ntc;
    const int32_t tc = g.col_major ? kk / g.ntr : kk % g.ntc;
    const int32_t r0 = tr * g.R, c0 = tc * g.C;
    const uint32_t rows = (uint32_t)min(g.R, A.n_t0 - r0), cols = (uint32_t)min(g.C, A.n_tau - c0);
    const uint32_t n = rows * cols, per = (n + (uint32_t)A.parts - 1u) / (uint32_t)A.parts;
    const uint32_t lo = (uint32_t)min((uint64_t)part * per, (uint64_t)n), hi = min(n, lo + per);
    const uint32_t dr = 32u / cols, dc = 32u - dr * cols;   // a step of 32 cells
    uint32_t r = (lo + lane) / cols, cc = lo + lane - r * cols;
    for (uint32_t q0 = lo; q0 < hi; q0 += 32u * U) {
      int32_t c[U];
      float v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        c[u] = (r0 + (int32_t)r) * A.n_tau + c0 + (int32_t)cc;
        v[u] = q0 + 32u * u + lane < hi ? mp[c[u]] : -INFINITY;
        r += dr;
        cc += dc;
        if (cc >= cols) {
          cc -= cols;
          ++r;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int b = ref_bin_of(v[u], M);
        bool take = b >= 0 && b <= last;
        if (!__any_sync(0xffffffffu, take)) continue;
        take = take && ref_valid_of(A.coef, A.shared, A.cells, j, c[u]) == 1.0f;
        f(c[u], b, take);
      }
    }
  } else {
    const int64_t cap = A.shared ? A.cells : A.cells * A.n_templates;
    const int64_t n = min((int64_t)*A.n_flag, cap);
    int64_t lo, hi;
    fix_slot_range((int32_t)(k - A.n_tiles), n, &lo, &hi);
    const int64_t m = hi - lo;
    const int64_t end = lo + m * (part + 1) / A.parts;
    for (int64_t e0 = lo + m * part / A.parts; e0 < end; e0 += 32) {
      bool take = e0 + lane < end;
      int64_t c = take ? A.flag_list[e0 + lane] : 0;
      if (!A.shared) c -= (int64_t)j * A.cells;   // (another template's entry: out of range)
      take = take && c >= 0 && c < A.cells;
      const int b = take ? ref_bin_of(mp[c], M) : -1;
      take = b >= 0 && b <= last;
      if (!__any_sync(0xffffffffu, take)) continue;
      take = take && ref_valid_of(A.coef, A.shared, A.cells, j, c) == 3.0f;
      f((int32_t)c, b, take);
    }
  }
}

// Calls f as above for the cells of the first nt listed tiles, whose shares go to
// `step` warps.
template <typename F>
__device__ __forceinline__ void ref_scan_cells(const ScanArgs& A, int32_t j, int32_t nt, float M,
                                               int32_t last, int64_t first, int64_t step, int lane,
                                               F f) {
  const uint32_t n = (uint32_t)nt * (uint32_t)A.parts;   // (at most kRefMaxTiles x 1024)
  for (uint32_t it = (uint32_t)first; it < n; it += (uint32_t)step) {
    const uint32_t k = it / (uint32_t)A.parts;
    ref_tile_cells(A, j, A.ref_tile[(int64_t)j * kRefMaxTiles + k],
                   (int32_t)(it - k * (uint32_t)A.parts), M, last, lane, f);
  }
}

// Pass 2 over the listed tiles' cells: the histogram of the bins up to the tile
// pass's bound (cut[j]; the cut never passes it), which also keeps those cells
// while they fit kRefCandCap; then, in the template's last block, the cut and the collection of
// the cells up to it from the kept cells when they fit (the same set: every
// cell the cut takes lies in a bin <= cut[j]), else a flag (done[0] < 0) that
// leaves the collection to a second scan of the tiles, k_ref_collect.  Grid (x, T),
// one warp per share of a tile.  The histogram and the counts were cleared by the
// first pass.
__global__ void __launch_bounds__(kRefThreads) k_ref_scan(const ScanArgs A) {
  stream_order();
  __shared__ int32_t h[kRefBins];
  __shared__ int32_t s_cut, s_n;
  const int32_t j = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NW = kRefThreads / 32;
  static_assert(kRefThreads == kRefBins, "one bin per thread");
  const TStat s = A.st[j];
  const int32_t keep = A.cut[j];   // bins the histogram pass keeps
  const int32_t nt = s.N > 0 ? min(A.ref_ntile[j], kRefMaxTiles) : 0;
  // the blocks that have a share (the first one always takes part)
  const int32_t n_blk = (int32_t)min(gridDim.x, max(1u, ((uint32_t)nt * (uint32_t)A.parts + NW - 1u) / NW));
  if ((int32_t)blockIdx.x >= n_blk) return;
  h[tid] = 0;
  __syncthreads();
  const float* mp = A.map + (int64_t)j * A.cells;
  int32_t* cand = A.ref_cand + (int64_t)j * kRefCandCap;
  ref_scan_cells(A, j, nt, s.M, keep, blockIdx.x * NW + warp, (int64_t)gridDim.x * NW, lane,
                 [&](int32_t c, int b, bool take) {
    if (take) atomicAdd(&h[b], 1);
    // one global atomic per warp step
    const unsigned sel = __ballot_sync(0xffffffffu, take);
    if (sel) {
      const int leader = __ffs(sel) - 1;
      int32_t base = 0;
      if (lane == leader) base = atomicAdd(A.ref_ncand + j, __popc(sel));
      base = __shfl_sync(0xffffffffu, base, leader);
      const int32_t at = base + __popc(sel & ((1u << lane) - 1u));
      if (take && at < kRefCandCap) cand[at] = c;
    }
  });
  __syncthreads();
  if (h[tid]) atomicAdd(A.hist + (int64_t)j * kRefBins + tid, h[tid]);
  if (!ref_last_block(&A.st[j].done[0], n_blk)) return;
  h[tid] = __ldcg(A.hist + (int64_t)j * kRefBins + tid);
  if (tid == 0) s_n = 0;
  __syncthreads();
  if (warp == 0) {
    const int32_t b = ref_cut_of(h, A.cap, keep, lane);
    if (lane == 0) s_cut = A.cut[j] = b;
  }
  __syncthreads();
  const int32_t last = s_cut;
  if (nt == 0 || last < 0) return;   // (ref_n stays 0)
  const int32_t n_kept = __ldcg(A.ref_ncand + j);
  if (n_kept > kRefCandCap) {
    if (tid == 0) A.st[j].done[0] = -1;
    return;
  }
  for (int32_t k = tid; k < n_kept; k += kRefThreads) {
    const int32_t c = __ldcg(cand + k);
    const int b = ref_bin_of(mp[c], s.M);
    if (b < 0 || b > last) continue;
    const int32_t slot = atomicAdd(&s_n, 1);
    if (slot < kRefMaxCells) A.ref_cell[(int64_t)j * kRefMaxCells + slot] = c;
  }
  __syncthreads();
  if (tid == 0) A.ref_n[j] = s_n;
}

// The second scan of the tiles of the templates whose kept cells overflowed
// (a strong signal's tiles hold many cells near the maximum).  Every block of
// the others ends at once.
__global__ void __launch_bounds__(kRefThreads) k_ref_collect(const ScanArgs A) {
  stream_order();
  const int32_t j = blockIdx.y;
  const TStat s = A.st[j];
  if (s.done[0] >= 0) return;
  constexpr int NW = kRefThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t last = A.cut[j], nt = min(A.ref_ntile[j], kRefMaxTiles);
  ref_scan_cells(A, j, nt, s.M, last, blockIdx.x * NW + warp, (int64_t)gridDim.x * NW, lane,
                 [&](int32_t c, int, bool take) {
    if (!take) return;
    const int32_t slot = atomicAdd(A.ref_n + j, 1);
    if (slot < kRefMaxCells) A.ref_cell[(int64_t)j * kRefMaxCells + slot] = c;
  });
}

struct RefArgs {
  const int32_t* rel_t;
  const int64_t* t_base;
  int32_t n_sft;
  fmap_grid g;
  const int64_t* ax;
  const float2* wtab;
  int32_t n_tab;
  const float4* perm_ant;   // exponential windows: the sweeps' copies of the atoms
  const float4* perm_x;     // (or null: the caller's rows)
  const int32_t* i0;
  const int32_t* jend;
  const float* antenna;
  const float* fafb;
  int32_t shared;
  float* map;
  int64_t cells;
  const int32_t* ref_n;
  const int32_t* ref_cell;
  float* ref_fast;
  double* ref_val;
  // the summaries
  TStat* st;
  const int32_t* cut;
  const int32_t* ref_ntile;
  double log_prior, tol;
  fmap_summary* out;
};

// Pass 3: one warp per collected cell, its atoms summed in float-float arithmetic (a
// value is an unevaluated pair h + l, ~2^-44 relative; GB300 runs FP64 at 1/64 of
// the FP32 rate).  The seven sums meet in a fixed butterfly; D and 2F are formed
// from them in FP64 by one lane.
// Exponential windows: ref_exp_sums.  The others: lane l takes the window's atoms
// i0 + l + 32 q (coalesced loads, a step ahead), added by TwoSum with the errors
// collected in l (Ogita, Rump and Oishi's cascaded form, ~n^2 2^-48 relative for a
// lane's n atoms); a table window evaluates w per atom in float-float and multiplies
// with the products' FMA error, a rectangular one has w = 1.
__device__ __forceinline__ void ref_acc(FF& s, FF w, float x) {
  const float p = __fmul_rn(w.h, x);
  const float e = fmaf(w.l, x, fmaf(w.h, x, -p));
  const FF t = two_sum(s.h, p);
  s.h = t.h;
  s.l += t.l + e;
}

// The butterfly over the lanes' seven sums (every lane gets the totals).
__device__ __forceinline__ void ref_butterfly(FF (&s)[7]) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1)
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      const FF o{__shfl_xor_sync(0xffffffffu, s[q].h, d), __shfl_xor_sync(0xffffffffu, s[q].l, d)};
      s[q] = ff_add(s[q], o);
    }
}

// The seven sums of an exponential window: lane l takes the l-th of 32 contiguous
// runs of its atoms, the first weight from an FP64 exp and the others as products
// of the gaps' decays.  2F of an exponential window does not change with t0 while
// the window holds the same atoms, so that at grid steps below one SFT the maximum
// is often shared by neighbouring cells up to rounding: this order of the
// operations is part of which of them is reported, and is not to be changed.
// Lane k holds the decay of k SFTs (the FP64 exp of that gap: with one for every
// gap of more than one SFT, the FP64 pipe was 66 % busy: 1034 us for 5 x 512
// cells of a year's data with 4 % missing SFTs, about 350 us so); the atoms come from
// the sweeps' copies, a step ahead.
__device__ __forceinline__ void ref_exp_sums(const RefArgs& A, int32_t j, int32_t c, int lane,
                                             FF (&s)[7]) {
  const fmap_grid& g = A.g;
  const int32_t m = c / g.n_tau, nn = c - m * g.n_tau;
  const int32_t i0 = A.i0[m], len = max(0, A.jend[c] - i0);
  const int64_t t0rel = grid_t0(g, A.ax, m) - *A.t_base;
  const double inv_tau = 1.0 / (double)grid_tau(g, A.ax, nn);
  const int64_t n = A.n_sft;
  const float4* ant = A.perm_ant + (A.shared ? 0 : (int64_t)j * n);
  const float4* px = A.perm_x ? A.perm_x + (int64_t)j * n : nullptr;
  const float* x = A.fafb + (int64_t)j * 4 * n;
#pragma unroll
  for (int q = 0; q < 7; ++q) s[q] = FF{0.0f, 0.0f};
  if (len > 0) {   // (the whole warp)
    const int32_t a_lo = i0 + (int32_t)((int64_t)len * lane / 32);
    const int32_t run = i0 + (int32_t)((int64_t)len * (lane + 1) / 32) - a_lo;
    const int32_t last = i0 + len - 1, most = (len + 31) / 32;
    const FF rk = ff_of(exp(-(double)((int64_t)lane * g.t_sft) * inv_tau));
    float4 va, vx;
    auto load = [&](int32_t a) {   // (past the lane's run: unused)
      a = min(a, last);
      va = ant[a];
      vx = px ? px[a] : make_float4(x[a], x[n + a], x[2 * n + a], x[3 * n + a]);
    };
    load(a_lo);
    FF w = ff_of(exp(-(double)((int64_t)A.rel_t[min(a_lo, last)] - t0rel) * inv_tau));
    int32_t k = 0;   // SFTs from the atom before (0: not a gap of the copies' codes)
    for (int32_t i = 0; i < most; ++i) {
      const float4 ua = va, ux = vx;
      if (i + 1 < most) load(a_lo + i + 1);
      FF r{__shfl_sync(0xffffffffu, rk.h, k & 31), __shfl_sync(0xffffffffu, rk.l, k & 31)};
      if (i < run) {
        if (i > 0) {
          if (k <= 0) {
            const int32_t gap = A.rel_t[a_lo + i] - A.rel_t[a_lo + i - 1];
            r = ff_of(exp(-(double)gap * inv_tau));
          }
          w = ff_mul(w, r);
        }
        const FF w2 = ff_mul(w, w);
        ff_acc(s[0], w2, ua.x);
        ff_acc(s[1], w2, ua.y);
        ff_acc(s[2], w2, ua.z);
        ff_acc(s[3], w, ux.x);
        ff_acc(s[4], w, ux.y);
        ff_acc(s[5], w, ux.z);
        ff_acc(s[6], w, ux.w);
        k = __float_as_int(ua.w);
      }
    }
  }
  ref_butterfly(s);
}

// The seven sums of collected cell c of template j (every lane gets them), other
// windows.
__device__ __forceinline__ void ref_cell_sums(const RefArgs& A, int32_t j, int32_t c, int lane,
                                              FF (&s)[7]) {
  const fmap_grid& g = A.g;
  const int32_t m = c / g.n_tau, nn = c - m * g.n_tau;
  const int32_t i0 = A.i0[m], je = A.jend[c];
  const int64_t t0rel = grid_t0(g, A.ax, m) - *A.t_base;
  const int64_t n = A.n_sft;
  const float* ant = A.antenna + (A.shared ? 0 : (int64_t)j * 3 * n);
  const float* x = A.fafb + (int64_t)j * 4 * n;
  const bool tw = g.window == FMAP_TABLE;
  const FF su = ff_of(tw ? tab_scale(A.n_tab, exp_cut8_of(g), grid_tau(g, A.ax, nn)) : 0.0);
#pragma unroll
  for (int q = 0; q < 7; ++q) s[q] = FF{0.0f, 0.0f};
  if (je > i0) {
    FF w{1.0f, 0.0f};
    float v[7];
    int32_t tn;
    auto load = [&](int32_t b) {   // (lanes past the window: its last atom, unused)
      const int32_t a = min(b + lane, je - 1);
      tn = A.rel_t[a];
#pragma unroll
      for (int q = 0; q < 3; ++q) v[q] = ant[q * n + a];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[3 + q] = x[q * n + a];
    };
    load(i0);
    for (int32_t b = i0; b < je; b += 32) {
      float u[7];
#pragma unroll
      for (int q = 0; q < 7; ++q) u[q] = v[q];
      const int32_t t = tn;
      const bool on = b + lane < je;
      if (b + 32 < je) load(b + 32);
      if (tw) w = tab_weight_ff((int32_t)((int64_t)t - t0rel), su, A.wtab, A.n_tab);
      if (on) {
        if (g.window == FMAP_RECT) {
#pragma unroll
          for (int q = 0; q < 7; ++q) {
            const FF y = two_sum(s[q].h, u[q]);
            s[q].h = y.h;
            s[q].l += y.l;
          }
        } else {
          const FF w2 = ff_mul(w, w);
#pragma unroll
          for (int q = 0; q < 3; ++q) ref_acc(s[q], w2, u[q]);
#pragma unroll
          for (int q = 3; q < 7; ++q) ref_acc(s[q], w, u[q]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 7; ++q) s[q] = fast_two_sum(s[q].h, s[q].l);
  ref_butterfly(s);
}

// a b + c d with the second product rounded and the first fused into the sum.
__device__ __forceinline__ double ref_sum2(double a, double b, double c, double d) {
  return __fma_rn(a, b, __dmul_rn(c, d));
}
// 2F of the cell in slot k of template j from its sums, in FP64 (one lane; records
// the fast and the refined value, and writes the latter to the map).  Which products
// are fused is part of which cell of a tie is reported, so the code says it rather
// than the compiler.
__device__ __forceinline__ void ref_cell_end(const RefArgs& A, int32_t j, int32_t k, const FF (&s)[7]) {
  const int64_t slot = (int64_t)j * kRefMaxCells + k;
  const int32_t c = A.ref_cell[slot];
  const int32_t len = A.jend[c] - A.i0[c / A.g.n_tau];
  double v7[7];
#pragma unroll
  for (int q = 0; q < 7; ++q) v7[q] = (double)s[q].h + (double)s[q].l;
  const double Aa = v7[0], Bb = v7[1], Cc = v7[2];
  const double D = __fma_rn(Aa, Bb, -__dmul_rn(Cc, Cc));
  const bool ok = len >= 2 && D > 0.0;
  double v = 0.0;
  if (ok) {
    const double fa2 = ref_sum2(v7[3], v7[3], v7[4], v7[4]);
    const double fb2 = ref_sum2(v7[5], v7[5], v7[6], v7[6]);
    const double fab = ref_sum2(v7[3], v7[5], v7[4], v7[6]);
    v = 2.0 * __fma_rn(-2.0 * Cc, fab, ref_sum2(Bb, fa2, Aa, fb2)) / D;
  }
  float* mp = A.map + (int64_t)j * A.cells + c;
  A.ref_fast[slot] = *mp;
  A.ref_val[slot] = ok ? v : -1.0;
  *mp = (float)v;
}

// Pass 4: a template's last block rebuilds its summary from the fast
// statistics and the collected cells.  Every exp-term is in (0, 1] (relative
// to the fast or the refined maximum, both held by a collected cell) and is
// summed as an integer in 2^-51 units, so the sums do not depend on the
// order in which the cells were collected (<= 4096 terms <= 2^63: no overflow,
// relative error < 1e-12).  Where no cell was collected, or none is valid, the
// fast reduction stands (flags 0).
__device__ __forceinline__ void ref_fast_summary(const RefArgs& A, int32_t j) {
  const TStat s = A.st[j];
  fmap_summary o;
  o.flags = 0;
  o.n_valid = s.N;
  o.max2F = s.N > 0 ? s.M : 0.0f;
  o.m = s.N > 0 ? s.arg / A.g.n_tau : -1;
  o.n = s.N > 0 ? s.arg % A.g.n_tau : -1;
  o.logB = s.N > 0 ? 0.5 * (double)s.M + log(s.S) - log((double)s.N) + A.log_prior : nan("");
  A.out[j] = o;
}
__device__ __forceinline__ void ref_summary(const RefArgs& A, int32_t j, int32_t n) {
  constexpr int NW = kRefThreads / 32;
  __shared__ double s_mx[NW];
  __shared__ unsigned long long s_sub[NW], s_add[NW];
  __shared__ int32_t s_nv[NW], s_arg[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TStat s = A.st[j];
  const int64_t base = (int64_t)j * kRefMaxCells;
  double mx = -1.0;
  for (int32_t k = threadIdx.x; k < n; k += kRefThreads) mx = fmax(mx, __ldcg(A.ref_val + base + k));
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, d));
  if (lane == 0) s_mx[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) mx = fmax(mx, s_mx[w]);
  if (mx < 0.0) {   // no collected cell valid in FP64
    if (threadIdx.x == 0) ref_fast_summary(A, j);
    return;
  }
  constexpr double kFix = 2251799813685248.0;   // 2^51
  unsigned long long sub = 0ull, add = 0ull;
  int32_t nv = 0, arg = 0x7fffffff;
  const double M = (double)s.M;
  for (int32_t k = threadIdx.x; k < n; k += kRefThreads) {
    const double ef = exp(0.5 * fmin((double)__ldcg(A.ref_fast + base + k) - M, 0.0));
    sub += (unsigned long long)__double2ull_rn(ef * kFix);
    const double v = __ldcg(A.ref_val + base + k);
    if (v >= 0.0) {
      add += (unsigned long long)__double2ull_rn(exp(0.5 * (v - mx)) * kFix);
      nv += 1;
      if (v == mx) arg = min(arg, A.ref_cell[base + k]);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    sub += __shfl_xor_sync(0xffffffffu, sub, d);
    add += __shfl_xor_sync(0xffffffffu, add, d);
  }
  nv = __reduce_add_sync(0xffffffffu, nv);
  arg = __reduce_min_sync(0xffffffffu, arg);
  if (lane == 0) {
    s_sub[warp] = sub;
    s_add[warp] = add;
    s_nv[warp] = nv;
    s_arg[warp] = arg;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < NW; ++w) {   // (integer sums: the order does not matter)
    sub += s_sub[w];
    add += s_add[w];
    nv += s_nv[w];
    arg = min(arg, s_arg[w]);
  }
  const double Sp = exp(0.5 * (M - mx)) * fmax(s.S - (double)sub / kFix, 0.0) + (double)add / kFix;
  const long long Np = s.N - n + nv;
  const int32_t b = A.cut[j];
  const double depth = b + 1 >= kRefBins ? (double)kRefWindow
                                         : (double)(b + 1) * (double)kRefWindow / kRefBins;
  fmap_summary o;
  o.max2F = (float)mx;
  o.m = arg / A.g.n_tau;
  o.n = arg % A.g.n_tau;
  const bool complete = A.ref_ntile[j] <= kRefMaxTiles;   // every candidate tile scanned
  o.flags = (int32_t)FMAP_SUMMARY_REFINED |
            (complete && depth > 2.0 * A.tol * fmax(mx, 1.0) ? (int32_t)FMAP_SUMMARY_ARGMAX_EXACT
                                                              : 0);
  o.logB = 0.5 * mx + log(Sp) - log((double)Np) + A.log_prior;
  o.n_valid = Np;
  A.out[j] = o;
}

__global__ void __launch_bounds__(kRefThreads) k_ref_cells(const RefArgs A) {
  stream_order();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t j = blockIdx.y;
  const int32_t n_cand = min(A.ref_n[j], kRefMaxCells);
  const bool ex = A.g.window == FMAP_EXP;
  constexpr int NW = kRefThreads / 32;
  __shared__ FF s_sum[NW][7];
  if (n_cand <= 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ref_fast_summary(A, j);
    return;
  }
  for (int32_t k0 = blockIdx.x * NW; k0 < n_cand; k0 += gridDim.x * NW) {
    if (k0 + warp < n_cand) {
      FF s[7];
      const int32_t c = A.ref_cell[(int64_t)j * kRefMaxCells + k0 + warp];
      if (ex) {
        ref_exp_sums(A, j, c, lane, s);
        if (lane == 0) ref_cell_end(A, j, k0 + warp, s);
      } else {
        ref_cell_sums(A, j, c, lane, s);
#pragma unroll
        for (int q = 0; q < 7; ++q)
          if (lane == q) s_sum[warp][q] = s[q];
      }
    }
    if (ex) continue;   // (the whole block)
    __syncthreads();
    if (warp == 0 && lane < NW && k0 + lane < n_cand) ref_cell_end(A, j, k0 + lane, s_sum[lane]);
    __syncthreads();
  }
  if (ref_last_block(&A.st[j].done[1], gridDim.x)) ref_summary(A, j, n_cand);
}

cudaError_t launch_refine(fmap_plan_s* p, const fmap_atoms* a, float* d_2F,
                          fmap_summary* d_summary, int64_t n_tiles, cudaStream_t s) {
  const int32_t cap = refine_cells_of(p);
  const fmap_grid& g = p->grid;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  const int32_t T = p->n_templates;
  if (cap <= 0 || !d_2F || !d_summary || T == 0 || cells == 0 || p->n_sft == 0)
    return launch_final_reduce(p, n_tiles, a, d_summary, s);
  Workspace& w = p->ws;
  const int32_t sh = a->shared_antenna ? 1 : 0;
  HeadArgs H;
  H.parts = w.partials;
  H.stride = p->part_stride;
  H.n_tiles = n_tiles;
  H.fix0 = p->n_tiles;
  H.entries = cells * (sh ? 1 : T);
  H.n_flag = w.n_flag;
  H.cap = cap;
  H.st = w.tstat;
  H.hist = w.ref_hist;
  H.ref_n = w.ref_n;
  H.ref_ncand = w.ref_ncand;
  H.ref_ntile = w.ref_ntile;
  H.ref_tile = w.ref_tile;
  H.cut = w.ref_bin;
  launch_after(p, k_ref_head, T, kTileThreads, s, H);
  ScanArgs S;
  S.map = d_2F;
  S.coef = w.coef;
  S.shared = sh;
  S.n_t0 = g.n_t0;
  S.n_tau = g.n_tau;
  S.cells = cells;
  S.geo = p->tiles;
  S.n_tiles = n_tiles;
  S.flag_list = w.flag_list;
  S.n_flag = w.n_flag;
  S.n_templates = T;
  S.st = w.tstat;
  S.ref_ntile = w.ref_ntile;
  S.ref_tile = w.ref_tile;
  S.hist = w.ref_hist;
  S.cap = cap;
  S.cut = w.ref_bin;
  S.ref_n = w.ref_n;
  S.ref_cell = w.ref_cell;
  S.ref_ncand = w.ref_ncand;
  S.ref_cand = w.ref_cand;
  // a warp per share of about kScanShare cells of a listed tile (about cap tiles per
  // template), between one and 32 blocks per SM over all templates: a block's own
  // costs (its launch, the histogram, its place in the count) are several shares'.
  // (128 blocks for each of 1024 templates, 2000 x 2000 cells: 357 us, and 60 us of
  // the launch that mostly has nothing to collect; 221 us so.)
  const int64_t tile_cells = (int64_t)S.geo.R * S.geo.C;
  S.parts = (int32_t)std::min<int64_t>(std::max<int64_t>((tile_cells + kScanShare - 1) / kScanShare, 1),
                                       1024);
  const int wpb = kRefThreads / 32;
  const int64_t gx = std::clamp<int64_t>((2 * (int64_t)cap * S.parts + wpb - 1) / wpb,
                                         ((int64_t)p->n_sm + T - 1) / T,
                                         ((int64_t)p->n_sm * 32 + T - 1) / T);
  const dim3 grid((unsigned)gx, (unsigned)T);
  launch_after(p, k_ref_scan, grid, kRefThreads, s, S);
  launch_after(p, k_ref_collect, grid, kRefThreads, s, S);
  RefArgs A;
  A.rel_t = w.rel_t;
  A.t_base = w.t_base;
  A.n_sft = p->n_sft;
  A.g = g;
  A.ax = plan_axes(p);
  A.wtab = w.wtab;
  A.n_tab = p->n_tab;
  A.i0 = w.i0;
  A.jend = w.jend;
  A.antenna = a->antenna;
  A.perm_ant = w.perm_ant;
  A.perm_x = w.perm_x;
  A.fafb = a->fafb;
  A.shared = sh;
  A.map = d_2F;
  A.cells = cells;
  A.ref_n = w.ref_n;
  A.ref_cell = w.ref_cell;
  A.ref_fast = w.ref_fast;
  A.ref_val = w.ref_val;
  A.st = w.tstat;
  A.cut = w.ref_bin;
  A.ref_ntile = w.ref_ntile;
  A.log_prior = p->log_prior;
  A.tol = fast_tol(p);
  A.out = d_summary;
  launch_after(p, k_ref_cells, dim3((unsigned)((cap + wpb - 1) / wpb), (unsigned)T), kRefThreads, s, A);
  p->launches += 4;
  return cudaGetLastError();
}

}  // namespace fmap
