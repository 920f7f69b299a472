// What every call does to its atoms before the sums: input checks, window index
// tables, and the copies each form reads (exponential sweeps, rectangular prefix
// sums, split tensor-core operands).  These steps depend on the atoms and the grid
// only, so a plan's call runs them side by side in one launch (fmap_front.cu); a
// batch runs them as phases.
#pragma once

#include "fmap_device.cuh"

namespace fmap {

// Decay after an atom, by its code in the copies: 1..kPowTab-1 the gap to the
// next atom in whole SFTs (the tau's float-float powers of the one-SFT decay), 0 any
// other gap (FP64 exp), -1 the last atom (no next one).
__host__ __device__ inline int32_t gap_code(int32_t gap, int32_t t_sft) {
  const int32_t k = gap / t_sft;
  return k >= 1 && k < kPowTab && k * t_sft == gap ? k : 0;
}

// Non-finite check of n values (antenna or data rows): DEV_ERR_NONFINITE
// is latched if any is NaN or infinite (|x| <= FLT_MAX fails for both; one
// atomic per warp at most).
__device__ __forceinline__ bool not_finite(float v) { return !(fabsf(v) <= 3.402823466e38f); }
__device__ __forceinline__ void finite_latch(bool bad, uint32_t* __restrict__ err) {
  const unsigned who = __ballot_sync(__activemask(), bad);
  if (bad && (int)(threadIdx.x & 31) == __ffs(who) - 1) atomicOr(err, DEV_ERR_NONFINITE);
}
__device__ __forceinline__ void finite_check(const float* __restrict__ v, int64_t n,
                                             int64_t i0, int64_t step, uint32_t* __restrict__ err) {
  bool bad = false;
#pragma unroll 4
  for (int64_t i = i0; i < n; i += step) bad |= not_finite(v[i]);
  finite_latch(bad, err);
}

// t -> t - t[0] as int32, with the data checks (strictly increasing,
// span < 2^31 s) latched into the plan's status word, and the atoms' values
// checked for NaN and infinities.
__device__ __forceinline__ void prep_body(const int64_t* __restrict__ t, int32_t n, int32_t n_alloc,
                       int32_t* __restrict__ rel_t, int64_t* __restrict__ t_base,
                       uint32_t* __restrict__ err, const float* __restrict__ ant, int64_t n_ant_vals,
                       const float* __restrict__ x, int64_t n_x_vals, int32_t* __restrict__ irr,
                       uint32_t* __restrict__ level, const uint3 bid, const dim3 gdim) {
  if (irr && bid.x == 0 && threadIdx.x < kIrrWords) irr[threadIdx.x] = 0;   // (set by the copies)
  if (level && bid.x == 0 && threadIdx.x < kLevelWords) level[threadIdx.x] = 0u;
  {
    const int64_t g0 = bid.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gdim.x * blockDim.x;
    if (ant) finite_check(ant, n_ant_vals, g0, step, err);
    if (x) finite_check(x, n_x_vals, g0, step, err);
  }
  if (n <= 0) return;
  const int64_t base = t[0];
  for (int64_t i = n + bid.x * (int64_t)blockDim.x + threadIdx.x; i < n_alloc;
       i += (int64_t)gdim.x * blockDim.x)
    rel_t[i] = 0;
  for (int64_t i = bid.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gdim.x * blockDim.x) {
    const int64_t ti = t[i];
    const int64_t d = ti - base;
    uint32_t e = 0;
    if (d < 0 || d > 0x7fffffffLL - 1) e |= DEV_ERR_SPAN;
    if (i + 1 < n && t[i + 1] <= ti) e |= DEV_ERR_ORDER;
    if (e) atomicOr(err, e);
    rel_t[i] = (int32_t)(d & 0x7fffffffLL);
    if (i == 0) *t_base = base;
  }
}

// Relative times: as stored by the checks above, or from the timestamps (the
// front kernel, where the checks run beside their readers).
struct RelStored {
  const int32_t* r;
  __device__ __forceinline__ int32_t operator[](int32_t i) const { return __ldg(r + i); }
};
struct RelTimes {
  const int64_t* t;
  int64_t base;
  __device__ __forceinline__ int32_t operator[](int32_t i) const {
    return (int32_t)((__ldg(t + i) - base) & 0x7fffffffLL);
  }
};

// irr: kIrrWords words, the longest gaps without a code (s) of parts of the atoms, 0
// where every gap has one (whole warps).
static_assert(kIrrWords == 32, "one word per lane");
__device__ __forceinline__ int32_t longest_gap(const int32_t* __restrict__ irr) {
  return __reduce_max_sync(0xffffffffu, irr[threadIdx.x & 31]);
}
__device__ __forceinline__ bool irregular(const int32_t* __restrict__ irr) {
  return longest_gap(irr) != 0;
}
// (1 where the times do not increase)
__device__ __forceinline__ int32_t uncoded_gap(int32_t gap, int32_t t_sft) {
  return gap_code(gap, t_sft) == 0 ? max(gap, 1) : 0;
}

// Word b of irr: the longest gap of the b-th of nb parts of the atoms that is not
// 1..kPowTab-1 whole SFTs; the words past nb are cleared.
template <typename Rel>
__device__ __forceinline__ void irregular_body(const Rel& t, int32_t n, int32_t t_sft,
                                               int32_t* __restrict__ irr, int32_t b, int32_t nb) {
  __shared__ int32_t s_gap;
  if (threadIdx.x == 0) s_gap = 0;
  __syncthreads();
  int32_t gap = 0;
  const int32_t per = (n + nb - 1) / nb, i0 = b * per, i1 = min(n - 1, i0 + per);
#pragma unroll 4
  for (int32_t i = i0 + threadIdx.x; i < i1; i += blockDim.x)
    gap = max(gap, uncoded_gap(t[i + 1] - t[i], t_sft));
  gap = __reduce_max_sync(0xffffffffu, gap);
  if ((threadIdx.x & 31) == 0 && gap) atomicMax(&s_gap, gap);
  __syncthreads();
  if (threadIdx.x == 0) irr[b] = s_gap;
  if (b == 0 && threadIdx.x >= nb && threadIdx.x < kIrrWords) irr[threadIdx.x] = 0;
}

// Window index tables: i0[m] = first atom with t >= t0_m; jend[m][n] = one
// past the last atom whose SFT ends by t0_m + L_n (L = window_len(tau_n)),
// clamped to >= i0[m], so the window holds atoms [i0, jend).  One block per
// group of kIdxGroup t0 rows: each warp finds one row's atom range
// [i0, j(n_tau - 1)) by a warp-wide search, the union of the group's ranges
// of relative times is staged in shared memory once (coalesced), and every
// (row, tau) searches it there; longer unions search global memory.
constexpr int kIdxThreads = 256;
constexpr int kIdxGroup = kIdxThreads / 32;   // t0 rows per block pass (one warp each)
constexpr int kIdxCap = 8192;   // staged relative times (32 KB)

// First index in [lo, hi) of the ascending int32 times with t > x (int64).
template <typename Rel>
__device__ __forceinline__ int32_t upper_bound_i32(const Rel& t, int32_t lo, int32_t hi,
                                                   int64_t x) {
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if ((int64_t)t[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The same search by one whole warp: 32 probes per round narrow the range
// 32-fold, so a data set of N atoms takes ~log32(N) dependent loads instead
// of log2(N).  Returns the first index in [lo, hi) whose time exceeds x (hi
// if none) to every lane.
template <typename Rel>
__device__ __forceinline__ int32_t warp_upper_bound_i32(const Rel& t, int32_t lo, int32_t hi,
                                                        int64_t x, int lane) {
  while (hi - lo > 32) {
    const int32_t step = (hi - lo + 31) / 32;
    const int32_t p = lo + lane * step;
    const bool le = p < hi && (int64_t)t[p] <= x;   // the probes below the answer
    const int c = __popc(__ballot_sync(0xffffffffu, le));
    if (c == 0) return lo;
    const int32_t base = lo;
    lo = base + (c - 1) * step + 1;
    hi = min(hi, base + c * step);
  }
  const int32_t p = lo + lane;
  const bool le = p < hi && (int64_t)t[p] <= x;
  return lo + __popc(__ballot_sync(0xffffffffu, le));
}

struct IndexSmem {
  int32_t t[kIdxCap], lo[kIdxGroup], hi[kIdxGroup];
};
template <typename Rel>
__device__ __forceinline__ void index_body(const Rel& rel_t, int64_t tb, int32_t n_sft,
                                           const fmap_grid g, const int64_t* __restrict__ ax,
                                           int32_t* __restrict__ i0tab,
                                           int32_t* __restrict__ jend, int32_t m0, int32_t R,
                                           IndexSmem& sm) {
  auto& s_t = sm.t;
  auto& s_lo = sm.lo;
  auto& s_hi = sm.hi;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t lmax = window_len(g, grid_tau(g, ax, g.n_tau - 1)) - g.t_sft;
  if (warp < R) {   // warp r: row m0 + r's first atom with t >= t0 and the last any window takes
    const int32_t m = m0 + warp;
    const int64_t t0rel = grid_t0(g, ax, m) - tb;
    const int32_t lo = warp_upper_bound_i32(rel_t, 0, n_sft, t0rel - 1, lane);
    const int32_t hi = max(lo, warp_upper_bound_i32(rel_t, lo, n_sft, t0rel + lmax, lane));
    if (lane == 0) {
      s_lo[warp] = lo;
      s_hi[warp] = hi;
      i0tab[m] = lo;
    }
  }
  __syncthreads();
  // The group's rows search within the union of their ranges, staged once when it
  // fits.  (Both ends grow with t0 where the timestamps increase, which the checks
  // only report: the union is taken over all of the rows, so that no search
  // leaves the staged part in any case.)
  int32_t base = s_lo[0], top = s_hi[0];
  for (int32_t r = 1; r < R; ++r) {
    base = min(base, s_lo[r]);
    top = max(top, s_hi[r]);
  }
  const int32_t span = top - base;
  const bool staged = span <= kIdxCap;
  if (staged)
    for (int k = tid; k < span; k += kIdxThreads) s_t[k] = rel_t[base + k];
  __syncthreads();
  for (int32_t r = 0; r < R; ++r) {   // no barrier between rows: their searches overlap
    const int32_t m = m0 + r, lo = s_lo[r], hi = s_hi[r];
    const int64_t t0rel = grid_t0(g, ax, m) - tb;
    int32_t* row = jend + (int64_t)m * g.n_tau;
    for (int32_t nn = tid; nn < g.n_tau; nn += kIdxThreads) {
      const int64_t lim = t0rel + window_len(g, grid_tau(g, ax, nn)) - g.t_sft;
      row[nn] = staged ? base + upper_bound_i32(s_t, lo - base, hi - base, lim)
                       : upper_bound_i32(rel_t, lo, hi, lim);
    }
  }
  __syncthreads();   // s_t, s_lo and s_hi are reused by the block's next group
}

// The data's range of levels, noted by the copies for the sweeps: level[0] the bits
// of the largest absolute value, level[1] the complement of the bits of the smallest
// maximum of 32 neighbouring atoms (all-zero ones do not count; 0: there are none).
// Both only grow; zero before the copies.
constexpr float kLevelRange = 128.0f;
__device__ __forceinline__ void level_note(uint32_t* level, unsigned hi, unsigned lo, int lane) {
  if (lane != 0) return;   // (most warps have nothing new: no atomic)
  if (hi > __ldcg(level)) atomicMax(level, hi);
  if (lo != 0xffffffffu && ~lo > __ldcg(level + 1)) atomicMax(level + 1, ~lo);
}
__device__ __forceinline__ bool level_varies(const uint32_t* level) {
  const uint32_t hi = level[0], lo = level[1];
  return lo != 0u && __uint_as_float(hi) > kLevelRange * __uint_as_float(~lo);
}

// Copies of one instance's atoms for the sweeps, one 16-byte entry per atom:
// sets 0..n_ant-1 the antenna rows with the code of the gap to the next atom
// (gap_code), sets n_ant.. the data rows of each template (recurrence plans);
// before them the per-tau constants (two entries per tau).  The values are checked
// on the way; irr, if given, takes the gaps without a code.  By whole warps of
// consecutive entries.
template <typename Rel>
__device__ __forceinline__ void exp_perm_body(const Rel& rel_t, int32_t n,
                                              const float* __restrict__ antenna, int32_t n_ant,
                                              const float* __restrict__ fafb, int32_t n_x,
                                              float4* __restrict__ perm_ant,
                                              float4* __restrict__ perm_x,
                                              int32_t* __restrict__ irr, uint32_t* level,
                                              uint32_t* __restrict__ err, const fmap_grid& g,
                                              const int64_t* __restrict__ ax,
                                              TauTab* __restrict__ tauc, int64_t e_begin,
                                              int64_t e_end, int64_t e_step) {
  const int64_t n_tau2 = 2 * (int64_t)g.n_tau;
  bool bad = false;
  auto copy = [&](int64_t e0) -> float {   // a data entry's largest absolute value, else -1
    if (e0 < n_tau2) {   // the longest entries first
      tau_tab_fill(g, grid_tau(g, ax, e0 >> 1), (int)(e0 & 1), tauc + (e0 >> 1));
      return -1.0f;
    }
    const int64_t e = e0 - n_tau2;
    const int64_t set = e / n, i = e - set * n;
    if (set < n_ant) {
      const float* a = antenna + set * 3 * (int64_t)n;
      const int32_t t = rel_t[i];
      const int32_t code = i + 1 < n ? gap_code(rel_t[i + 1] - t, (int32_t)g.t_sft) : -1;
      const float4 v = make_float4(a[i], a[n + i], a[2 * (int64_t)n + i], __int_as_float(code));
      bad |= not_finite(v.x) || not_finite(v.y) || not_finite(v.z);
      perm_ant[e] = v;
      if (irr && set == 0 && code == 0)   // (a batch; cleared by the input checks)
        atomicMax(irr + (i & (kIrrWords - 1)), uncoded_gap(rel_t[i + 1] - t, (int32_t)g.t_sft));
      return -1.0f;
    }
    const int64_t tq = set - n_ant;
    const float* x = fafb + tq * 4 * (int64_t)n;
    const float4 v = make_float4(x[i], x[n + i], x[2 * (int64_t)n + i], x[3 * (int64_t)n + i]);
    bad |= not_finite(v.x) || not_finite(v.y) || not_finite(v.z) || not_finite(v.w);
    perm_x[tq * n + i] = v;
    return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
  };
  unsigned hi = 0u, lo = 0xffffffffu;
  for (int64_t e0 = e_begin; __any_sync(0xffffffffu, e0 < e_end); e0 += e_step) {
    const float top = e0 < e_end ? copy(e0) : -1.0f;
    if (n_x == 0) continue;
    const bool whole = __all_sync(0xffffffffu, top >= 0.0f);
    const unsigned m = __reduce_max_sync(0xffffffffu, top > 0.0f ? __float_as_uint(top) : 0u);
    hi = max(hi, m);
    if (whole && m) lo = min(lo, m);
  }
  if (n_x > 0) level_note(level, hi, lo, threadIdx.x & 31);
  finite_latch(bad, err);
}

constexpr int kScanThreads = 256;
constexpr int kScanPer = 4;
constexpr int kScanTile = kScanThreads * kScanPer;

// Antenna prefix entry: (sum a2, sum b2, sum ab, 0) as float pairs.
struct __align__(32) P4 {
  float4 hi, lo;
};

// Prefix sums of NC rows of n atoms by one block: out[2 i], out[2 i + 1] = hi,
// lo of sum_{a < i} for i = 0..n (columns past NC are 0).  The sums are exact
// 64-bit integers in units of 2^-S, S the largest with sum|x| 2^S < 2^62 per
// row, and the pair holds the top 48 bits.  (The same scan in FP64, which GB300
// runs at 1/64 of the FP32 rate, took eight FP64 operations per atom and row:
// 423 us for 1024 templates of 5000 atoms, and 24 us for one block alone.)
// The unit is fixed by the row's sum, so rows with two neighbouring atoms (not both 0)
// below 2^-37 of it, which the unit holds to less than 25 bits (before an outlier or a
// step the windows, of two atoms at least, would lose their sums), rows below 2^-57
// and blocks of fewer than 64 atoms are summed in FP64.  (By the maxima of stretches of
// 32 atoms a glitch in every stretch hid the small atoms before the first of them,
// whose windows lost up to all of their sums; by every atom for itself a zero crossing
// of the antenna pattern put a year's b^2, and 18 us more, on the FP64 path.)
// A tile of kScanTile atoms at a time: each thread sums kScanPer neighbours,
// the warps scan the threads' sums by shuffles, and the entries leave through
// shared memory so that the block writes whole lines.
struct ScanSmem {
  float tile[4][kScanTile];
  float4 ent[2 * kScanTile];
  unsigned long long wsum[4][kScanThreads / 32];
  float wabs[4][kScanThreads / 32], wmin[4][kScanThreads / 32];
};
constexpr int32_t kScanFixMin = 64;   // fewest atoms of an integer scan

// Exponent e of v >= 0 (v < 2^e; 0 of 0).
__host__ __device__ inline int scan_exponent(float v) {
  int e = 0;
  if (v > 0.0f) frexpf(v, &e);
  return e;
}
// Place of entry float4 k in the staging buffer: a thread's entries are 2 kScanPer
// float4 apart, so the low three bits take its number and a warp's stores spread
// over the banks.
__device__ __forceinline__ int scan_place(int k) { return k ^ ((k / (2 * kScanPer)) & 7); }

// The two accumulators: integers in units of down = 1 / up (both powers of two;
// the scaling is exact but for underflow), and FP64.
template <typename Acc> struct ScanAcc;
template <> struct ScanAcc<unsigned long long> {
  static __device__ __forceinline__ unsigned long long in(float x, float up) {
    return (unsigned long long)__float2ll_rn(x * up);
  }
  static __device__ __forceinline__ float2 pair(unsigned long long v, float down) {
    const float h = __ll2float_rn((long long)v);
    return make_float2(h * down, __ll2float_rn((long long)v - __float2ll_rn(h)) * down);
  }
};
template <> struct ScanAcc<double> {
  static __device__ __forceinline__ double in(float x, float) { return (double)x; }
  static __device__ __forceinline__ float2 pair(double v, float) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
  }
};

template <int NC, typename Acc>
__device__ __forceinline__ void rect_scan_tiles(const float* __restrict__ x, int32_t n,
                                                const float (&up)[NC], const float (&down)[NC],
                                                float4* __restrict__ out, ScanSmem& sm) {
  constexpr int NW = kScanThreads / 32;
  using A = ScanAcc<Acc>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  Acc(*wsum)[NW] = reinterpret_cast<Acc(*)[NW]>(sm.wsum);
  Acc carry[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) carry[c] = Acc(0);
  for (int32_t base = 0; base < n; base += kScanTile) {
    __syncthreads();
    for (int k = tid; k < kScanTile; k += kScanThreads)
#pragma unroll
      for (int c = 0; c < NC; ++c) sm.tile[c][k] = base + k < n ? x[c * (int64_t)n + base + k] : 0.0f;
    __syncthreads();
    Acc v[NC][kScanPer], own[NC], inc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      own[c] = Acc(0);
      const float4* t4 = reinterpret_cast<const float4*>(&sm.tile[c][tid * kScanPer]);
#pragma unroll
      for (int e = 0; e < kScanPer; e += 4) {
        const float4 t = t4[e / 4];
        v[c][e] = A::in(t.x, up[c]);
        v[c][e + 1] = A::in(t.y, up[c]);
        v[c][e + 2] = A::in(t.z, up[c]);
        v[c][e + 3] = A::in(t.w, up[c]);
        own[c] += v[c][e] + v[c][e + 1] + v[c][e + 2] + v[c][e + 3];
      }
      inc[c] = own[c];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const Acc y = __shfl_up_sync(0xffffffffu, inc[c], d);
        if (lane >= d) inc[c] += y;
      }
    if (lane == 31)
#pragma unroll
      for (int c = 0; c < NC; ++c) wsum[c][warp] = inc[c];
    __syncthreads();
    Acc run[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      run[c] = carry[c];
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const Acc t = wsum[c][w];
        if (w < warp) run[c] += t;
        carry[c] += t;
      }
      const Acc before = __shfl_up_sync(0xffffffffu, inc[c], 1);
      if (lane > 0) run[c] += before;
    }
#pragma unroll
    for (int e = 0; e < kScanPer; ++e) {
      float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        run[c] += v[c][e];
        const float2 p = A::pair(run[c], down[c]);
        hi[c] = p.x;
        lo[c] = p.y;
      }
      const int k = 2 * (tid * kScanPer + e);
      sm.ent[scan_place(k)] = make_float4(hi[0], hi[1], hi[2], hi[3]);
      sm.ent[scan_place(k + 1)] = make_float4(lo[0], lo[1], lo[2], lo[3]);
    }
    __syncthreads();
    const int32_t m = 2 * min(kScanTile, n - base);
    for (int32_t k = tid; k < m; k += kScanThreads) out[2 * (int64_t)(base + 1) + k] = sm.ent[scan_place(k)];
  }
}

// (out of line: the common path's registers and instructions stay its own)
template <int NC>
__device__ __noinline__ void rect_scan_fp64(const float* __restrict__ x, int32_t n,
                                            float4* __restrict__ out, ScanSmem& sm) {
  const float one[NC] = {};
  rect_scan_tiles<NC, double>(x, n, one, one, out, sm);
}

template <int NC>
__device__ __forceinline__ void rect_scan_body(const float* __restrict__ x, int32_t n,
                                               float4* __restrict__ out,
                                               uint32_t* __restrict__ err, ScanSmem& sm) {
  constexpr int NW = kScanThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 2) out[tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  bool fix = n >= kScanFixMin;
  float up[NC], down[NC];
  if (fix) {
    // each row's sum of absolute values, and the smallest maximum of two neighbours
    // (two zeros do not count)
    float sum[NC], mn[NC];
    bool bad = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      sum[c] = 0.0f;
      mn[c] = 3.402823466e38f;
    }
#pragma unroll 2
    for (int32_t a0 = 32 * warp; a0 < n; a0 += kScanThreads) {   // (the rows' loads together)
      const int32_t a = a0 + lane;
      float m[NC], next[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float* r = x + c * (int64_t)n + a;
        m[c] = a < n ? fabsf(r[0]) : 0.0f;
        next[c] = lane == 31 && a + 1 < n ? fabsf(r[1]) : 0.0f;
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        bad |= not_finite(m[c]);
        sum[c] += m[c];
        const float y = __shfl_down_sync(0xffffffffu, m[c], 1);
        const float top = fmaxf(m[c], lane < 31 ? y : next[c]);
        if (a + 1 < n && top > 0.0f) mn[c] = fminf(mn[c], top);
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) sum[c] += __shfl_xor_sync(0xffffffffu, sum[c], d);
      mn[c] = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(mn[c])));
      if (lane == 0) {
        sm.wabs[c][warp] = sum[c];
        sm.wmin[c][warp] = mn[c];
      }
    }
    finite_latch(bad, err);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      sum[c] = 0.0f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        sum[c] += sm.wabs[c][w];
        mn[c] = fminf(mn[c], sm.wmin[c][w]);
      }
      // (a thread adds n / 256 values: up to 2^24 atoms the FP32 sum is within 2^-8)
      const int e = scan_exponent(sum[c] * 1.00390625f), S = 62 - e;
      fix = fix && n <= 1 << 24 && !not_finite(sum[c] * 1.00390625f) &&
            (sum[c] == 0.0f || (S <= 119 && S >= -100 && scan_exponent(mn[c]) >= e - 36));
      const int Sc = max(-100, min(119, S));
      up[c] = __int_as_float((Sc + 127) << 23);
      down[c] = __int_as_float((127 - Sc) << 23);
    }
  } else {
    finite_check(x, (int64_t)NC * n, tid, kScanThreads, err);
  }
  if (fix) rect_scan_tiles<NC, unsigned long long>(x, n, up, down, out, sm);
  else rect_scan_fp64<NC>(x, n, out, sm);
}

// Scans of the antenna sets (blocks [0, n_ant)), then of the templates' data.
__device__ __forceinline__ void rect_scan_unit(const float* antenna, const float* fafb, int32_t n,
                                               int32_t n_ant, P4* pa, float4* px, int32_t b,
                                               uint32_t* err, ScanSmem& sm) {
  if (b < n_ant)
    rect_scan_body<3>(antenna + (int64_t)b * 3 * n, n, (float4*)(pa + (int64_t)b * (n + 1)), err, sm);
  else
    rect_scan_body<4>(fafb + (int64_t)(b - n_ant) * 4 * n, n,
                      px + (int64_t)(b - n_ant) * 2 * (n + 1), err, sm);
}

__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t y;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(x));
  return y;
}
// Pack (lo_elem -> bits 15:0, hi_elem -> bits 31:16) as bf16x2, round to nearest.
__device__ __forceinline__ uint32_t pack_bf16(float even, float odd) {
  uint32_t y;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(y) : "f"(odd), "f"(even));
  return y;
}
// Split X into hi + lo operands ([4T][n_pad], zero padded): TF32 (stored as
// FP32 bit patterns with 13 low zero bits) or BF16.
template <bool BF16>
__device__ __forceinline__ void split_x_body(const float* __restrict__ fafb, int32_t n_sft,
                                             int32_t ncols, int32_t n_pad, void* __restrict__ hi,
                                             void* __restrict__ lo, uint32_t* __restrict__ err,
                                             int64_t first, int64_t step) {
  const int64_t total = (int64_t)ncols * n_pad;
  bool bad = false;
  for (int64_t i = first; i < total; i += step) {
    const int64_t c = i / n_pad;
    const int32_t a = (int32_t)(i - c * n_pad);
    const float x = a < n_sft ? fafb[c * n_sft + a] : 0.0f;
    bad |= not_finite(x);
    if constexpr (BF16) {
      const uint32_t hp = pack_bf16(x, 0.0f);
      const float hx = __uint_as_float(hp << 16);
      const uint32_t lp = pack_bf16(x - hx, 0.0f);
      ((uint16_t*)hi)[i] = (uint16_t)(hp & 0xffffu);
      ((uint16_t*)lo)[i] = (uint16_t)(lp & 0xffffu);
    } else {
      const uint32_t hb = to_tf32(x);
      ((uint32_t*)hi)[i] = hb;
      ((uint32_t*)lo)[i] = to_tf32(x - __uint_as_float(hb));
    }
  }
  finite_latch(bad, err);
}
}  // namespace fmap
