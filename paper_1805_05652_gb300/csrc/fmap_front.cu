// The first launch of a plan's call (fmap_front.cuh): blocks of each role side by
// side, the longest chains first.  As separate launches (bitmask memset, checks,
// index, copies or scans, operand split) each waited for the one before; on a small
// map they were a quarter of the call.
#include <algorithm>

#include "fmap_front.cuh"

namespace fmap {

struct FrontArgs {
  fmap_grid g;
  int32_t n, n_ant, T;
  int32_t n_alloc;              // entries of rel_t
  const int64_t* t;
  const float* antenna;
  const float* fafb;
  const int64_t* ax;
  uint32_t* err;
  int32_t* rel_t;
  int64_t* t_base;
  int32_t* irr;
  uint32_t* level;
  uint4* bits;                  // marked-entry bitmask, cleared here
  int64_t n_bits;               // uint4s
  int32_t* i0;
  int32_t* jend;
  int32_t idx_rows;             // t0 rows per index group
  // blocks of each role, in this order
  int32_t b_scan, b_idx, b_irr, b_copy, b_split, b_prep;
  // exponential copies
  float4* perm_ant;
  float4* perm_x;
  int32_t n_x;
  TauTab* tauc;
  // rectangular prefix sums
  P4* pa;
  float4* px;
  // tensor-core operands
  void* hi;
  void* lo;
  int32_t n_pad, bf16;
  // values not checked by the copies
  int64_t n_ant_vals, n_x_vals;
};

constexpr int kFrontThreads = 256;
static_assert(kFrontThreads == kIdxThreads && kFrontThreads == kScanThreads, "roles share blocks");

// (three blocks per SM: at two, by registers, 329 scans of 4606 atoms took a second wave
// and the call 399 us for 363)
__global__ void __launch_bounds__(kFrontThreads, 3) k_front(const FrontArgs F) {
  extern __shared__ __align__(16) unsigned char s_front[];
  int32_t b = blockIdx.x;
  if (b < F.b_scan) {
    rect_scan_unit(F.antenna, F.fafb, F.n, F.n_ant, F.pa, F.px, b, F.err,
                   *reinterpret_cast<ScanSmem*>(s_front));
    return;
  }
  b -= F.b_scan;
  const int64_t tb = F.n > 0 ? F.t[0] : 0;
  const RelTimes rel{F.t, tb};
  if (b < F.b_idx) {
    const int32_t n_grp = (F.g.n_t0 + F.idx_rows - 1) / F.idx_rows;
    for (int32_t q = b; q < n_grp; q += F.b_idx)
      index_body(rel, tb, F.n, F.g, F.ax, F.i0, F.jend, q * F.idx_rows,
                 min(F.idx_rows, F.g.n_t0 - q * F.idx_rows),
                 *reinterpret_cast<IndexSmem*>(s_front));
    return;
  }
  b -= F.b_idx;
  if (b < F.b_irr) {
    irregular_body(rel, F.n, (int32_t)F.g.t_sft, F.irr, b, F.b_irr);
    return;
  }
  b -= F.b_irr;
  if (b < F.b_copy) {
    exp_perm_body(rel, F.n, F.antenna, F.n_ant, F.fafb, F.n_x, F.perm_ant, F.perm_x, nullptr, F.level, F.err, F.g,
                  F.ax, F.tauc, (int64_t)b * kFrontThreads + threadIdx.x,
                  exp_copy_entries(F.n, F.n_ant, F.n_x, F.g.n_tau),
                  (int64_t)F.b_copy * kFrontThreads);
    return;
  }
  b -= F.b_copy;
  if (b < F.b_split) {
    const int64_t first = (int64_t)b * kFrontThreads + threadIdx.x;
    const int64_t step = (int64_t)F.b_split * kFrontThreads;
    if (F.bf16) split_x_body<true>(F.fafb, F.n, 4 * F.T, F.n_pad, F.hi, F.lo, F.err, first, step);
    else split_x_body<false>(F.fafb, F.n, 4 * F.T, F.n_pad, F.hi, F.lo, F.err, first, step);
    return;
  }
  b -= F.b_split;
  for (int64_t i = (int64_t)b * kFrontThreads + threadIdx.x; i < F.n_bits;
       i += (int64_t)F.b_prep * kFrontThreads)
    F.bits[i] = make_uint4(0u, 0u, 0u, 0u);
  prep_body(F.t, F.n, F.n_alloc, F.rel_t, F.t_base, F.err, F.n_ant_vals ? F.antenna : nullptr,
            F.n_ant_vals, F.n_x_vals ? F.fafb : nullptr, F.n_x_vals, nullptr, nullptr,
            make_uint3((unsigned)b, 0, 0), dim3((unsigned)F.b_prep));
}

cudaError_t launch_front(fmap_plan_s* p, const fmap_atoms* a, cudaStream_t s) {
  const fmap_grid& g = p->grid;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  const bool sh = a->shared_antenna != 0;
  const bool rec = g.window == FMAP_EXP && (p->flags & FMAP_PLAN_EXP_RECURRENCE);
  const bool tc = g.window != FMAP_RECT && !rec &&
                  (p->precision == FMAP_TF32 || p->precision == FMAP_BF16X3);
  FrontArgs F{};
  F.g = g;
  F.n = p->n_sft;
  F.T = p->n_templates;
  F.n_ant = sh ? 1 : F.T;
  F.n_alloc = rel_t_entries(F.n);
  F.t = a->t;
  F.antenna = a->antenna;
  F.fafb = a->fafb;
  F.ax = plan_axes(p);
  F.err = p->ws.dev_err;
  F.rel_t = p->ws.rel_t;
  F.t_base = p->ws.t_base;
  F.irr = p->ws.irr;
  F.level = p->ws.level;
  F.bits = (uint4*)p->ws.flag_bits;
  F.i0 = p->ws.i0;
  F.jend = p->ws.jend;
  F.perm_ant = p->ws.perm_ant;
  F.perm_x = p->ws.perm_x;
  F.tauc = p->ws.tauc;
  F.pa = (P4*)p->ws.pa;
  F.px = p->ws.px;
  const int64_t n = F.n;
  const int64_t most = (int64_t)p->n_sm * 16;   // blocks of a streaming role
  auto blocks = [&](int64_t items) {
    return (int32_t)std::min<int64_t>((items + kFrontThreads - 1) / kFrontThreads, most);
  };
  bool ant_checked = false, x_checked = F.T == 0;
  size_t smem = 0;
  if (cells > 0) {
    F.n_bits = flag_words(cells * (sh ? 1 : std::max<int32_t>(F.T, 1))) / 4;
    // rows per index group: as many as keep about four blocks per SM busy (1..8)
    F.idx_rows = (int32_t)std::max<int64_t>(
        1, std::min<int64_t>(kIdxGroup, g.n_t0 / ((int64_t)p->n_sm * 4)));
    F.b_idx = (int32_t)std::min<int64_t>((g.n_t0 + F.idx_rows - 1) / F.idx_rows, (int64_t)p->n_sm * 8);
    smem = sizeof(IndexSmem);
    if (g.window == FMAP_RECT) {
      // (the FP32 form takes its data sums from the atoms)
      const int32_t n_x = p->precision == FMAP_FP32 ? 0 : F.T;
      F.b_scan = F.n_ant + n_x;
      ant_checked = F.n_ant > 0;
      x_checked = x_checked || n_x > 0;
      smem = std::max(smem, sizeof(ScanSmem));
    } else if (g.window == FMAP_EXP) {
      F.n_x = F.perm_x ? F.T : 0;
      F.b_irr = (int32_t)std::max<int64_t>(1, std::min<int64_t>(kIrrWords, n / 2048));
      F.b_copy = blocks(exp_copy_entries(F.n, F.n_ant, F.n_x, g.n_tau));
      ant_checked = F.n_ant > 0;
      x_checked = x_checked || F.n_x > 0;
    }
    if (tc && F.T > 0) {
      F.bf16 = p->precision == FMAP_BF16X3;
      exp_tc_operands(p, &F.hi, &F.lo, &F.n_pad);
      F.b_split = blocks((int64_t)4 * F.T * F.n_pad);
      x_checked = true;
    }
  }
  F.n_ant_vals = ant_checked ? 0 : 3 * n * F.n_ant;
  F.n_x_vals = x_checked ? 0 : 4 * n * F.T;
  // enough threads for the timestamps and the bitmask, and for the value checks at
  // a few values per thread
  F.b_prep = blocks(std::max({n, F.n_bits / 4, (F.n_ant_vals + F.n_x_vals) / 8, (int64_t)1}));
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_front, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int64_t total = (int64_t)F.b_scan + F.b_idx + F.b_irr + F.b_copy + F.b_split + F.b_prep;
  k_front<<<(unsigned)total, kFrontThreads, smem, s>>>(F);
  p->launches += 1;
  return cudaGetLastError();
}

}  // namespace fmap
