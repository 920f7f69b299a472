// Exponential-window F-map (Eq. winexp, cut after 3 tau).
//
// Antenna part (shared by every template of a sky position): A, B, C with the
// squared weight w^2 = e^{-2(t - t0)/tau}, from a decayed suffix sum per tau in
// float-float arithmetic (the FP32 pipe; GB300's FP64 rate is 1/64 of it):
//     E[i] = x_i + e^{-2(t_{i+1} - t_i)/tau} E[i+1],
//     A(t0, tau) = e^{-2(t_{i0} - t0)/tau} (E[i0] - e^{-2(t_j - t_{i0})/tau} E[j])
// for the window's atoms [i0, j).  The recurrence is contractive, so the
// subtraction loses at most a factor 1/(1 - e^{-6}) of relative accuracy.
// Then D = AB - C^2 in float-float and the per-cell 2F coefficients.
//
// Data part: Fa, Fb = sum_a w(t_a) X[a, col] over the window, a contraction
// of the weight matrix W[(t0, tau), a] with the 4T data columns.  Here the
// plain CUDA-core form (the paper's brute-force exp kernel, Sec. 3, restated
// with shared-memory staging and one thread per cell): FP32 or FP64
// accumulation.  The tensor-core form lives in fmap_exp_tc.cu.
#include <math.h>

#include <type_traits>

#include <algorithm>

#include "fmap_batch.cuh"
#include "fmap_front.cuh"
#include "fmap_sweep.cuh"

namespace fmap {

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------------------
// Antenna sums and coefficients, in two launches of independent warps.
//
//   k_sweep_agg (fmap_exp_rec.cu): per (32 tau, chunk of atoms) the affine map E[first] = S + R
//     E[next chunk's first] of the decayed suffix recurrence, in float-float.
//   k_exp_antenna: per (32 tau, run of t0 rows) a warp composes the chunks'
//     maps down to the chunks that hold its last row's i0 and j, steps both
//     cursors to those atoms, and sweeps its rows (fmap_sweep.cuh).
//
// Bound by instruction issue: about 45 float-float operations per cell for the
// sums and 75 for the coefficients.  The chunk maps keep a short run of rows
// cheap to start (a window's atoms would otherwise be summed again by each run),
// so that the rows split into enough warps to fill the GPU.
// ---------------------------------------------------------------------------
constexpr int kAntWarps = kSweepWarps;
constexpr int kAntThreads = 32 * kAntWarps;

// Tail factors above this size are taken from FP64 exp as float pairs: the
// window sum E[i0] - tail E[j] then loses 1 / (1 - tail) of relative accuracy
// to the tail's own error, which the ill-conditioned D = AB - C^2 amplifies
// further (windows cut well before 3 tau, or starting in a long gap).
constexpr float kTailExact = 1.0f / 32.0f;

// (out of line, as slow_decay)
static __device__ __noinline__ float2 exact_tail(int32_t dj, double inv_s) {
  const FF v = ff_of(exp(-(double)dj * inv_s));
  return make_float2(v.h, v.l);
}

template <bool IRR>
__device__ __forceinline__ void exp_antenna_unit(
    const int32_t* __restrict__ rel_t, const int64_t* __restrict__ t_base, int32_t n,
    const fmap_grid& g, const float4* __restrict__ ant, const TauTab* __restrict__ tauc,
    const int64_t* __restrict__ ax, const int32_t* __restrict__ i0tab,
    const int32_t* __restrict__ jend, const AntGeom& q, const float* __restrict__ agg,
    Coef* __restrict__ coef, uint32_t* __restrict__ bits, int64_t unit, float2* s_pw, int lane) {
  const int32_t seg = (int32_t)(unit % q.n_seg);
  const int64_t ag = unit / q.n_seg;
  const int32_t grp = (int32_t)(ag % q.n_grp);
  const int64_t ta = ag / q.n_grp;
  const int32_t ni = grp * 32 + lane, nn = min(ni, g.n_tau - 1);
  const int32_t m_lo = seg * q.rows, m_hi = min(g.n_t0, m_lo + q.rows);
  const TauTab* tt = tauc + nn;
  sweep_tab_load<2>(s_pw, tt, lane);
  const float c2 = tt->c2[1];
  const int64_t tb = n > 0 ? *t_base : 0;
  const float4* x = ant + ta * n;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  // (each cursor's next atom is loaded one step ahead)
  auto step = [&](AntE& e, float4& v, int32_t a) {
    const float4 w = v;
    v = __ldg(x + max(a - 1, 0));
    ant_step(e, sweep_decay<2, IRR>(s_pw, __float_as_int(w.w), lane, rel_t, a, tt), w);
  };
  const int32_t jt = jend[(int64_t)(m_hi - 1) * g.n_tau + nn];
  const int32_t it = i0tab[m_hi - 1];
  AntE Ei = ant_zero(), Ej = ant_zero();
  int32_t ic, jc;
  if (q.n_chunks > 0) {
    // E at the first atoms of the chunks after those holding j and i0 of the
    // last row (E = 0 at the end of the chunk of the warp's last window end)
    const int32_t bj = (jt + q.chunk - 1) / q.chunk, bi = (it + q.chunk - 1) / q.chunk;
    FF E[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    const float* o = agg + ag * q.n_chunks * 256 + lane;
    constexpr int B = 2;   // chunk maps loaded ahead
    for (int32_t b0 = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)bj);; b0 -= B) {
      float w[B][8];
#pragma unroll
      for (int u = 0; u < B; ++u)
#pragma unroll
        for (int e = 0; e < 8; ++e) w[u][e] = o[(int64_t)max(b0 - 1 - u, 0) * 256 + 32 * e];
      bool done = false;
#pragma unroll
      for (int u = 0; u < B; ++u) {
        if (b0 - u == bj) ant_put(Ej, E);
        if (b0 - u <= bi) {
          done = true;
          break;
        }
        const FF R{w[u][6], w[u][7]};
#pragma unroll
        for (int c = 0; c < 3; ++c) E[c] = ff_fma_sum(FF{w[u][2 * c], w[u][2 * c + 1]}, R, E[c]);
      }
      if (done) break;
    }
    ant_put(Ei, E);
    ic = min(n, bi * q.chunk);
    jc = min(n, bj * q.chunk);
  } else {
    // E starts from zero at each lane's window end of the last row
    jc = jt;
    ic = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)jt);
    const int32_t j_all = (int32_t)__reduce_min_sync(0xffffffffu, (unsigned)jt);
    while (ic > max(it, j_all)) {   // atoms past some lanes' ends
      --ic;
      const float4 v = __ldg(x + ic);
      if (ic < jt)
        ant_step(Ei, sweep_decay<2, IRR>(s_pw, __float_as_int(v.w), lane, rel_t, ic, tt), v);
    }
  }
  float4 vi = n > 0 ? __ldg(x + max(ic - 1, 0)) : float4{}, vj = n > 0 ? __ldg(x + max(jc - 1, 0)) : float4{};
  // the window ends and starts of a row are loaded one row ahead
  int32_t i0 = it, j = jt;
  for (int32_t m = m_hi - 1; m >= m_lo; --m) {
    const int64_t cell = (int64_t)m * g.n_tau + nn;
    int32_t i0n = 0, jn = 0;
    if (m > m_lo) {
      i0n = i0tab[m - 1];
      jn = jend[cell - g.n_tau];
    }
    while (ic > i0) step(Ei, vi, --ic);
    while (jc > j) step(Ej, vj, --jc);
    ant_norm(Ei);
    ant_norm(Ej);
    // The prefactor scales A, B, C alike (F changes by its relative error
    // only): FP32 exp2 is accurate enough.  The tail is FP32 exp2 while it is
    // small (~e^{-6} of the window sum for the default 3 tau cut), FP64 exp
    // otherwise.
    FF S[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    if (j > i0) {
      const int32_t ti = rel_t[i0];
      const int64_t d0 = (int64_t)ti - (grid_t0(g, ax, m) - tb);
      FF ei[3], ej[3];
      ant_get(Ei, ei);
      ant_get(Ej, ej);
      FF tail{0.0f, 0.0f};
      if (j < n) {
        const int32_t dj = rel_t[j] - ti;
        tail.h = ex2_approx(c2 * (float)dj);
        if (tail.h > kTailExact) {
          const float2 v = exact_tail(dj, 2.0 * tt->inv_tau);
          tail = {v.x, v.y};
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) S[c] = ff_sub(ei[c], ff_mul(ej[c], tail));
      if (d0 != 0) {
        const float pre = ex2_approx(c2 * (float)d0);
#pragma unroll
        for (int c = 0; c < 3; ++c) S[c] = ff_mul_f(S[c], pre);
      }
    }
    const Coef cf = make_coef_ff(S[0], S[1], S[2], j - i0);
    if (ni < g.n_tau) store_coef(coef, bits, ta * cells + cell, cf);
    i0 = i0n;
    j = jn;
  }
}

__global__ void __launch_bounds__(kAntThreads, 3)
k_exp_antenna(const int32_t* __restrict__ rel_t, const int64_t* __restrict__ t_base, int32_t n,
              const fmap_grid g, const float4* __restrict__ ant, const TauTab* __restrict__ tauc,
              const int64_t* __restrict__ ax, const int32_t* __restrict__ i0tab,
              const int32_t* __restrict__ jend, const AntGeom q, const float* __restrict__ agg,
              Coef* __restrict__ coef, uint32_t* __restrict__ bits,
              const int32_t* __restrict__ irr, int64_t units) {
  __shared__ float2 s_pw[kAntWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t unit = (int64_t)blockIdx.x * kAntWarps + warp;
  if (unit >= units) return;
  if (irregular(irr))
    exp_antenna_unit<true>(rel_t, t_base, n, g, ant, tauc, ax, i0tab, jend, q, agg, coef, bits,
                           unit, s_pw[warp], lane);
  else
    exp_antenna_unit<false>(rel_t, t_base, n, g, ant, tauc, ax, i0tab, jend, q, agg, coef, bits,
                            unit, s_pw[warp], lane);
}

// Chunks of 16 atoms for short data sets (a warp's start is then a handful
// of steps), 128 for long ones (fewer maps to compose), larger ones where the
// maps have no room (agg_room bytes), none where the rows make a single run per
// 32 tau anyway; rows
// per warp so that about 16 warps per SM run at once, at least 4 (the start
// costs about as much as eight); in a batch, whose instances fill the GPU
// together, 64, or fewer where a row's step spans many SFTs.
AntGeom ant_geom(const fmap_grid& g, int32_t n_sft, int64_t n_ant, bool batch, int64_t agg_room) {
  AntGeom q{};
  q.n_grp = std::max(1, (g.n_tau + 31) / 32);
  const int64_t warps = q.n_grp * std::max<int64_t>(n_ant, 1);   // per run of rows
  const int64_t want = ((int64_t)kSms * 16 + warps - 1) / warps;
  // SFTs per row (a single row's dt0 is not restricted, nor used)
  const int64_t step = g.n_t0 > 1 ? g.dt0 / std::max<int64_t>(g.t_sft, 1) : 1;
  q.rows = batch ? (int32_t)std::clamp<int64_t>(1024 / (step + 3), 8, 64)
                 : (int32_t)std::max<int64_t>(4, (g.n_t0 + want - 1) / want);
  q.n_seg = std::max(1, (g.n_t0 + q.rows - 1) / q.rows);
  q.chunk = n_sft <= 1024 ? 16 : n_sft <= 4096 ? 32 : 128;
  q.n_chunks = (n_sft + q.chunk - 1) / q.chunk;
  if (q.n_seg == 1 && q.n_chunks > 0 && g.n_t0 > 64) q.n_chunks = 0;
  while (1024 * warps * q.n_chunks > agg_room && q.chunk < 1024) {
    q.chunk *= 2;
    q.n_chunks = (n_sft + q.chunk - 1) / q.chunk;
  }
  if (1024 * warps * q.n_chunks > agg_room) q.n_chunks = 0;
  return q;
}

cudaError_t launch_exp_coef(fmap_plan_s* p, const fmap_atoms* a, cudaStream_t s) {
  const fmap_grid& g = p->grid;
  if ((int64_t)g.n_t0 * g.n_tau == 0) return cudaSuccess;
  const int n_ant = a->shared_antenna ? 1 : p->n_templates;
  if (n_ant == 0) return cudaSuccess;
  const AntGeom& q = p->ant[a->shared_antenna ? 1 : 0];
  const int64_t ag = (int64_t)q.n_grp * n_ant;
  const int64_t units = ag * q.n_seg;
  k_exp_antenna<<<(unsigned)((units + kAntWarps - 1) / kAntWarps), kAntThreads, 0, s>>>(
      p->ws.rel_t, p->ws.t_base, p->n_sft, g, p->ws.perm_ant, p->ws.tauc, plan_axes(p), p->ws.i0,
      p->ws.jend, q, p->ws.agg, p->ws.coef, p->ws.flag_bits, p->ws.irr, units);
  p->launches += 1;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Plain contraction on the CUDA cores.  Tile = 128 cells: one t0 row m and
// 128 consecutive tau; they share i0, so the tile's atoms are [i0, max j).
// The weights are computed once per (cell, atom) and reused for the TC
// templates of the block; atoms are staged KC at a time in shared memory.
// ---------------------------------------------------------------------------
constexpr int kExpCells = 128;
constexpr int kKC = 32;

int64_t exp_tiles(const fmap_grid& g) {
  return (int64_t)g.n_t0 * ((g.n_tau + kExpCells - 1) / kExpCells);
}

// TAB: the weights come from the window table wtab (n_tab samples; FMAP_TABLE
// grids) instead of the exponential.
template <typename Acc, int TC, bool TAB>
__global__ void __launch_bounds__(kExpCells)
k_exp_plain(const int32_t* __restrict__ rel_t, const int64_t* __restrict__ t_base,
            int32_t n_sft, fmap_grid g, const float2* __restrict__ wtab, int32_t n_tab,
            const int64_t* __restrict__ ax,
            const int32_t* __restrict__ i0tab, const int32_t* __restrict__ jend,
            const Coef* __restrict__ coef, int32_t shared_antenna, const float* __restrict__ fafb,
            int32_t n_templates, float* __restrict__ map, Partial* __restrict__ parts,
            int64_t stride) {
  constexpr int NCOL = 4 * TC;
  constexpr int LD = NCOL + 4;
  __shared__ __align__(16) float sx[kKC][LD];
  __shared__ int32_t srel[kKC];
  __shared__ Partial scratch[kExpCells / 32];
  __shared__ int32_t s_jmax;
  const int64_t tile = blockIdx.x;
  const int32_t nblk = (g.n_tau + kExpCells - 1) / kExpCells;
  const int32_t m = (int32_t)(tile / nblk);
  const int32_t nn = (int32_t)(tile - (int64_t)m * nblk) * kExpCells + threadIdx.x;
  const bool in_grid = nn < g.n_tau;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  const int64_t cell = (int64_t)m * g.n_tau + (in_grid ? nn : 0);
  const int32_t tq0 = blockIdx.y * TC;
  const int32_t i0 = i0tab[m];
  const int32_t jc = in_grid ? jend[cell] : i0;
  if (threadIdx.x == 0) s_jmax = i0;
  __syncthreads();
  const int32_t jw = __reduce_max_sync(0xffffffffu, jc);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_jmax, jw);
  __syncthreads();
  const int32_t jmax = s_jmax;
  int32_t t0rel = 0;
  if (jmax > i0) t0rel = (int32_t)(grid_t0(g, ax, m) - *t_base);
  const double tau = (double)grid_tau(g, ax, in_grid ? nn : 0);
  const float c2 = (float)(-1.4426950408889634 / tau);
  const double su64 = TAB ? tab_scale(n_tab, exp_cut8_of(g), grid_tau(g, ax, in_grid ? nn : 0)) : 0.0;
  const float su = (float)su64;
  Acc acc[NCOL];
#pragma unroll
  for (int q = 0; q < NCOL; ++q) acc[q] = Acc(0);
  for (int32_t k0 = i0; k0 < jmax; k0 += kKC) {
    __syncthreads();
    for (int e = threadIdx.x; e < NCOL * kKC; e += kExpCells) {
      const int col = e / kKC, kk = e - col * kKC;
      const int32_t a = k0 + kk;
      const int32_t tq = tq0 + (col >> 2);
      float v = 0.0f;
      if (a < jmax && tq < n_templates) v = fafb[((int64_t)tq * 4 + (col & 3)) * n_sft + a];
      sx[kk][col] = v;
    }
    if (threadIdx.x < kKC) {
      const int32_t a = k0 + threadIdx.x;
      srel[threadIdx.x] = a < jmax ? rel_t[a] : 0;
    }
    __syncthreads();
    const int kend = min(kKC, jmax - k0);
    for (int kk = 0; kk < kend; ++kk) {
      const int32_t d = srel[kk] - t0rel;
      Acc w;
      if constexpr (TAB) {
        if constexpr (std::is_same<Acc, double>::value)
          w = (k0 + kk < jc) ? tab_weight64((double)d * su64, wtab, n_tab) : 0.0;
        else
          w = (k0 + kk < jc) ? tab_weight((float)d * su, wtab, n_tab) : 0.0f;
      } else if constexpr (std::is_same<Acc, double>::value) {
        w = (k0 + kk < jc) ? exp(-(double)d / tau) : 0.0;
      } else {
        w = (k0 + kk < jc) ? exp2f((float)d * c2) : 0.0f;
      }
      const float4* row = reinterpret_cast<const float4*>(&sx[kk][0]);
#pragma unroll
      for (int q = 0; q < NCOL / 4; ++q) {
        const float4 v = row[q];
        acc[4 * q + 0] += w * (Acc)v.x;
        acc[4 * q + 1] += w * (Acc)v.y;
        acc[4 * q + 2] += w * (Acc)v.z;
        acc[4 * q + 3] += w * (Acc)v.w;
      }
    }
  }
  const Coef cf0 = coef[cell];
#pragma unroll
  for (int q = 0; q < TC; ++q) {
    const int32_t tq = tq0 + q;
    if (tq >= n_templates) break;
    const Coef cf = shared_antenna ? cf0 : coef[(int64_t)tq * cells + cell];
    const float v = two_f(cf, (float)acc[4 * q], (float)acc[4 * q + 1], (float)acc[4 * q + 2],
                          (float)acc[4 * q + 3]);
    const bool ok = in_grid && cf.valid == 1.0f;
    if (map && in_grid && cf.valid != 2.0f) map[(int64_t)tq * cells + cell] = ok ? v : 0.0f;
    Partial pt = partial_empty();
    partial_add(pt, v, (int32_t)cell, ok);
    pt = partial_block_reduce<kExpCells / 32>(pt, scratch);
    if (threadIdx.x == 0) parts[(int64_t)tq * stride + tile] = pt;
  }
}

cudaError_t launch_exp_plain(fmap_plan_s* p, const fmap_atoms* a, float* d_2F, cudaStream_t s,
                             int64_t* tiles_used) {
  const fmap_grid& g = p->grid;
  const int64_t tiles = exp_tiles(g);
  *tiles_used = tiles;
  p->tiles = TileGeom{0, 1, kExpCells, g.n_t0, (g.n_tau + kExpCells - 1) / kExpCells};
  if (tiles == 0 || p->n_templates == 0) return cudaSuccess;
  const bool tab = g.window == FMAP_TABLE;
  auto run = [&](auto kern, int tc) {
    dim3 grid((unsigned)tiles, (unsigned)((p->n_templates + tc - 1) / tc));
    kern<<<grid, kExpCells, 0, s>>>(p->ws.rel_t, p->ws.t_base, p->n_sft, g, p->ws.wtab, p->n_tab,
                                    plan_axes(p), p->ws.i0, p->ws.jend, p->ws.coef, a->shared_antenna,
                                    a->fafb, p->n_templates, d_2F, p->ws.partials, p->part_stride);
  };
  if (p->precision == FMAP_FP64) {
    if (tab) run(k_exp_plain<double, 8, true>, 8); else run(k_exp_plain<double, 8, false>, 8);
  } else {
    if (tab) run(k_exp_plain<float, 16, true>, 16); else run(k_exp_plain<float, 16, false>, 16);
  }
  p->launches += 1;
  return cudaGetLastError();
}


// ---- persistent multi-instance dispatcher (uneven batches) ----
__global__ void __launch_bounds__(256) kb_exp_perm(const BItem* __restrict__ items, BUnits u) {
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int32_t n_x = it.perm_x ? it.T : 0;
    const int64_t total = exp_copy_entries(it.n_sft, it.n_ant, n_x, it.g.n_tau);
    const int64_t e0 = k * kPermPerUnit;
    exp_perm_body(RelStored{it.rel_t}, it.n_sft, it.antenna, it.n_ant, it.fafb, n_x, it.perm_ant, it.perm_x,
                  it.irr, it.level, it.dev_err, it.g, it.ax, it.tauc, e0 + threadIdx.x, min(total, e0 + kPermPerUnit), 256);
  });
}
// (three blocks per SM, with a few spills, against two at 110 registers: 48 uneven
// instances 707 against 766 us)
__global__ void __launch_bounds__(kAntThreads, 3) kb_exp_ant(const BItem* __restrict__ items,
                                                             BUnits u) {
  __shared__ float2 s_pw[kAntWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int64_t unit = k * kAntWarps + warp;
    if (unit >= (int64_t)it.ag.n_grp * it.n_ant * it.ag.n_seg) return;
    if (irregular(it.irr))
      exp_antenna_unit<true>(it.rel_t, it.t_base, it.n_sft, it.g, it.perm_ant, it.tauc, it.ax,
                             it.i0, it.jend, it.ag, it.agg, it.coef, it.flag_bits, unit,
                             s_pw[warp], lane);
    else
      exp_antenna_unit<false>(it.rel_t, it.t_base, it.n_sft, it.g, it.perm_ant, it.tauc, it.ax,
                              it.i0, it.jend, it.ag, it.agg, it.coef, it.flag_bits, unit,
                              s_pw[warp], lane);
  });
}
const void* batch_kernel_exp(int phase) {
  switch (phase) {
    case BP_EXP_PERM: return (const void*)kb_exp_perm;
    case BP_EXP_ANT: return (const void*)kb_exp_ant;
  }
  return nullptr;
}

}  // namespace fmap
