// Exponential window by the decayed suffix recurrence (plan flag
// FMAP_PLAN_EXP_RECURRENCE): the data sums, 2F and its reductions.
//
// fmap_sweep.cuh states the rearrangement and the mapping: a warp takes 32
// consecutive tau, a run of t0 rows from the last to the first, and G templates;
// each lane carries E at i0 and at j of its tau and advances both atom by atom.
//
// Arithmetic.  E at i0 is kept as L + Q K: K the value at the atom of the last
// renormalisation in float-float, Q the (float-float) product of the decays
// since, L the FP32 sum of the atoms since (decayed by float pairs, so that its
// rounding error is a few ulp of its own partial sums and the decays add none);
// every rec_run(N) atoms K <- L + Q K in float-float, so nothing accumulates over
// the data set.  E at j enters through
// the tail factor e^{-(t_j - t_{i0})/tau} <= e^{-3}..e^{-2} for the 3 tau cut:
// there a plain FP32 recurrence with float-pair decays (no systematic decay
// error; its random rounding error, up to 4e-6 of E for tau of thousands of SFTs, is
// scaled by the tail) is enough, as long as E at j is of the window sum's size.
// Windows cut before 3 tau, whose tail is near 1, carry E at j like E at i0.
//
// Where E at j can be much larger than the window's sum, the sweep takes care (CARE):
// both E, the tail and the difference in float-float, as in the antenna sums.  That is
// for warps whose windows may start in a long outage (they hold their last atoms only,
// and the tail is near 1), by the data's longest gap, and for data whose level varies
// more than kLevelRange-fold (a glitch behind the windows).  2F against the FP64 oracle
// at worst: in an outage of 3500 SFTs, tau of 1000-1750, 2.8e-5 without and 5e-7 with; an
// atom 4000 times the noise up to 1350 SFTs behind the windows 4.0e-5 and 3e-7; both on
// small coarse grids up to 2.7e-3 and 3e-6.  Four templates per warp take it as two pairs
// (registers); 1024 templates of 5000 SFTs, 2000 x 2000 cells: 22.9 ms, with an outage
// of 400 / 1500 SFTs 33.7 / 38.2 ms (31.9 / 38.0 without the care: gaps off the table take
// an FP64 exp), with a glitch 56 ms.  (Plain sums that start anew from the window where
// little is left of it: the same accuracy within a factor of ten, a glitch 110 ms, a band of 16
// templates 4.4 ms instead of 0.48.)
//
// A warp starts from zero at its last row's window ends and sums those windows
// first (long runs of rows, many templates), or, where the rows must be split
// into short runs to make enough warps, from the decayed sums of chunks of
// atoms formed ahead by k_sweep_agg.
//
// Bound by waits for the atoms' loads and by issue: about 340 instructions per row
// and four templates, starts included, at 42 % issue, 12 warps per SM (168 registers):
// 22.1 ms for 1024 templates x 5000 SFTs over 2000 x 2000 cells.  One block per tau with E in
// shared memory and a scan over the atoms per template (two block barriers, four
// passes over shared memory) took 73.8 ms there.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fmap_batch.cuh"
#include "fmap_sweep.cuh"

namespace fmap {

constexpr int kRecMaxSft = 9000;    // the recurrence's declared range
// Atoms between renormalisations: one in 256 of the data set, 3 to 21.  The
// FP32 sums of a run are the largest rounding error of short windows (measured
// against 64 bits, 400-630 SFTs: 1.2e-7 of the map's norm with runs of 3, 3e-7
// with 24), while a renormalisation costs 26 instructions per template.
// (A row run's first sums: kRecRun for any N.)
constexpr int32_t kRecRun = 21;
__host__ __device__ __forceinline__ int32_t rec_run(int32_t n) {
  return min(kRecRun, max(3, ((n + 255) / 256) | 1));
}
constexpr int kRecThreads = 32 * kRecWarps;
constexpr int kAggThreads = 32 * kSweepWarps;
constexpr int kRecTileRows = 32;    // t0 rows of a reduction tile (32 tau wide), at most

__device__ __forceinline__ float rec_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One atom of G templates: (re, im) pairs of Fa and Fb.
template <int G>
struct Atom {
  ulonglong2 x[G];
  // xs: the templates' strides (the last group's missing templates repeat its
  // last one)
  __device__ __forceinline__ void load(const float4* __restrict__ xp, const uint2& xs, int32_t a) {
    const uint32_t i = (uint32_t)max(a, 0);
#pragma unroll
    for (int g = 0; g < G; ++g)
      x[g] = __ldg(reinterpret_cast<const ulonglong2*>(xp) + (i + min((uint32_t)g, xs.y) * xs.x));
  }
};

// E = L + Q K of G templates (re/im pairs of Fa and Fb as f32x2).
template <int G>
struct Cursor {
  uint64_t L[G][2], Kh[G][2], Kl[G][2];
  float Qh, Qc;
  int32_t run;
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int g = 0; g < G; ++g) L[g][0] = L[g][1] = 0ull;
    Qh = 1.0f;
    Qc = 0.0f;
    run = 0;
  }
  __device__ __forceinline__ void zero() {
    reset();
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int c = 0; c < 2; ++c) Kh[g][c] = Kl[g][c] = 0ull;
  }
  // K <- L + Q K, L <- 0, Q <- 1
  __device__ __forceinline__ void renorm() {
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const FF2 k = ff2_fma_sum(L[g][c], FF{Qh, Qc}, FF2{Kh[g][c], Kl[g][c]});
        Kh[g][c] = k.h;
        Kl[g][c] = k.l;
      }
    reset();
  }
  // one atom earlier, r its decay
  __device__ __forceinline__ void step(FF r, const Atom<G>& a) {
    const uint64_t rh = pk2(r.h, r.h), rl = pk2(r.l, r.l);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      L[g][0] = fma2(rh, L[g][0], fma2(rl, L[g][0], a.x[g].x));
      L[g][1] = fma2(rh, L[g][1], fma2(rl, L[g][1], a.x[g].y));
    }
    ch_mul(r, Qh, Qc);
    ++run;
  }
  // E as float pairs / in FP32
  __device__ __forceinline__ void set(int g, int c, const FF2& v) {
    Kh[g][c] = v.h;
    Kl[g][c] = v.l;
  }
  __device__ __forceinline__ uint64_t scale() const { return pk2(Qh + Qc, Qh + Qc); }
  __device__ __forceinline__ uint64_t get(int g, int c, uint64_t q) const {
    return fma2(q, Kh[g][c], L[g][c]);
  }
};
// E of G templates by the plain recurrence with float-pair decays.
template <int G>
struct PlainCursor {
  uint64_t E[G][2];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int g = 0; g < G; ++g) E[g][0] = E[g][1] = 0ull;
  }
  __device__ __forceinline__ void step(FF r, const Atom<G>& a) {
    const uint64_t rh = pk2(r.h, r.h), rl = pk2(r.l, r.l);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      E[g][0] = fma2(rh, E[g][0], fma2(rl, E[g][0], a.x[g].x));
      E[g][1] = fma2(rh, E[g][1], fma2(rl, E[g][1], a.x[g].y));
    }
  }
  __device__ __forceinline__ void set(int g, int c, const FF2& v) { E[g][c] = v.h; }
  __device__ __forceinline__ uint64_t scale() const { return 0ull; }
  __device__ __forceinline__ uint64_t get(int g, int c, uint64_t) const { return E[g][c]; }
};

// E of G templates in float-float, an atom at a time (the careful sweep).
template <int G>
struct CareCursor {
  uint64_t Kh[G][2], Kl[G][2];
  static constexpr int32_t run = 0;
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int c = 0; c < 2; ++c) Kh[g][c] = Kl[g][c] = 0ull;
  }
  __device__ __forceinline__ void renorm() {}
  __device__ __forceinline__ void step(FF r, const Atom<G>& a) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      set(g, 0, ff2_fma_sum(a.x[g].x, r, FF2{Kh[g][0], Kl[g][0]}));
      set(g, 1, ff2_fma_sum(a.x[g].y, r, FF2{Kh[g][1], Kl[g][1]}));
    }
  }
  __device__ __forceinline__ void set(int g, int c, const FF2& v) {
    Kh[g][c] = v.h;
    Kl[g][c] = v.l;
  }
};
// E at i0 - tail E at j
template <int G>
__device__ __forceinline__ uint64_t care_diff(const CareCursor<G>& i, const CareCursor<G>& j, int g,
                                              int c, FF tail) {
  const FF2 d = ff2_fma_sum(i.Kh[g][c], FF{-tail.h, -tail.l}, FF2{j.Kh[g][c], j.Kl[g][c]});
  return add2(d.h, add2(d.l, i.Kl[g][c]));
}
// 1 / r for a decay r in (0, 1] that is not tiny
__device__ __forceinline__ FF ff_rcp(FF r) {
  const float y = __frcp_rn(r.h);
  return fast_two_sum(y, y * fmaf(-r.l, y, fmaf(-r.h, y, 1.0f)));
}

struct RecArgs {
  const int32_t* rel_t;
  const int64_t* t_base;
  const int32_t* irr;   // any word nonzero: some gap has code 0
  const uint32_t* level;   // the data's range of levels (level_note)
  int32_t n, T;
  fmap_grid g;
  RecGeom q;
  const int32_t* i0tab;
  const int32_t* jend;
  const Coef* coef;
  const float4* x;      // [T][n]
  const TauTab* tauc;
  const int64_t* ax;
  float* agg;           // chunk maps: S [T][n_grp][n_chunks][8][32], then R [n_grp][n_chunks][2][32]
  float* map;
  Partial* parts;
  int64_t stride;
};
__device__ __forceinline__ float* rec_agg_r(const RecArgs& A) {
  return A.agg + (int64_t)A.T * A.q.n_grp * A.q.n_chunks * 256;
}

__device__ __forceinline__ uint32_t gap_inverse(int32_t t_sft) {
  return (uint32_t)(((1ull << 31) + (uint32_t)t_sft - 1) / (uint32_t)t_sft);
}
// Relative time of atom a; one SFT past the last for a = n (E is zero there).
__device__ __forceinline__ int32_t atom_time(const RecArgs& A, int32_t a) {
  return a < A.n ? __ldg(A.rel_t + a) : __ldg(A.rel_t + A.n - 1) + (int32_t)A.g.t_sft;
}

// Whether the sweep of a group of 32 tau takes care (see the top).  A window whose tail is
// above 1/4 ends within 1.4 tau of its first atom: its t0 lies in a gap of more than the
// rest of its length (of shorter ones, more than half of it); gap: the data's longest.
__device__ __forceinline__ bool rec_careful(const RecArgs& A, int32_t grp, int32_t gap) {
  const float cut = (float)exp_cut8_of(A.g) / 8.0f, rest = fmaxf(cut - 1.4f, 0.5f * cut);
  return (gap > 0 && (float)gap > rest * (float)grid_tau(A.g, A.ax, grp * 32)) || level_varies(A.level);
}

// Chunk maps of one (template group, 32 tau, chunk): E[first] = S + R E[next].
template <int G, bool IRR>
__device__ __forceinline__ void rec_agg_unit(const RecArgs& A, int64_t unit, float2* s_pw,
                                             int lane) {
  const RecGeom& q = A.q;
  const int32_t tg0 = (int32_t)(unit % q.n_tgrp) * G;
  const int64_t u1 = unit / q.n_tgrp;
  const int32_t ch = (int32_t)(u1 % q.n_chunks);
  const int32_t grp = (int32_t)(u1 / q.n_chunks);
  const TauTab* tt = A.tauc + min(grp * 32 + lane, A.g.n_tau - 1);
  sweep_tab_load<1>(s_pw, tt, lane);
  const int32_t n_t = min(G, A.T - tg0);
  const float4* x = A.x + (int64_t)tg0 * A.n;
  const uint2 xs = make_uint2((uint32_t)A.n, (uint32_t)(n_t - 1));
  const int32_t lo = ch * q.chunk, hi = min(A.n, lo + q.chunk);
  const int32_t run = rec_run(A.n);
  const bool care = rec_careful(A, grp, longest_gap(A.irr));   // every atom in float-float
  Cursor<G> E;
  E.zero();
  FF R{1.0f, 0.0f};
  const int32_t t_sft = (int32_t)A.g.t_sft;
  const uint32_t inv = gap_inverse(t_sft);
  int32_t tn = atom_time(A, hi);
  constexpr int B = G == 4 ? 2 : 4;   // atoms loaded ahead of the serial chain
  for (int32_t a1 = hi; a1 > lo; a1 -= B) {
    Atom<G> at[B];
    int32_t t[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      at[u].load(x, xs, a1 - 1 - u);
      t[u] = __ldg(A.rel_t + max(a1 - 1 - u, 0));
    }
#pragma unroll
    for (int u = 0; u < B; ++u) {
      if (a1 - 1 - u < lo) break;
      E.step(sweep_gap_decay<1, IRR>(s_pw, tn - t[u], inv, t_sft, lane, tt), at[u]);
      tn = t[u];
      if (care) {
        R = ff_mul(R, FF{E.Qh, E.Qc});
        E.renorm();
      }
    }
    if (E.run >= run) {
      R = ff_mul(R, FF{E.Qh, E.Qc});
      E.renorm();
    }
  }
  R = ff_mul(R, FF{E.Qh, E.Qc});
  E.renorm();
#pragma unroll
  for (int k = 0; k < G; ++k) {
    if (k >= n_t) break;
    float* o = A.agg + (((int64_t)(tg0 + k) * q.n_grp + grp) * q.n_chunks + ch) * 256 + lane;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      up2(E.Kh[k][c], o[128 * c], o[128 * c + 32]);
      up2(E.Kl[k][c], o[128 * c + 64], o[128 * c + 96]);
    }
  }
  if (tg0 == 0) {
    float* o = rec_agg_r(A) + ((int64_t)grp * q.n_chunks + ch) * 64 + lane;
    o[0] = R.h;
    o[32] = R.l;
  }
}

// SHORT: windows cut before 3 tau.  SH: coefficients shared by the templates.
// IRR: some gap is not 1..15 whole SFTs.  CARE: see the top.  The unit's templates
// from tg0 on; u1: its rows and tau.
template <int G, bool SHORT, bool SH, bool IRR, bool CARE>
__device__ __forceinline__ void exp_rec_unit(const RecArgs& A, int32_t tg0, int64_t u1,
                                             float2* s_pw, int lane) {
  const fmap_grid& g = A.g;
  const RecGeom& q = A.q;
  constexpr int NC = SH ? 1 : G;   // coefficient sets
  // each cursor's next atom is loaded a step ahead, where registers allow
  constexpr bool PF = G < 4;
  constexpr bool END = SHORT && !CARE;   // E at j is carried like E at i0
  static_assert(PF || !(SHORT || CARE), "four templates: the 3 tau cut, level data");
  const int32_t seg = (int32_t)(u1 % q.n_seg);
  const int32_t grp = q.n_grp - 1 - (int32_t)(u1 / q.n_seg);
  const int32_t n = A.n, n_tau = g.n_tau, run = rec_run(n);
  const int32_t ni = grp * 32 + lane, nn = min(ni, n_tau - 1);
  const bool in_grid = ni < n_tau;
  const int32_t m_lo = seg * q.rows, m_hi = min(g.n_t0, m_lo + q.rows);
  const int32_t n_t = min(G, A.T - tg0);        // templates present
  const TauTab* tt = A.tauc + nn;
  sweep_tab_load<1>(s_pw, tt, lane);
  const float c2 = tt->c2[0];
  const int64_t cells = (int64_t)g.n_t0 * n_tau;
  const int64_t tb = n > 0 ? *A.t_base : 0;
  const float4* x = A.x + (int64_t)tg0 * n;
  const uint2 xs = make_uint2((uint32_t)n, (uint32_t)(n_t - 1));
  const int32_t t_sft = (int32_t)g.t_sft;
  const uint32_t inv = gap_inverse(t_sft);
  int32_t i0 = A.i0tab[m_hi - 1], j = A.jend[(int64_t)(m_hi - 1) * n_tau + nn];
  typename std::conditional<CARE, CareCursor<G>, Cursor<G>>::type Ei;
  Ei.zero();
  typename std::conditional<CARE, CareCursor<G>,
                            typename std::conditional<END, Cursor<G>, PlainCursor<G>>::type>::type Ej;
  Ej.zero();
  // CARE: the tail factor in float-float, by the decays that the cursors pass; lost: too
  // small a decay or tail to go on from (formed anew by an FP64 exp when it counts again)
  constexpr float kTailLost = 1e-18f, kDecayLost = 1e-6f;
  FF tail_ff{0.0f, 0.0f};
  bool lost = true;
  int32_t run_j = 0;   // END: the most atoms a lane's Ej took since its renormalisation
  int32_t ic, jc;
  if (q.n_chunks > 0) {
    // E at the first atoms of the chunks after those holding j and i0
    const int32_t bj = (j + q.chunk - 1) / q.chunk, bi = (i0 + q.chunk - 1) / q.chunk;
    FF2 E[G][2];
#pragma unroll
    for (int k = 0; k < G; ++k) E[k][0] = E[k][1] = FF2{0ull, 0ull};
    const float* ro = rec_agg_r(A) + (int64_t)grp * q.n_chunks * 64 + lane;
    const float* so = A.agg + ((int64_t)tg0 * q.n_grp + grp) * q.n_chunks * 256 + lane;
    const int64_t sk = (int64_t)q.n_grp * q.n_chunks * 256;
    constexpr int B = G == 1 ? 4 : 1;   // chunk maps loaded ahead
    for (int32_t b0 = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)bj);; b0 -= B) {
      FF R[B];
      float v[B][G][8];
#pragma unroll
      for (int u = 0; u < B; ++u) {
        const int32_t c = max(b0 - 1 - u, 0);
        R[u] = {ro[c * 64], ro[c * 64 + 32]};
#pragma unroll
        for (int k = 0; k < G; ++k)
#pragma unroll
          for (int e = 0; e < 8; ++e) v[u][k][e] = so[(int64_t)c * 256 + min(k, n_t - 1) * sk + 32 * e];
      }
      bool done = false;
#pragma unroll
      for (int u = 0; u < B; ++u) {
        const int32_t b = b0 - u;
        if (b == bj) {
#pragma unroll
          for (int k = 0; k < G; ++k) {
            Ej.set(k, 0, E[k][0]);
            Ej.set(k, 1, E[k][1]);
          }
        }
        if (b <= bi) {
          done = true;
          break;
        }
#pragma unroll
        for (int k = 0; k < G; ++k)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float* w = &v[u][k][4 * c];
            const FF2 p = ff2_fma_sum(pk2(w[0], w[1]), R[u], E[k][c]);
            E[k][c] = fast_two_sum2(p.h, add2(p.l, pk2(w[2], w[3])));
          }
      }
      if (done) break;
    }
#pragma unroll
    for (int k = 0; k < G; ++k) {
      Ei.set(k, 0, E[k][0]);
      Ei.set(k, 1, E[k][1]);
    }
    ic = min(n, bi * q.chunk);
    jc = min(n, bj * q.chunk);
  } else {
    // E starts from zero at each lane's window end of the last row
    jc = j;
    ic = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)j);
    const int32_t j_all = (int32_t)__reduce_min_sync(0xffffffffu, (unsigned)j);
    int32_t tn = n > 0 ? atom_time(A, ic) : 0;
    for (const int32_t end = max(i0, j_all); ic > end;) {   // atoms past some lanes' ends
      // (without a renormalisation the FP32 sums span up to 31 tau steps: 2F of the
      // first rows off by 3.4e-7 rms at steps of 30 SFTs, against 1.3e-7)
      const int32_t stop = max(end, ic - kRecRun);
      while (ic > stop) {
        --ic;
        Atom<G> at;
        at.load(x, xs, ic);
        const int32_t t = __ldg(A.rel_t + ic);
        const FF r = sweep_gap_decay<1, IRR>(s_pw, tn - t, inv, t_sft, lane, tt);
        tn = t;
        if (ic < j) Ei.step(r, at);
      }
      Ei.renorm();   // (the lanes' runs differ: from here they are equal)
    }
  }
  // times of the cursors' atoms, and of the next ones (loaded a step ahead)
  int32_t ti = n > 0 ? atom_time(A, ic) : 0, tj = n > 0 ? atom_time(A, jc) : 0;
  int32_t ei = n > 0 ? __ldg(A.rel_t + max(ic - 1, 0)) : 0;
  int32_t ej = n > 0 ? __ldg(A.rel_t + max(jc - 1, 0)) : 0;
  Atom<G> ai, aj;
  if (PF) {
    ai.load(x, xs, ic - 1);
    aj.load(x, xs, jc - 1);
  } else {   // to the last row's window (below, the first row's loop does it)
    Atom<G> at;
    at.load(x, xs, ic - 1);
    while (ic > i0) {
      --ic;
      const Atom<G> cur = at;
      const int32_t t = ei;
      at.load(x, xs, ic - 1);
      ei = __ldg(A.rel_t + max(ic - 1, 0));
      Ei.step(sweep_gap_decay<1, IRR>(s_pw, ti - t, inv, t_sft, lane, tt), cur);
      ti = t;
      if (Ei.run >= run) Ei.renorm();
    }
  }
  // per template and tile: maximum, its row, sum of e^{(v - maximum) / 2};
  // valid cells
  float M[G], sum[G];
  int32_t arg[G], nv[NC];
  auto clear = [&]() {
#pragma unroll
    for (int k = 0; k < G; ++k) {
      M[k] = -1.0f;
      sum[k] = 0.0f;
      arg[k] = 0;
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) nv[k] = 0;
  };
  clear();
  constexpr float kHalfLog2e = 0.72134752044448170368f;   // log2(e) / 2
  const uint64_t tiny2 = pk2(1e-30f, 1e-30f);
  int32_t m_flush = ((m_hi - 1) / q.tile_rows) * q.tile_rows;   // the tile's first row
  int64_t t0r = grid_t0(g, A.ax, m_hi - 1) - tb;
  uint32_t cell = (uint32_t)(m_hi - 1) * (uint32_t)n_tau + (uint32_t)nn;   // (cells < 2^31)
  const float4* cp = reinterpret_cast<const float4*>(A.coef) + (SH ? 0 : (int64_t)tg0 * cells);
  float4 cf[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) cf[k] = __ldg(cp + min(k, n_t - 1) * cells + cell);
  float* const mp = A.map ? A.map + (int64_t)tg0 * cells : nullptr;
  const bool store = mp && in_grid;
  for (int32_t m = m_hi - 1; m >= m_lo; --m) {
    if (!PF) {   // the atoms this row most often steps over, before anything waits
      ai.load(x, xs, ic - 1);
      aj.load(x, xs, jc - 1);
    }
    int32_t i0n = 0, jn = 0;
    float4 cn[NC];
    if (m > m_lo) {
      i0n = __ldg(A.i0tab + (m - 1));
      jn = __ldg(A.jend + (cell - (uint32_t)n_tau));
#pragma unroll
      for (int k = 0; k < NC; ++k)
        cn[k] = __ldg(cp + min(k, n_t - 1) * cells + (cell - (uint32_t)n_tau));
    }
    if constexpr (PF) {
      while (ic > i0) {
        --ic;
        const Atom<G> cur = ai;
        const int32_t t = ei;
        ei = __ldg(A.rel_t + max(ic - 1, 0));
        ai.load(x, xs, ic - 1);
        const FF r = sweep_gap_decay<1, IRR>(s_pw, ti - t, inv, t_sft, lane, tt);
        Ei.step(r, cur);
        if constexpr (CARE) {
          tail_ff = ff_mul(tail_ff, r);
          lost |= r.h < kDecayLost || tail_ff.h < kTailLost;
        }
        ti = t;
        if (Ei.run >= run) Ei.renorm();
      }
      // (END: the lanes step together, so that they renormalise together)
      while (END ? __any_sync(0xffffffffu, jc > j) : jc > j) {
        if (!END || jc > j) {
          --jc;
          const Atom<G> cur = aj;
          const int32_t t = ej;
          ej = __ldg(A.rel_t + max(jc - 1, 0));
          aj.load(x, xs, jc - 1);
          const FF r = sweep_gap_decay<1, IRR>(s_pw, tj - t, inv, t_sft, lane, tt);
          Ej.step(r, cur);
          if constexpr (CARE) {
            tail_ff = ff_mul(tail_ff, ff_rcp(r));
            lost |= r.h < kDecayLost;
          }
          tj = t;
        }
        if constexpr (END)
          if (++run_j >= run) {
            Ej.renorm();
            run_j = 0;
          }
      }
    } else {
      const FF ri = sweep_gap_decay<1, IRR>(s_pw, ti - ei, inv, t_sft, lane, tt);
      const FF rj = sweep_gap_decay<1, IRR>(s_pw, tj - ej, inv, t_sft, lane, tt);
      if (ic > i0) {
        --ic;
        Ei.step(ri, ai);
        ti = ei;
        while (ic > i0) {
          --ic;
          ei = __ldg(A.rel_t + ic);
          ai.load(x, xs, ic);
          Ei.step(sweep_gap_decay<1, IRR>(s_pw, ti - ei, inv, t_sft, lane, tt), ai);
          ti = ei;
          if (Ei.run >= run) Ei.renorm();
        }
        ei = __ldg(A.rel_t + max(ic - 1, 0));
        if (Ei.run >= run) Ei.renorm();
      }
      if (jc > j) {
        --jc;
        Ej.step(rj, aj);
        tj = ej;
        while (jc > j) {
          --jc;
          ej = __ldg(A.rel_t + jc);
          aj.load(x, xs, jc);
          Ej.step(sweep_gap_decay<1, IRR>(s_pw, tj - ej, inv, t_sft, lane, tt), aj);
          tj = ej;
        }
        ej = __ldg(A.rel_t + max(jc - 1, 0));
      }
    }
    // Tail factor and squared prefactor of the window [i0, j) (an empty one is
    // invalid).  Approximate FP32 exp2 for the tail: ~e^{-3} of the window sum
    // for the default 3 tau cut.  Windows cut before 3 tau make it large, where
    // the difference E[i0] - tail E[j] loses 1 / (1 - tail): there a tail
    // above 1/2 comes from the correctly rounded-to-1-ulp exp2f.
    const float dj = (float)(tj - ti), xj = c2 * dj;
    float tail = rec_ex2(xj);
    if (END && tail > 0.5f) tail = exp2f(xj);
    if constexpr (CARE) {
      lost |= tail < kTailLost;
      if (lost) {
        tail_ff = FF{tail, 0.0f};
        if (tail >= kTailLost) {
          const float2 v = slow_decay(tj - ti, tt->inv_tau);
          tail_ff = FF{v.x, v.y};
          lost = false;
        }
      }
    }
    float pre2 = 1.0f;
    const int32_t d0 = (int32_t)(ti - t0r);
    if (d0 != 0) {
      const float pre = rec_ex2(c2 * (float)d0);
      pre2 = pre * pre;
    }
    uint64_t qi = 0ull, qj = 0ull;
    const uint64_t nt = pk2(-tail, -tail);
    if constexpr (!CARE) {
      qi = Ei.scale();
      qj = Ej.scale();
    }
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const float4 c = cf[SH ? 0 : k];
      // cells that take no part (invalid, or left to the fix-up): -inf, which
      // no maximum takes, whose exp-term is 0 and whose map entry is 0
      const bool ok = c.w == 1.0f && in_grid;
      const float k1 = ok ? c.x * pre2 : -INFINITY, k2 = ok ? c.z * pre2 : 0.0f;
      if (SH ? k == 0 : true) nv[SH ? 0 : k] += ok ? 1 : 0;
      uint64_t f0, f1;
      if constexpr (CARE) {
        f0 = care_diff(Ei, Ej, k, 0, tail_ff);
        f1 = care_diff(Ei, Ej, k, 1, tail_ff);
      } else {
        f0 = fma2(nt, Ej.get(k, 0, qj), Ei.get(k, 0, qi));
        f1 = fma2(nt, Ej.get(k, 1, qj), Ei.get(k, 1, qi));
      }
      const float v = two_f_pairs(f0, f1, pk2(-c.y, -c.y), k1, k2, tiny2);
      if (store && k < n_t) (mp + k * cells)[cell] = fmaxf(v, 0.0f);
      // rows come in descending order: the later one wins a tie
      const float ex = rec_ex2(fabsf(v - M[k]) * -kHalfLog2e);
      const bool up = v >= M[k];
      sum[k] = up ? fmaf(sum[k], ex, 1.0f) : sum[k] + ex;
      M[k] = fmaxf(M[k], v);
      arg[k] = up ? m : arg[k];
    }
    if (m == m_flush) {   // one partial per (template, tile)
      m_flush -= q.tile_rows;
      const int64_t slot = (int64_t)(m / q.tile_rows) * q.n_grp + grp;
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const Partial r = partial_warp_reduce(
            Partial{M[k], arg[k] * n_tau + ni, sum[k], nv[SH ? 0 : k]});
        if (lane == 0 && k < n_t) A.parts[(int64_t)(tg0 + k) * A.stride + slot] = r;
      }
      clear();
    }
    i0 = i0n;
    j = jn;
#pragma unroll
    for (int k = 0; k < NC; ++k) cf[k] = cn[k];
    cell -= (uint32_t)n_tau;
    t0r = A.ax ? (m > m_lo ? A.ax[m - 1] - tb : 0) : t0r - g.dt0;
  }
}

// unit: template groups fastest (they share the rows' indices and coefficients),
// then row runs, then tau from the longest windows down.
// Sweeps of data that is not regular, out of line: their registers and instructions
// stay out of the others' (in a plan's kernel the careful one only: one gap of 20 SFTs
// in 1024 templates' data 27.7 ms, 34.4 with both; in a batch's both: 48 uneven
// instances 2808 us, 2878 with one).  G templates from tg0 on, up to tg1.
template <int G, bool SHORT, bool SH, bool CARE>
__device__ __noinline__ void rec_unit_apart(const RecArgs& A, int32_t tg0, int32_t tg1, int64_t u1,
                                            float2* s_pw, int lane) {
  for (int32_t t0 = tg0; t0 < tg1; t0 += G)
    exp_rec_unit<G, SHORT, SH, true, CARE>(A, t0, u1, s_pw, lane);
}
template <int G, bool SHORT, bool SH, bool BATCH>
__device__ __forceinline__ void rec_unit(const RecArgs& A, int64_t unit, float2* s_pw, int lane) {
  const int32_t tg0 = (int32_t)(unit % A.q.n_tgrp) * G;
  const int64_t u1 = unit / A.q.n_tgrp;
  const int32_t gap = longest_gap(A.irr);
  if (!gap && !level_varies(A.level))
    return exp_rec_unit<G, SHORT, SH, false, false>(A, tg0, u1, s_pw, lane);
  if (rec_careful(A, A.q.n_grp - 1 - (int32_t)(u1 / A.q.n_seg), gap)) {
    const RecArgs B = A;   // (its address is taken)
    return rec_unit_apart<G < 4 ? G : 2, SHORT, SH, true>(B, tg0, min(tg0 + G, A.T), u1, s_pw, lane);
  }
  if constexpr (BATCH) {
    const RecArgs B = A;
    rec_unit_apart<G, SHORT, SH, false>(B, tg0, min(tg0 + G, A.T), u1, s_pw, lane);
  } else {
    exp_rec_unit<G, SHORT, SH, true, false>(A, tg0, u1, s_pw, lane);
  }
}

// (registers: the state of four templates takes about 160, of one about 100)
template <int G, bool SHORT, bool SH>
__global__ void __launch_bounds__(kRecThreads, G == 4 ? 3 : G == 2 ? 4 : 5)
k_exp_rec(const RecArgs A, int64_t units) {
  __shared__ float2 s_pw[kRecWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t unit = (int64_t)blockIdx.x * kRecWarps + warp;
  if (unit >= units) return;
  rec_unit<G, SHORT, SH, false>(A, unit, s_pw[warp], lane);
}
// Chunk maps of the antenna rows (units [0, ant_units)), then of the data.
struct AntAgg {
  const float4* ant;
  float* agg;
  AntGeom q;
  int64_t units;
};
template <int G, bool IRR>
__device__ __forceinline__ void sweep_agg_unit(const RecArgs& A, const AntAgg& N, int64_t unit,
                                               float2* s_pw, int lane) {
  if (unit < N.units)
    exp_agg_unit<IRR>(A.rel_t, A.n, N.ant, A.tauc, A.g, N.q, N.agg, unit, s_pw, lane);
  else
    rec_agg_unit<G, IRR>(A, unit - N.units, s_pw, lane);
}
template <int G>
__global__ void __launch_bounds__(kAggThreads)
k_sweep_agg(const RecArgs A, const AntAgg N, int64_t units) {
  __shared__ float2 s_pw[kSweepWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t unit = (int64_t)blockIdx.x * kSweepWarps + warp;
  if (unit >= units) return;
  if (irregular(A.irr)) sweep_agg_unit<G, true>(A, N, unit, s_pw[warp], lane);
  else sweep_agg_unit<G, false>(A, N, unit, s_pw[warp], lane);
}

bool exp_rec_supported(int32_t n_sft, int32_t) { return n_sft <= kRecMaxSft; }

// The work split, by a count of issue slots (as measured, at the issue rate
// each form reaches: 233 instructions a row at 40 % for two templates, 352 at 36 %
// for four).  A warp's start costs the window's atoms, or the composition of
// half the chunk maps and the atoms of a chunk for each cursor.  A scheduler needs
// about three warps to hide the latencies: below that, time goes with one warp's
// work.
RecGeom rec_geom(const fmap_grid& g, int32_t n_sft, int32_t T, bool shared, bool batch, int32_t tpb,
                 int64_t agg_room) {
  RecGeom best{};
  double best_t = 0.0;
  const int32_t n_grp = std::max(1, (g.n_tau + 31) / 32);
  // (four templates per warp only with coefficients in common and the 3 tau cut,
  // by registers)
  int32_t g_max = shared && exp_cut8_of(g) >= 24 ? 4 : 2;
  if (tpb > 0) g_max = std::min(g_max, tpb);
  double win = 0.0;   // atoms of the windows, averaged over tau
  for (int k = 0; k < 16; ++k) {
    const int64_t tau = g.tau_min + (int64_t)std::max(0, g.n_tau - 1) * k / 15 * g.dtau;
    win += std::min<double>(n_sft, (double)window_len(g, tau) / (double)g.t_sft) / 16.0;
  }
  const double more = g.n_t0 > 1 ? std::min<double>((double)n_sft, std::max(0.0, (double)g.dt0 / (double)g.t_sft - 1.0))
                                 : 0.0;
  const int32_t chunk0 = n_sft <= 512 ? 16 : n_sft <= 1024 ? 32 : n_sft <= 4096 ? 64 : 128;
  const double slots = kSms * 4.0;
  // (a batch's instances run side by side: runs of 48 rows, or of as much work where
  // a row's step spans several SFTs: 44 instances of up to 456 x 456 cells and 5329
  // SFTs 1319 -> 951 us)
  const double batch_rows = std::max(8.0, 48.0 * 360.0 / (360.0 + 110.0 * more));
  for (int G = 1; G <= g_max && (G == 1 || G <= T); G *= 2) {
    const int32_t tgrp = std::max(1, (T + G - 1) / G);
    if (G == 4 && (double)n_grp * tgrp < slots) break;   // (few warps per scheduler: two templates)
    for (int maps = 0; maps < 4; ++maps) {   // none, or chunks of chunk0, 2 chunk0, 4 chunk0
      const int32_t chunk = chunk0 << std::max(0, maps - 1);
      const int32_t n_chunks = (n_sft + chunk - 1) / chunk;
      // chunk maps only where there are few warps, and room for them
      if (maps && (n_sft == 0 || (!batch && (int64_t)n_grp * T > 4096) ||
                   4 * (int64_t)n_grp * n_chunks * ((int64_t)T * 256 + 64) > agg_room))
        continue;
      const double start = maps ? 0.5 * n_chunks * (30.0 + 90.0 * G) + 1.5 * chunk * (40.0 + 30.0 * G)
                                : win * (40.0 + 30.0 * G);
      const double ahead = maps ? chunk * (60.0 + 35.0 * G) *
                                      std::max(3.0, (double)n_grp * tgrp * n_chunks / slots)
                                : 0.0;
      for (int32_t seg = 1; seg <= 256; seg = seg < 4 ? seg + 1 : seg + seg / 3) {
        const int32_t rows = (g.n_t0 + seg - 1) / seg;
        if (seg > 1 && rows < 4) break;
        if (batch && seg > 1 && rows < batch_rows) break;
        const double work = start + rows * (150.0 + 210.0 * G + more * (60.0 + 50.0 * G));
        // a batch has other instances to fill the GPU: total work counts
        const double t = ahead + work * (batch ? (double)n_grp * tgrp * seg / slots + 0.3
                                               : std::max(3.0, (double)n_grp * tgrp * seg / slots));
        if (best.G == 0 || t < best_t) {
          best_t = t;
          best.G = G;
          best.rows = std::max(1, rows);
          best.chunk = maps ? chunk : 0;
          best.n_chunks = maps ? n_chunks : 0;
        }
      }
    }
  }
  RecGeom& q = best;
  q.n_grp = n_grp;
  if (q.rows > kRecTileRows) q.rows = (q.rows + kRecTileRows - 1) / kRecTileRows * kRecTileRows;
  q.tile_rows = std::min(q.rows, kRecTileRows);
  q.n_seg = std::max(1, (g.n_t0 + q.rows - 1) / q.rows);
  q.ntr = std::max(1, (g.n_t0 + q.tile_rows - 1) / q.tile_rows);
  q.n_tgrp = std::max(1, (T + q.G - 1) / q.G);
  return q;
}
// (the data's chunk maps follow the antenna rows')
static RecArgs rec_args(const fmap_plan_s* p, const RecGeom& q, const AntGeom& a, int64_t n_ant,
                        float* d_2F) {
  return RecArgs{p->ws.rel_t, p->ws.t_base, p->ws.irr, p->ws.level, p->n_sft, p->n_templates, p->grid, q,
                 p->ws.i0, p->ws.jend, p->ws.coef, p->ws.perm_x, p->ws.tauc,
                 plan_axes(p), p->ws.agg + ant_agg_floats(a, n_ant), d_2F, p->ws.partials, p->part_stride};
}

cudaError_t launch_exp_agg(fmap_plan_s* p, const fmap_atoms* a, cudaStream_t s) {
  const fmap_grid& g = p->grid;
  const int n_ant = a->shared_antenna ? 1 : p->n_templates;
  if ((int64_t)g.n_t0 * g.n_tau == 0 || n_ant == 0 || p->n_sft == 0) return cudaSuccess;
  AntAgg N{p->ws.perm_ant, p->ws.agg, p->ant[a->shared_antenna ? 1 : 0], 0};
  N.units = (int64_t)N.q.n_grp * n_ant * N.q.n_chunks;
  RecGeom q{};
  q.G = 1;
  if ((p->flags & FMAP_PLAN_EXP_RECURRENCE) && p->n_templates > 0)
    q = p->rec[a->shared_antenna ? 1 : 0];
  const int64_t units = N.units + (int64_t)q.n_grp * q.n_chunks * q.n_tgrp;
  if (units == 0) return cudaSuccess;
  const RecArgs A = rec_args(p, q, N.q, n_ant, nullptr);
  auto run = [&](auto kern) {
    kern<<<(unsigned)((units + kSweepWarps - 1) / kSweepWarps), kAggThreads, 0, s>>>(A, N, units);
  };
  q.G == 1 ? run(k_sweep_agg<1>) : q.G == 2 ? run(k_sweep_agg<2>) : run(k_sweep_agg<4>);
  p->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_exp_rec(fmap_plan_s* p, const fmap_atoms* a, float* d_2F, cudaStream_t s,
                           int64_t* tiles_used) {
  const fmap_grid& g = p->grid;
  *tiles_used = 0;
  if ((int64_t)g.n_t0 * g.n_tau == 0 || p->n_templates == 0) return cudaSuccess;
  const RecGeom q = p->rec[a->shared_antenna ? 1 : 0];
  *tiles_used = (int64_t)q.ntr * q.n_grp;
  p->tiles = TileGeom{0, q.tile_rows, 32, q.ntr, q.n_grp};
  const RecArgs A = rec_args(p, q, p->ant[a->shared_antenna ? 1 : 0],
                             a->shared_antenna ? 1 : p->n_templates, d_2F);
  auto run = [&](auto kern, int64_t units) {
    kern<<<(unsigned)((units + kRecWarps - 1) / kRecWarps), kRecThreads, 0, s>>>(A, units);
    p->launches += 1;
  };
  const int64_t units = (int64_t)q.n_grp * q.n_seg * q.n_tgrp;
  const bool brief = exp_cut8_of(g) < 24;
  auto pick = [&](auto one, auto two, auto four) {
    q.G == 1 ? run(one, units) : q.G == 2 ? run(two, units) : run(four, units);
  };
  if (a->shared_antenna)
    brief ? pick(k_exp_rec<1, true, true>, k_exp_rec<2, true, true>, k_exp_rec<2, true, true>)
          : pick(k_exp_rec<1, false, true>, k_exp_rec<2, false, true>, k_exp_rec<4, false, true>);
  else
    brief ? pick(k_exp_rec<1, true, false>, k_exp_rec<2, true, false>, k_exp_rec<2, true, false>)
          : pick(k_exp_rec<1, false, false>, k_exp_rec<2, false, false>, k_exp_rec<2, false, false>);
  return cudaGetLastError();
}


// ---- persistent multi-instance dispatchers (uneven batches) ----
static __device__ __forceinline__ RecArgs rec_args(const BItem& it) {
  return RecArgs{it.rel_t, it.t_base, it.irr, it.level, it.n_sft, it.T, it.g, it.rg, it.i0, it.jend, it.coef,
                 it.perm_x, it.tauc, it.ax, it.agg + ant_agg_floats(it.ag, it.n_ant), it.map,
                 it.partials, it.part_stride};
}
__global__ void __launch_bounds__(kAggThreads, 2) kb_sweep_agg(const BItem* __restrict__ items,
                                                               BUnits u) {
  __shared__ float2 s_pw[kSweepWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int64_t unit = k * kSweepWarps + warp;
    const AntAgg N{it.perm_ant, it.agg, it.ag, (int64_t)it.ag.n_grp * it.n_ant * it.ag.n_chunks};
    if (unit >= N.units + (int64_t)it.rg.n_grp * it.rg.n_chunks * it.rg.n_tgrp) return;
    const RecArgs A = rec_args(it);
    if (it.rg.G == 1) {
      if (irregular(it.irr)) sweep_agg_unit<1, true>(A, N, unit, s_pw[warp], lane);
      else sweep_agg_unit<1, false>(A, N, unit, s_pw[warp], lane);
    } else if (it.rg.G == 2) {
      if (irregular(it.irr)) sweep_agg_unit<2, true>(A, N, unit, s_pw[warp], lane);
      else sweep_agg_unit<2, false>(A, N, unit, s_pw[warp], lane);
    } else {
      if (irregular(it.irr)) sweep_agg_unit<4, true>(A, N, unit, s_pw[warp], lane);
      else sweep_agg_unit<4, false>(A, N, unit, s_pw[warp], lane);
    }
  });
}
// MAXG: the most templates per warp of the wave's instances (registers).  Three
// blocks per SM: the body holds every variant of its unit, and at four (128
// registers) it spilt 250 bytes in the row loop (the 48-instance batch: 1181 us
// against 915).
template <int MAXG>
__global__ void __launch_bounds__(kRecThreads, 3)
kb_exp_rec(const BItem* __restrict__ items, BUnits u) {
  __shared__ float2 s_pw[kRecWarps][kSweepTab];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  batch_loop(items, u, [&](const BItem& it, int64_t k) {
    const int64_t unit = k * kRecWarps + warp;
    if (unit >= (int64_t)it.rg.n_grp * it.rg.n_seg * it.rg.n_tgrp) return;
    const RecArgs A = rec_args(it);
    const bool brief = exp_cut8_of(it.g) < 24;
    if constexpr (MAXG >= 4)
      if (it.rg.G == 4) return rec_unit<4, false, true, true>(A, unit, s_pw[warp], lane);
    if constexpr (MAXG >= 2)
      if (it.rg.G == 2) {
        if (it.shared) {
          if (brief) rec_unit<2, true, true, true>(A, unit, s_pw[warp], lane);
          else rec_unit<2, false, true, true>(A, unit, s_pw[warp], lane);
        } else {
          if (brief) rec_unit<2, true, false, true>(A, unit, s_pw[warp], lane);
          else rec_unit<2, false, false, true>(A, unit, s_pw[warp], lane);
        }
        return;
      }
    if (it.shared) {
      if (brief) rec_unit<1, true, true, true>(A, unit, s_pw[warp], lane);
      else rec_unit<1, false, true, true>(A, unit, s_pw[warp], lane);
    } else {
      if (brief) rec_unit<1, true, false, true>(A, unit, s_pw[warp], lane);
      else rec_unit<1, false, false, true>(A, unit, s_pw[warp], lane);
    }
  });
}
const void* batch_kernel_exp_rec(int phase, int max_g) {
  if (phase == BP_EXP_AGG) return (const void*)kb_sweep_agg;
  if (phase != BP_EXP_REC) return nullptr;
  return max_g >= 4 ? (const void*)kb_exp_rec<4>
                    : max_g == 2 ? (const void*)kb_exp_rec<2> : (const void*)kb_exp_rec<1>;
}

}  // namespace fmap
