// Shared pieces of the exponential-window sweeps (antenna sums in fmap_exp.cu,
// data sums in fmap_exp_rec.cu).
//
// The weight factorises in t0: for the atoms [i0, j) of a window,
//   sum_a e^{-s(t_a - t0)/tau} x_a
//     = e^{-s(t_{i0} - t0)/tau} (E[i0] - e^{-s(t_j - t_{i0})/tau} E[j]),
//   E[i] = x_i + e^{-s(t_{i+1} - t_i)/tau} E[i+1]
// (s = 1 for the data, 2 for the antenna rows; E may start from zero anywhere
// at or after the window's end, which cancels), an exact rearrangement of the
// window sums of Eq. (winexp).  A warp takes 32 consecutive tau (one per lane)
// and a run of t0 rows, from the last row to the first: i0 and j only move
// towards earlier atoms, so each lane carries E at its two cursors in
// registers and advances them atom by atom (on a grid with T_sft steps one
// atom per row each).  i0 is the same for the warp's lanes (its atom is a
// broadcast load), j differs by lane (a gather within a few cache lines); the
// coefficients, window ends and the map are read and written 32 consecutive
// tau at a time.  Nothing passes between warps.
#pragma once

#include "fmap_front.cuh"

namespace fmap {

// (out of line: the FP64 exp's registers stay out of the sweeps' loops)
static __device__ __noinline__ float2 slow_decay(int32_t gap, double inv_s) {
  const FF v = ff_of(exp(-(double)gap * inv_s));
  return make_float2(v.h, v.l);
}

// A warp's table of decays: entry [k][lane] for gaps of k SFTs.
constexpr int kSweepTab = kPowTab * 32;   // float2 entries per warp (4 KB)
template <int S>
__device__ __forceinline__ void sweep_tab_load(float2* s_pw, const TauTab* __restrict__ tt,
                                               int lane) {
  __syncwarp();   // (the warp's previous unit is done with the table)
#pragma unroll
  for (int k = 0; k < kPowTab; ++k) s_pw[k * 32 + lane] = tt->pw[S - 1][k];
  __syncwarp();
}
// IRR: the data set has gaps of code 0.  (The sweeps branch once per warp on
// whether any gap has: the call, even where it is never made, costs the loops
// around it registers and moves.)
template <int S, bool IRR>
__device__ __forceinline__ FF sweep_decay(const float2* s_pw, int32_t code, int lane,
                                          const int32_t* __restrict__ rel_t, int32_t a,
                                          const TauTab* __restrict__ tt) {
  if (IRR && code == 0) {
    const float2 v = slow_decay(rel_t[a + 1] - rel_t[a], (double)S * tt->inv_tau);
    return {v.x, v.y};
  }
  // (after the last atom E is zero: any decay does)
  const float2 v = s_pw[max(code, 0) * 32 + lane];
  return {v.x, v.y};
}

// The same from the gap itself (the data sweep keeps its cursors' times): gaps of
// k SFTs by a multiplication (inv = ceil(2^31 / T_sft), exact for multiples
// below 2^31).
template <int S, bool IRR>
__device__ __forceinline__ FF sweep_gap_decay(const float2* s_pw, int32_t gap, uint32_t inv,
                                              int32_t t_sft, int lane,
                                              const TauTab* __restrict__ tt) {
  const int32_t k = (int32_t)__umulhi((uint32_t)gap << 1, inv);
  if (IRR && (k < 1 || k >= kPowTab || k * t_sft != gap)) {
    const float2 v = slow_decay(gap, (double)S * tt->inv_tau);
    return {v.x, v.y};
  }
  const float2 v = s_pw[(k & (kPowTab - 1)) * 32 + lane];
  return {v.x, v.y};
}

// E of one tau: columns a^2 and b^2 packed, ab alone; unnormalised pairs.
struct AntE {
  uint64_t h2, c2;
  float h, c;
};
__device__ __forceinline__ AntE ant_zero() { return {0ull, 0ull, 0.0f, 0.0f}; }
// E <- x + r E (compensated Horner step per column, as ch_step)
__device__ __forceinline__ void ant_step(AntE& e, FF r, const float4& x) {
  const uint64_t rh = pk2(r.h, r.h), x2 = pk2(x.x, x.y);
  const uint64_t p = mul2_apart(r.h, e.h2);
  const uint64_t pe = fma2(rh, e.h2, mul2(pk2(-r.h, -r.h), e.h2));
  const uint64_t s = add2(p, x2);
  const uint64_t bb = sub2(s, p);
  const uint64_t se = add2(sub2(p, sub2(s, bb)), sub2(x2, bb));
  e.c2 = fma2(rh, e.c2, fma2(pk2(r.l, r.l), e.h2, add2(pe, se)));
  e.h2 = s;
  ch_step(r, x.z, e.h, e.c);
}
__device__ __forceinline__ void ant_norm(AntE& e) {
  const FF2 n = fast_two_sum2(e.h2, e.c2);
  e.h2 = n.h;
  e.c2 = n.l;
  ch_norm(e.h, e.c);
}
__device__ __forceinline__ void ant_get(const AntE& e, FF (&v)[3]) {
  up2(e.h2, v[0].h, v[1].h);
  up2(e.c2, v[0].l, v[1].l);
  v[2] = {e.h, e.c};
}
__device__ __forceinline__ void ant_put(AntE& e, const FF (&v)[3]) {
  e.h2 = pk2(v[0].h, v[1].h);
  e.c2 = pk2(v[0].l, v[1].l);
  e.h = v[2].h;
  e.c = v[2].l;
}

// Chunk maps: agg[((ta n_grp + grp) n_chunks + chunk) 8 + q][32 lanes], q = the
// float pairs of S (3 columns), then of R.
template <bool IRR>
__device__ __forceinline__ void exp_agg_unit(const int32_t* __restrict__ rel_t, int32_t n,
                                             const float4* __restrict__ ant,
                                             const TauTab* __restrict__ tauc, const fmap_grid& g,
                                             const AntGeom& q, float* __restrict__ agg,
                                             int64_t unit, float2* s_pw, int lane) {
  const int32_t ch = (int32_t)(unit % q.n_chunks);
  const int64_t ag = unit / q.n_chunks;            // ta n_grp + grp
  const int32_t grp = (int32_t)(ag % q.n_grp);
  const int64_t ta = ag / q.n_grp;
  const TauTab* tt = tauc + min(grp * 32 + lane, g.n_tau - 1);
  sweep_tab_load<2>(s_pw, tt, lane);
  const float4* x = ant + ta * n;
  const int32_t lo = ch * q.chunk, hi = min(n, lo + q.chunk);
  AntE e = ant_zero();
  float Rh = 1.0f, Rc = 0.0f;
  for (int32_t a1 = hi; a1 > lo; a1 -= 8) {
    float4 v[8];   // loaded ahead of the serial chain
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = a1 - 1 - k >= lo ? __ldg(x + a1 - 1 - k) : float4{};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int32_t a = a1 - 1 - k;
      if (a < lo) break;
      const FF r = sweep_decay<2, IRR>(s_pw, __float_as_int(v[k].w), lane, rel_t, a, tt);
      ant_step(e, r, v[k]);
      ch_mul(r, Rh, Rc);
    }
    ant_norm(e);
    ch_norm(Rh, Rc);
  }
  FF S[3];
  ant_get(e, S);
  float* o = agg + (ag * q.n_chunks + ch) * 256 + lane;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    o[64 * c] = S[c].h;
    o[64 * c + 32] = S[c].l;
  }
  o[192] = Rh;
  o[224] = Rc;
}

}  // namespace fmap
