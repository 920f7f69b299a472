// Generic window functions (FMAP_TABLE grids).
//
// The paper's kernels take the rectangular and exponential windows; its
// method is the same for any amplitude envelope w of the transient: the atoms
// of a window enter Fa, Fb with the weight w((t - t0) / tau) and A, B, C with
// w^2.  Here w is a table of samples on [0, X], X = exp_cut8 / 8 (linear
// between samples, 0 past X), over the exponential window's support.
//
// The data sums go through the same contraction kernels as the exponential
// window (W generated from the table instead of exp2).  The antenna sums
// have no recurrence for a generic w, so this file sums them directly over
// each window: one block per (t0 row, 64 tau cells, antenna set), two cells per
// lane, its four warps taking the atoms 64 at a time in turn, staged in shared
// memory; every cell accumulates its window by cascaded (Sum2) summation with exact
// products (the FP32 weights act as a slightly perturbed window, the same for A, B
// and C; the sums carry about twice-working-precision accuracy, enough for
// D = AB - C^2 up to AB/D = 100).
//
// Bound by the FP32 pipe: three error-free product sums per cell and atom.  Two
// cells per lane make their operations packed f32x2 ones and share each atom's
// load; the table index comes from an addition rounded towards zero instead of two
// conversions (which run at an eighth of the rate); the loop is uniform over the
// warp so that it unrolls.  With a warp per 64 cells, every block was resident at
// once and the SMs' shares differed by half: 192 us for 8 templates' shared
// rows, 301 x 500 cells and 1000 SFTs (one cell per lane: 196 us); blocks of a
// quarter of the work each, more of them than fit at once: 166 us.
#include <math.h>

#include "fmap_device.cuh"

namespace fmap {

constexpr int kTabThreads = 128;
constexpr int kTabWarps = kTabThreads / 32;
constexpr int kTabCells = 64;   // tau cells of a block (one t0 row)
constexpr int kTabKC = 64;      // atoms staged per round

// S += w a for two cells side by side (a is common to them) in the cascaded form
// of Ogita, Rump and Oishi's Sum2 with an exact product: h is the plain FP32
// running sum, l collects the product's FMA error and the TwoSum error of each
// addition (folded into h once, at the end, by ff_fold); the result is as accurate
// as summing in twice the working precision.  aa = (a, a), nw = -w.
__device__ __forceinline__ void ff2_add_prod(FF2& S, uint64_t w, uint64_t nw, uint64_t aa) {
  float a, a1;
  up2(aa, a, a1);
  const uint64_t p = mul2_apart(a, w);
  const uint64_t pe = fma2(w, aa, mul2(nw, aa));   // (the addend is -p)
  const uint64_t s = add2(S.h, p);
  const uint64_t bb = sub2(s, S.h);
  const uint64_t se = add2(sub2(S.h, sub2(s, bb)), sub2(p, bb));
  S.l = add2(S.l, add2(se, pe));
  S.h = s;
}
// tab_weight by an addition: for 0 <= u < 2^12 the index floor(u) is the mantissa of
// the sum of u and 2^23 rounded towards zero.  Any other u (an atom past the cell's
// window, whose weight the caller drops, or one before t0, where the timestamps do not
// increase) gives some index of the table (n < 2^11 entries and the sentinel).
__device__ __forceinline__ float tab_weight_pos(float u, const float2* tab, uint32_t n) {
  const float r = __fadd_rz(u, 8388608.0f);
  const float2 e = tab[min(__float_as_uint(r) & 0xfffu, n)];
  return fmaf(u - (r - 8388608.0f), e.y, e.x);
}
__device__ __forceinline__ FF ff_fold(FF S) { return fast_two_sum(S.h, S.l); }

__global__ void __launch_bounds__(kTabThreads)
k_table_antenna(const int32_t* __restrict__ rel_t, const int64_t* __restrict__ t_base, int32_t n,
                fmap_grid g, const int64_t* __restrict__ ax, const float2* __restrict__ wtab,
                int32_t n_tab, const float* __restrict__ antenna,
                const int32_t* __restrict__ i0tab, const int32_t* __restrict__ jend,
                Coef* __restrict__ coef, uint32_t* __restrict__ bits) {
  __shared__ float4 s_at[kTabWarps][kTabKC][2];   // (a2, a2, b2, b2), (ab, ab, t, t)
  __shared__ float2 s_tab[kTabMax + 1];
  __shared__ FF s_sum[kTabWarps][3][kTabCells];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int32_t nblk = (g.n_tau + kTabCells - 1) / kTabCells;
  const int32_t m = (int32_t)(blockIdx.x / nblk);
  const int32_t n0 = (int32_t)(blockIdx.x - m * nblk) * kTabCells + lane;
  const int ta = blockIdx.y;
  const int64_t cells = (int64_t)g.n_t0 * g.n_tau;
  for (int k = tid; k <= n_tab; k += kTabThreads) s_tab[k] = wtab[k];
  const int32_t i0 = i0tab[m];
  int32_t jc[2];
  float su[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {   // cells n0 and n0 + 32
    const int32_t nn = n0 + 32 * c;
    const bool in_grid = nn < g.n_tau;
    jc[c] = in_grid ? jend[(int64_t)m * g.n_tau + nn] : i0;
    su[c] = in_grid ? (float)tab_scale(n_tab, exp_cut8_of(g), grid_tau(g, ax, nn)) : 0.0f;
  }
  __syncthreads();   // the table is staged
  const int32_t jmax = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)max(jc[0], jc[1]));   // (every warp's: the same cells)
  const int64_t tb = n > 0 ? *t_base : 0;
  const int64_t t0rel = grid_t0(g, ax, m) - tb;
  const float* ant = antenna + (int64_t)ta * 3 * n;
  const uint32_t nt = (uint32_t)n_tab;
  const uint64_t su2 = pk2(su[0], su[1]);
  FF2 S[3] = {{0ull, 0ull}, {0ull, 0ull}, {0ull, 0ull}};
  for (int32_t k0 = i0 + w * kTabKC; k0 < jmax; k0 += kTabWarps * kTabKC) {
    __syncwarp();   // the warp's previous round is read
    for (int e = lane; e < kTabKC; e += 32) {
      const int32_t a = k0 + e;
      const bool in = a < jmax;
      const float t = in ? (float)((int64_t)rel_t[a] - t0rel) : 0.0f;
      float v[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = in ? ant[(int64_t)c * n + a] : 0.0f;
      s_at[w][e][0] = make_float4(v[0], v[0], v[1], v[1]);
      s_at[w][e][1] = make_float4(v[2], v[2], t, t);
    }
    __syncwarp();
    // (atoms past a cell's window weigh 0)
    const int kmax = min(kTabKC, jmax - k0), ke0 = jc[0] - k0, ke1 = jc[1] - k0;
#pragma unroll 4
    for (int kk = 0; kk < kmax; ++kk) {
      const ulonglong2 ab = *reinterpret_cast<const ulonglong2*>(&s_at[w][kk][0]);
      const ulonglong2 ct = *reinterpret_cast<const ulonglong2*>(&s_at[w][kk][1]);
      float u0, u1;
      up2(mul2(ct.y, su2), u0, u1);
      float w0 = tab_weight_pos(u0, s_tab, nt), w1 = tab_weight_pos(u1, s_tab, nt);
      w0 = kk < ke0 ? w0 * w0 : 0.0f;
      w1 = kk < ke1 ? w1 * w1 : 0.0f;
      const uint64_t w2 = pk2(w0, w1), nw2 = pk2(-w0, -w1);
      ff2_add_prod(S[0], w2, nw2, ab.x);
      ff2_add_prod(S[1], w2, nw2, ab.y);
      ff2_add_prod(S[2], w2, nw2, ct.x);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float h0, h1, l0, l1;
    up2(S[k].h, h0, h1);
    up2(S[k].l, l0, l1);
    s_sum[w][k][lane] = ff_fold(FF{h0, l0});
    s_sum[w][k][lane + 32] = ff_fold(FF{h1, l1});
  }
  __syncthreads();
  const int32_t nn = n0 - lane + tid;
  if (tid < kTabCells && nn < g.n_tau) {   // a thread per cell adds the warps' sums
    FF s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      s[k] = s_sum[0][k][tid];
#pragma unroll
      for (int q = 1; q < kTabWarps; ++q) s[k] = ff_add(s[k], s_sum[q][k][tid]);
    }
    store_coef(coef, bits, (int64_t)ta * cells + (int64_t)m * g.n_tau + nn,
               make_coef_ff(s[0], s[1], s[2], tid < 32 ? jc[0] - i0 : jc[1] - i0));
  }
}

cudaError_t launch_table_antenna(fmap_plan_s* p, const fmap_atoms* a, cudaStream_t s) {
  const fmap_grid& g = p->grid;
  if ((int64_t)g.n_t0 * g.n_tau == 0) return cudaSuccess;
  const int n_ant = a->shared_antenna ? 1 : p->n_templates;
  const int64_t blocks = (int64_t)g.n_t0 * ((g.n_tau + kTabCells - 1) / kTabCells);
  k_table_antenna<<<dim3((unsigned)blocks, (unsigned)n_ant), kTabThreads, 0, s>>>(
      p->ws.rel_t, p->ws.t_base, p->n_sft, g, plan_axes(p), p->ws.wtab, p->n_tab, a->antenna,
      p->ws.i0, p->ws.jend, p->ws.coef, p->ws.flag_bits);
  p->launches += 1;
  return cudaGetLastError();
}

}  // namespace fmap
