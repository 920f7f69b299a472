// Device helpers shared by the F-map kernels: window index search, the 2F
// epilogue and the (max, argmax, log-sum-exp) partial reduction.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fmap_internal.h"

namespace fmap {

// The short kernels that end a call follow one another on its stream with
// programmatic dependence (launch_after): the next one's blocks are placed as soon
// as this one's have all started, and wait there for its end, so that a launch
// costs no drain and refill (331 SFTs, 150 x 177 cells: 110 -> 97 us a call).
// Each calls stream_order() first, in all of its threads: it returns when
// everything earlier on the stream is done and visible (each waits for the one
// before, so the order is complete).  What a kernel of the chain writes, the later
// ones read by plain loads only: the read-only path (__ldg, or a const __restrict__
// parameter) may be taken ahead of the wait.
__device__ __forceinline__ void stream_order() {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

constexpr int32_t kNoArg = 0x7fffffff;

// ---- PTX helpers: shared-memory addresses, the global timer, mbarriers ----
// Every spin on an mbarrier is bounded by a limit in ns of %globaltimer: the
// plan's wait limit (kWaitNs by default), and kWaitNs for the drains that let
// copies already in flight land before a block that gave up exits.
constexpr uint64_t kWaitNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Non-blocking test of one phase (try_wait may suspend the thread for a
// hardware-defined time; a zero wait limit polls with this instead).
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait on one phase; false if it did not complete within limit_ns
// (0: give up when one non-blocking poll finds it incomplete).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  uint64_t limit_ns = kWaitNs) {
  if (limit_ns == 0) return mbar_test_wait(bar, parity);
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (!mbar_try_wait(bar, parity))
    if (globaltimer() - t0 > limit_ns) return false;
  return true;
}
// Bounded wait that also gives up at once when another block has already
// timed out (DEV_ERR_TIMEOUT set in *err), so a broken phase costs one
// timeout per launch, not one per block.  Sets the flag on its own timeout.
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t* bar, uint32_t parity,
                                                   uint32_t* err, uint64_t limit_ns = kWaitNs) {
  if (limit_ns == 0) {
    if (mbar_test_wait(bar, parity)) return true;
    atomicOr(err, DEV_ERR_TIMEOUT);
    return false;
  }
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    if (*(volatile uint32_t*)err & DEV_ERR_TIMEOUT) return false;
    if (globaltimer() - t0 > limit_ns) {
      atomicOr(err, DEV_ERR_TIMEOUT);
      return false;
    }
    if (mbar_try_wait(bar, parity)) return true;
  }
}
// Bulk copy global -> shared (16-byte aligned addresses, size a multiple of
// 16), completing `bytes` of transaction count on the mbarrier.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---- float-float (compensated FP32) arithmetic: a value is h + l with
// |l| <= ulp(h)/2, about 2^-44 relative after a chain of operations.  Built
// from the error-free transformations TwoSum (Knuth) and FMA-based TwoProd.
struct FF {
  float h, l;
};

__device__ __forceinline__ FF two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ FF fast_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = fmaf(a.h, b.h, -p);
  return fast_two_sum(p, e + fmaf(a.h, b.l, a.l * b.h));
}
__device__ __forceinline__ FF ff_mul_f(FF a, float b) {
  const float p = __fmul_rn(a.h, b);
  const float e = fmaf(a.h, b, -p);
  return fast_two_sum(p, fmaf(a.l, b, e));
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const FF s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, s.l + a.l + b.l);
}
__device__ __forceinline__ FF ff_sub(FF a, FF b) { return ff_add(a, FF{-b.h, -b.l}); }
// s <- s + w x: the product by FMA-based TwoProd, then a float-float addition
// (~2^-47 relative to the running sum per step).
__device__ __forceinline__ void ff_acc(FF& s, FF w, float x) {
  s = ff_add(s, ff_mul_f(w, x));
}
// s + r e with the product's low part folded into the sum's (no separate
// normalisation of r e): TwoProd of the high parts, TwoSum with s, one
// final renormalisation; ~2^-46 relative, as ff_add(s, ff_mul(r, e)).
__device__ __forceinline__ FF ff_fma_sum(FF s, FF r, FF e) {
  const float p = __fmul_rn(r.h, e.h);
  const float pe = fmaf(r.h, e.h, -p);
  const float t = s.h + p;
  const float bb = t - s.h;
  const float te = (s.h - (t - bb)) + (p - bb);
  return fast_two_sum(t, (s.l + fmaf(r.h, e.l, fmaf(r.l, e.h, pe))) + te);
}
__device__ __forceinline__ FF ff_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

// ---- packed f32x2 arithmetic (.x in the low half): two FP32 operations an
// instruction.
__device__ __forceinline__ uint64_t pk2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void up2(uint64_t a, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(x), "=f"(y) : "l"(a));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// 2F of one cell from its window sums (fa, fb as f32x2 re/im pairs);
// nb2 = (-beta, -beta); k1 = -inf marks a cell that takes no part.
__device__ __forceinline__ float two_f_pairs(uint64_t fa, uint64_t fb, uint64_t nb2, float k1,
                                             float k2, uint64_t tiny2) {
  const uint64_t e = fma2(nb2, fa, fb);
  const uint64_t pa = fma2(fa, fa, tiny2);
  const uint64_t pe = mul2(e, e);
  float a0, a1, e0, e1;
  up2(pa, a0, a1);
  up2(pe, e0, e1);
  return fmaf(k1, a0 + a1, k2 * (e0 + e1));
}

// r a per half as two scalar products: ptxas contracts a packed product into a
// packed addition that follows it (.rn or not: measured), and an error-free
// transformation of the sum would then count the product's error twice.
__device__ __forceinline__ uint64_t mul2_apart(float r, uint64_t a) {
  float x, y;
  up2(a, x, y);
  return pk2(__fmul_rn(r, x), __fmul_rn(r, y));
}
// Two float-float values side by side (h and l as f32x2).
struct FF2 {
  uint64_t h, l;
};
__device__ __forceinline__ FF2 fast_two_sum2(uint64_t a, uint64_t b) {
  const uint64_t s = add2(a, b);
  return {s, sub2(b, sub2(s, a))};
}
// s + r e per half, s a plain f32x2 value and r a float pair common to both
// halves: TwoProd of the high parts, TwoSum with s, one renormalisation
// (~2^-46 relative).
__device__ __forceinline__ FF2 ff2_fma_sum(uint64_t s, FF r, const FF2& e) {
  const uint64_t rh = pk2(r.h, r.h);
  const uint64_t p = mul2_apart(r.h, e.h);
  const uint64_t pe = fma2(rh, e.h, mul2(pk2(-r.h, -r.h), e.h));   // (the addend is -p)
  const uint64_t t = add2(s, p);
  const uint64_t bb = sub2(t, s);
  const uint64_t te = add2(sub2(s, sub2(t, bb)), sub2(p, bb));
  return fast_two_sum2(t, add2(fma2(rh, e.l, fma2(pk2(r.l, r.l), e.h, pe)), te));
}

// Fills one half (s = 0: the weight w, s = 1: w^2) of the per-tau constants of
// one tau value (one thread).  The one-SFT decay is an FP64 exp split into a
// float pair; its powers come by repeated multiplication in float-float (k
// roundings of ~2^-47).  One thread per (tau, half) and 15 products: binary
// powering of every entry by one thread per tau was a chain of ~2000
// instructions, the longest of the copy kernel.
__device__ __forceinline__ void tau_tab_fill(const fmap_grid& g, int64_t tau, int s, TauTab* out) {
  const double inv_tau = 1.0 / (double)tau;
  const double inv_s = (double)(s + 1) * inv_tau;
  if (s == 0) out->inv_tau = inv_tau;
  out->c2[s] = (float)(-1.4426950408889634 * inv_s);
  const FF rho1 = ff_of(exp(-(double)g.t_sft * inv_s));
  FF acc{1.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < kPowTab; ++k) {
    out->pw[s][k] = make_float2(acc.h, acc.l);
    acc = ff_mul(acc, rho1);
  }
}
// Generic window w(x) from its table (entries k = 0..n-1: (w_k, w_{k+1} -
// w_k), then the sentinel (0, 0)): linear between samples, 0 past the last.
// u = x (n - 1) / X is the position in sample units.  u >= 0 where the timestamps
// increase; a window may hold an earlier atom where they do not (which the checks
// only report): the index stays in the table there too (as unsigned numbers,
// negative ones lie past the sentinel).
__device__ __forceinline__ float tab_weight(float u, const float2* tab, int32_t n) {
  const uint32_t k = min((uint32_t)__float2int_rz(u), (uint32_t)n);   // u beyond the table: the sentinel
  const float2 e = tab[k];
  return fmaf(u - (float)k, e.y, e.x);
}
__device__ __forceinline__ double tab_weight64(double u, const float2* tab, int32_t n) {
  const double fk = fmax(floor(u), 0.0);
  const int32_t k = fk >= (double)n ? n : (int32_t)fk;
  const float2 e = tab[k];
  return (double)e.x + (u - (double)k) * (double)e.y;
}
// The same in float-float (~2^-46 relative) for dt = t - t0 in [0, 2^31) and su a
// float pair: FP64 runs at 1/64 of the FP32 rate.
__device__ __forceinline__ FF tab_weight_ff(int32_t dt, FF su, const float2* tab, int32_t n) {
  const float dh = (float)dt;
  const FF u = ff_mul(FF{dh, (float)((int64_t)dt - (int64_t)dh)}, su);
  if (u.h >= (float)n) return FF{0.0f, 0.0f};   // (the sentinel)
  float k = floorf(u.h);
  FF f = two_sum(u.h - k, u.l);
  if (f.h < 0.0f) {
    k -= 1.0f;
    f = two_sum(u.h - k, u.l);
  }
  const float2 e = tab[max((int32_t)k, 0)];
  const float p = __fmul_rn(f.h, e.y);
  const FF s = two_sum(e.x, p);
  return fast_two_sum(s.h, s.l + fmaf(f.l, e.y, fmaf(f.h, e.y, -p)));
}
// Sample units per second of (t - t0) for a tau: (n - 1) / (X tau), X = c / 8.
__host__ __device__ __forceinline__ double tab_scale(int32_t n, int32_t cut8, int64_t tau) {
  return (double)(n - 1) * 8.0 / ((double)cut8 * (double)tau);
}

// Compensated recurrence E <- x + r E (Horner's rule with error-free
// transformations, after Graillat, Langlois and Louvet's compensated Horner
// scheme): E = h + c with h the plain FP32 recurrence and c carrying its
// rounding errors (the TwoProd error of r.h h, the TwoSum error of adding x,
// and the low part r.l of the decay).  The pair is left unnormalised between
// calls; ch_norm folds c back into h.
__device__ __forceinline__ void ch_step(FF r, float x, float& h, float& c) {
  const float p = __fmul_rn(r.h, h);
  const float pe = fmaf(r.h, h, -p);
  const float s = p + x;
  const float bb = s - p;
  const float se = (p - (s - bb)) + (x - bb);
  c = fmaf(r.h, c, fmaf(r.l, h, pe + se));
  h = s;
}
// R <- r R for the compensated running product of the decays.
__device__ __forceinline__ void ch_mul(FF r, float& h, float& c) {
  const float p = __fmul_rn(r.h, h);
  const float pe = fmaf(r.h, h, -p);
  c = fmaf(r.h, c, fmaf(r.l, h, pe));
  h = p;
}
__device__ __forceinline__ void ch_norm(float& h, float& c) {
  const float s = h + c;
  c = c - (s - h);
  h = s;
}

__device__ __forceinline__ Partial partial_empty() {
  Partial p;
  p.max2F = -1.0f;
  p.arg = kNoArg;
  p.sum = 0.0f;
  p.nvalid = 0;
  return p;
}

// Merge two partials (max 2F, lowest argmax on ties, rescaled exp-sum).
__device__ __forceinline__ Partial partial_merge(const Partial& a, const Partial& b) {
  if (a.nvalid == 0) return b;
  if (b.nvalid == 0) return a;
  Partial r;
  if (a.max2F > b.max2F) {
    r.max2F = a.max2F;
    r.arg = a.arg;
    r.sum = a.sum + b.sum * __expf(0.5f * (b.max2F - a.max2F));
  } else if (b.max2F > a.max2F) {
    r.max2F = b.max2F;
    r.arg = b.arg;
    r.sum = b.sum + a.sum * __expf(0.5f * (a.max2F - b.max2F));
  } else {
    r.max2F = a.max2F;
    r.arg = min(a.arg, b.arg);
    r.sum = a.sum + b.sum;
  }
  r.nvalid = a.nvalid + b.nvalid;
  return r;
}

// Add one cell to a running partial.
__device__ __forceinline__ void partial_add(Partial& p, float twoF, int32_t idx, bool valid) {
  if (!valid) return;
  if (p.nvalid == 0) {
    p.max2F = twoF;
    p.arg = idx;
    p.sum = 1.0f;
    p.nvalid = 1;
    return;
  }
  if (twoF > p.max2F) {
    p.sum = p.sum * __expf(0.5f * (p.max2F - twoF)) + 1.0f;
    p.max2F = twoF;
    p.arg = idx;
  } else {
    p.sum += __expf(0.5f * (twoF - p.max2F));
    if (twoF == p.max2F && idx < p.arg) p.arg = idx;
  }
  p.nvalid += 1;
}

// Warp-wide merge (all 32 lanes; the result in every lane).  2F >= 0, so a
// valid partial's maximum orders like its bit pattern: the warp maximum is
// one integer max reduction, each lane rescales its sum to it (one exp),
// the sums add in a fixed butterfly order, and the lowest index among the
// lanes at the maximum and the valid count are integer reductions.
__device__ __forceinline__ Partial partial_warp_reduce(Partial p) {
  const bool has = p.nvalid > 0;
  const unsigned mu = __reduce_max_sync(0xffffffffu, has ? __float_as_uint(p.max2F) + 1u : 0u);
  if (mu == 0u) return partial_empty();
  const float M = __uint_as_float(mu - 1u);
  float s = has ? p.sum * __expf(0.5f * (p.max2F - M)) : 0.0f;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  Partial r;
  r.max2F = M;
  r.arg = (int32_t)__reduce_min_sync(0xffffffffu,
                                     has && p.max2F == M ? (unsigned)p.arg : (unsigned)kNoArg);
  r.sum = s;
  r.nvalid = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)p.nvalid);
  return r;
}

// Block-wide reduction into lane 0 of warp 0 (warp partials merged by warp
// 0); scratch holds >= nwarps entries.  All threads of the block must call it.
template <int NWARPS>
__device__ __forceinline__ Partial partial_block_reduce(Partial p, Partial* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  p = partial_warp_reduce(p);
  if (lane == 0) scratch[warp] = p;
  __syncthreads();
  Partial r = partial_empty();
  if (warp == 0) {
    r = lane < NWARPS ? scratch[lane] : partial_empty();
    r = partial_warp_reduce(r);
  }
  __syncthreads();
  return r;
}

// 2F from the sums of one template and the cell's coefficients.
__device__ __forceinline__ float two_f(const Coef& c, float fa_re, float fa_im, float fb_re,
                                       float fb_im) {
  const float e_re = fmaf(-c.beta, fa_re, fb_re);
  const float e_im = fmaf(-c.beta, fa_im, fb_im);
  const float fa2 = fmaf(fa_re, fa_re, fa_im * fa_im);
  const float e2 = fmaf(e_re, e_re, e_im * e_im);
  return fmaf(c.k1, fa2, c.k2 * e2);
}

// Stores the coefficients of entry e and marks it in the bitmask of the
// ill-conditioned entries when it goes to the fix-up (valid == 2).
__device__ __forceinline__ void store_coef(Coef* __restrict__ coef, uint32_t* __restrict__ bits,
                                           int64_t e, const Coef& c) {
  coef[e] = c;
  if (c.valid == 2.0f) atomicOr(bits + (e >> 5), 1u << (uint32_t)(e & 31));
}

// Coefficients from float-float sums: D = AB - C^2 from exact FMA products
// (relative error ~2^-44 AB, so ~1e-11 of D for AB/D <= 100); the
// divisions in FP32.  A cell whose D is not clearly positive or whose
// AB/D > 100 goes to the fix-up, which decides its validity from
// float-float sums of the window.
__device__ __forceinline__ Coef make_coef_ff(FF A, FF B, FF C, int32_t count) {
  Coef c{0.0f, 0.0f, 0.0f, 0.0f};
  if (count < 2) return c;
  const FF D = ff_sub(ff_mul(A, B), ff_mul(C, C));
  const float af = A.h, cf = C.h, df = D.h;
  if (!(af > 0.0f)) {
    c.valid = 2.0f;
    return c;
  }
  // two correctly rounded reciprocals instead of three divisions (k1 is
  // exact as before; beta and k2 within 1.5 ulp)
  const float ia = __frcp_rn(af);
  c.k1 = 2.0f * ia;
  c.beta = cf * ia;
  c.k2 = (2.0f * af) * __frcp_rn(df);
  // A B > 100 D, compared in float-float
  const FF ab = ff_mul(A, B), d100 = ff_mul_f(D, kCondThreshold);
  const FF gap = ff_sub(d100, ab);
  c.valid = (df > 0.0f && gap.h + gap.l >= 0.0f) ? 1.0f : 2.0f;
  return c;
}

}  // namespace fmap
