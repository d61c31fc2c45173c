// ff_math.cuh -- float-float arithmetic and fixed-order block reductions
// shared by the acceptance and draft-sampling kernels.  A float-float number
// is an unevaluated sum hi + lo of two fp32 values (~44 significant bits),
// built from exactly rounded fp32 operations (Knuth's TwoSum, FMA-based
// TwoProduct); every reduction runs in a fixed order, so results are
// deterministic.  Blocks are kFfThreads threads.
#pragma once

#include <climits>
#include <cmath>

#include "sf_device.cuh"

namespace sf {

constexpr int kFfThreads = 256;
constexpr int kFfWarps = kFfThreads / 32;

struct ff {       // float-float number hi + lo, |lo| <= ulp(hi) / 2
  float hi, lo;
};

// Softmax statistics of one chunk of one row: written by the projection
// epilogue (draft_tail.cu), read by the samplers and the fused acceptance.
struct SampStat {
  float m;  // largest logit of the chunk
  int arg;  // its first index
  ff S;     // sum of exp((x - m) / tau) over the chunk; 0 for greedy rows
};
static_assert(sizeof(SampStat) == 16, "SampStat is 16 bytes");

// (value, index) order for argmax: larger value first, then lower index.
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

// Float-float arithmetic (Knuth's TwoSum and an FMA-based TwoProduct); the
// explicit _rn intrinsics keep the compiler from contracting or reordering.
__device__ __forceinline__ ff ff_of(float x) { return ff{x, 0.f}; }

// a + b exactly, as a float-float number.
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  return ff{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float v = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  const float hi = __fadd_rn(s, e);
  return ff{hi, __fsub_rn(e, __fsub_rn(hi, s))};
}

__device__ __forceinline__ ff ff_mul(ff a, float b) {
  const float p = __fmul_rn(a.hi, b);
  float e = __fmaf_rn(a.hi, b, -p);
  e = __fmaf_rn(a.lo, b, e);
  const float hi = __fadd_rn(p, e);
  return ff{hi, __fsub_rn(e, __fsub_rn(hi, p))};
}

__device__ __forceinline__ ff ff_mul(ff a, ff b) { return ff_add(ff_mul(a, b.hi), ff_of(__fmul_rn(a.hi, b.lo))); }

__device__ __forceinline__ bool ff_lt(ff a, ff b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

__device__ __forceinline__ bool ff_pos(ff a) { return a.hi > 0.f || (a.hi == 0.f && a.lo > 0.f); }

// a / b rounded to fp32 (one Newton correction of the fp32 quotient).
__device__ __forceinline__ float ff_div_to_f(float a, ff b) {
  const float q = __fdiv_rn(a, b.hi);
  float r = __fmaf_rn(-q, b.hi, a);  // a - q * b.hi, exact
  r = __fmaf_rn(-q, b.lo, r);
  return __fadd_rn(q, __fdiv_rn(r, b.hi));
}

// exp((x - m) / tau) with the argument carried to float-float, so that the
// result is as accurate as expf itself even for large |x - m|; 0 for a
// masked token (x = -inf), where the float-float split would give NaN.
__device__ __forceinline__ float exp_diff_accurate(float x, float m, float tau) {
  if (x == -INFINITY) return 0.f;
  float hi = __fsub_rn(x, m);
  const float v = __fsub_rn(hi, x);
  float lo = __fadd_rn(__fsub_rn(x, __fsub_rn(hi, v)), __fsub_rn(-m, v));
  if (tau != 1.0f) {
    const float qh = __fdiv_rn(hi, tau);
    const float r = __fmaf_rn(-qh, tau, hi);  // hi - qh * tau, exact
    lo = __fdiv_rn(__fadd_rn(r, lo), tau);
    hi = qh;
  }
  return __fmul_rn(expf(hi), __fadd_rn(1.0f, lo));
}

// The same with 1 / tau at hand (rounded; tau from 2^-64 to 2^64), for loops over
// many tokens of one temperature: the quotient's high part is a product, off by up
// to 1.5 units in its last place, and its low part, from the exact remainder, makes
// up for that, so that hi + lo is as close to the quotient as after a division.
constexpr float kRecipTauMin = 5.421010862427522e-20f, kRecipTauMax = 1.8446744073709552e19f;

__device__ __forceinline__ float exp_diff_recip(float x, float m, float tau, float inv_tau) {
  if (x == -INFINITY) return 0.f;
  const float d = __fsub_rn(x, m);
  const float v = __fsub_rn(d, x);
  const float lo = __fadd_rn(__fsub_rn(x, __fsub_rn(d, v)), __fsub_rn(-m, v));
  const float hi = __fmul_rn(d, inv_tau);
  const float rest = __fmaf_rn(-hi, tau, d);  // d - hi * tau, exact
  return __fmul_rn(expf(hi), __fmaf_rn(__fadd_rn(rest, lo), inv_tau, 1.0f));
}

// exp((x - m) / tau), x <= m, as a float-float number with a relative error of
// about 1e-8, for factors that scale a whole partial sum (where the error of
// many terms averages out and that of one factor would not).  Cody and Waite's
// reduction, (x - m) / tau = n ln 2 + r with ln 2 in two parts, then 1 + r exact and the
// rest of the power series, at most 0.07, in fp32.  0 below e^-87.
__device__ __forceinline__ ff exp_diff_ff(float x, float m, float tau) {
  float hi = __fsub_rn(x, m);
  const float v = __fsub_rn(hi, x);
  float lo = __fadd_rn(__fsub_rn(x, __fsub_rn(hi, v)), __fsub_rn(-m, v));
  if (tau != 1.0f) {
    const float qh = __fdiv_rn(hi, tau);
    const float rest = __fmaf_rn(-qh, tau, hi);  // hi - qh * tau, exact
    lo = __fdiv_rn(__fadd_rn(rest, lo), tau);
    hi = qh;
  }
  if (hi <= -87.0f) return ff_of(0.f);  // a masked part (x = -inf) too
  const float n = rintf(__fmul_rn(hi, 1.44269504f));
  constexpr float kLn2Hi = 0.693145751953125f;     // 15 bits of ln 2: n kLn2Hi is exact
  constexpr float kLn2Lo = 1.42860682030941723e-6f;  // ln 2 - kLn2Hi
  const ff r = two_sum(__fmaf_rn(-n, kLn2Hi, hi), __fmaf_rn(-n, kLn2Lo, lo));
  float q = 1.0f / 40320.0f;
  q = __fmaf_rn(q, r.hi, 1.0f / 5040.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 720.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 120.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 24.0f);
  q = __fmaf_rn(q, r.hi, 1.0f / 6.0f);
  q = __fmaf_rn(q, r.hi, 0.5f);
  q = __fmul_rn(q, __fmul_rn(r.hi, r.hi));
  const ff s = two_sum(1.0f, r.hi);
  const ff e = two_sum(s.hi, __fadd_rn(__fadd_rn(s.lo, r.lo), q));
  const float scale = __int_as_float((static_cast<int>(n) + 127) << 23);  // 2^n, n >= -126
  return ff{__fmul_rn(e.hi, scale), __fmul_rn(e.lo, scale)};
}

// Hardware base-2 exponential (approximate, subnormal results kept).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// exp(a) = 2^(a log2 e) with a * log2 e carried as hi + lo (log2 e split
// into the float nearest it and the remainder, an FMA for the rounding of
// hi), 2^hi from ex2.approx and 2^lo ~ 1 + lo ln 2 (|lo| is a few ulp of
// hi).  Measured against expf on GB300 over [-103, 1]: max relative error
// 2.4e-7 (expf 1.5e-7).  For the hot loops of the acceptance, where it
// replaces expf.
__device__ __forceinline__ float exp_fast(float a) {
  constexpr float kL2eHi = 1.44269502162933349609375f;   // nearest float to log2 e
  constexpr float kL2eLo = 1.9259630335000111e-08f;       // log2 e - kL2eHi
  const float hi = __fmul_rn(a, kL2eHi);
  const float lo = __fmaf_rn(a, kL2eLo, __fmaf_rn(a, kL2eHi, -hi));
  const float r = __fmul_rn(ex2_approx(hi), __fmaf_rn(lo, 0.69314718055994531f, 1.0f));
  return a == -INFINITY ? 0.f : r;  // lo is NaN there
}

__device__ __forceinline__ ff shfl_xor_ff(ff a, int o) {
  return ff{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

__device__ __forceinline__ ff shfl_up_ff(ff a, int o) {
  return ff{__shfl_up_sync(0xffffffffu, a.hi, o), __shfl_up_sync(0xffffffffu, a.lo, o)};
}

// Sum over the warp's lanes; with LANES < 32, over each aligned group of them.
template <int LANES = 32>
__device__ __forceinline__ ff warp_sum_ff(ff v) {
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) v = ff_add(v, shfl_xor_ff(v, o));
  return v;
}

// The largest value of the warp (no NaN) and its lowest index, by two integer
// reductions: the floats' order as unsigned integers (-0 taken as +0).
__device__ __forceinline__ void warp_argmax(float &v, int &i) {
  const int s = __float_as_int(__fadd_rn(v, 0.0f));
  const unsigned key = s < 0 ? ~static_cast<unsigned>(s) : static_cast<unsigned>(s) ^ 0x80000000u;
  const unsigned top = __reduce_max_sync(0xffffffffu, key);
  i = __reduce_min_sync(0xffffffffu, key == top ? i : INT_MAX);
  v = __uint_as_float(top & 0x80000000u ? top ^ 0x80000000u : ~top);
}

// Block-wide float-float sum (fixed tree order).
__device__ inline ff block_sum(ff v, ff *s_buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum_ff(v);
  __syncthreads();
  if (lane == 0) s_buf[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < kFfWarps ? s_buf[lane] : ff_of(0.f);
    v = warp_sum_ff(v);
    if (lane == 0) s_buf[0] = v;
  }
  __syncthreads();
  return s_buf[0];
}

__device__ inline void block_argmax(float &v, int &i, float *s_v, int *s_i) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  warp_argmax(v, i);
  __syncthreads();
  if (lane == 0) { s_v[warp] = v; s_i[warp] = i; }
  __syncthreads();
  if (warp == 0) {
    v = lane < kFfWarps ? s_v[lane] : -INFINITY;
    i = lane < kFfWarps ? s_i[lane] : INT_MAX;
    warp_argmax(v, i);
    if (lane == 0) { s_v[0] = v; s_i[0] = i; }
  }
  __syncthreads();
  v = s_v[0];
  i = s_i[0];
}

// Inclusive float-float prefix over the first `n` lanes (n a power of two): a
// lane's exclusive value is the inclusive value of the lane before, bit for bit.
__device__ __forceinline__ ff warp_scan_ff(ff v, int n, ff *excl) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o >= n) break;
    const ff t = shfl_up_ff(v, o);
    if (lane >= o) v = ff_add(t, v);
  }
  *excl = shfl_up_ff(v, 1);
  if (lane == 0) *excl = ff_of(0.f);
  return v;
}

__device__ __forceinline__ ff shfl_ff(ff v, int lane) {
  return ff{__shfl_sync(0xffffffffu, v.hi, lane), __shfl_sync(0xffffffffu, v.lo, lane)};
}

// The same over the block, with two barriers; returns the thread's exclusive
// value, and in *next (if asked for) the exclusive value of the thread after
// it, bit for bit (*total after the last), so that [excl, next) tile [0, total).
__device__ __forceinline__ ff block_scan2(ff v, ff *s_warp, ff *total, ff *next = nullptr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ff ex, wex;
  v = warp_scan_ff(v, 32, &ex);
  __syncthreads();  // s_warp may be in use
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  const ff w = warp_scan_ff(lane < kFfWarps ? s_warp[lane] : ff_of(0.f), kFfWarps, &wex);
  *total = shfl_ff(w, kFfWarps - 1);
  const ff off = shfl_ff(wex, warp);
  const ff prev = shfl_up_ff(ff_add(off, v), 1);
  const ff excl = lane > 0 ? prev : off;
  if (next) {
    const ff after = shfl_ff(excl, (lane + 1) & 31), warp_end = shfl_ff(w, warp);
    *next = lane < 31 ? after : warp_end;
  }
  return excl;
}

}  // namespace sf
