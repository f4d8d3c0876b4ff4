// Integer helpers of the FP64-accurate Lanczos path (dtype ED_F64).
//
// GB300 runs FP64 arithmetic at about 1/70 of its FP32 rate, so a Lanczos vector of the
// FP64 path is stored as int64 fixed point: f = s * X with one FP64 scale s per vector and
// |X_i| <= 2^VB. Hop sums of H.v are then exact int64 additions; the few products with
// run-time scalars (t, U, a_j, b_j) are 64x64 -> 128-bit integer products rounded once per
// element; dot products and norms are accumulated exactly in 192-bit integers and rounded
// once to FP64 per step. No FP64 instruction runs per vector element.
#pragma once

#include <stdint.h>

#include "ed_internal.cuh"

namespace ed {

typedef __int128 i128;
typedef unsigned __int128 u128;

// Signed 192-bit accumulator (two's complement): value = hi * 2^128 + lo.
struct I192 {
  u128 lo;
  long long hi;
};

__device__ __forceinline__ void i192_zero(I192& a) {
  a.lo = 0;
  a.hi = 0;
}

__device__ __forceinline__ void i192_add(I192& a, i128 p) {
  const u128 u = (u128)p;
  const u128 s = a.lo + u;
  a.hi += (long long)(s < a.lo) + (p < 0 ? -1LL : 0LL);
  a.lo = s;
}

__device__ __forceinline__ void i192_add(I192& a, const I192& b) {
  const u128 s = a.lo + b.lo;
  a.hi += b.hi + (long long)(s < a.lo);
  a.lo = s;
}

__device__ __forceinline__ I192 i192_shfl_down(const I192& a, int off) {
  I192 r;
  const unsigned long long l0 = (unsigned long long)a.lo, l1 = (unsigned long long)(a.lo >> 64);
  const unsigned long long r0 = __shfl_down_sync(0xffffffffu, l0, off);
  const unsigned long long r1 = __shfl_down_sync(0xffffffffu, l1, off);
  r.lo = ((u128)r1 << 64) | (u128)r0;
  r.hi = __shfl_down_sync(0xffffffffu, a.hi, off);
  return r;
}

// x 2^e, exactly ldexp: an addition to the exponent field while x and the result are normal (one
// thread waits 270 cycles for an ldexp on GB300, and the scalars of a step are one thread's work).
__device__ __forceinline__ double scale2(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF), r = ex + e;
  if (ex == 0 || ex == 0x7FF || r < 1 || r > 0x7FE) return ldexp(x, e);
  return __longlong_as_double(b + ((long long)e << 52));
}

// ilogb of a finite nonzero x.
__device__ __forceinline__ int exponent2(double x) {
  const int ex = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return ex ? ex - 1023 : ilogb(x);
}

// Correctly rounded (nearest) conversion of the 192-bit integer to double.
__device__ __forceinline__ double i192_to_double(const I192& a) {
  const bool neg = a.hi < 0;
  unsigned long long w2 = (unsigned long long)a.hi;
  u128 lo = a.lo;
  if (neg) {  // magnitude = -a
    lo = ~lo + 1;
    w2 = ~w2 + (lo == 0 ? 1ull : 0ull);
  }
  const unsigned long long w1 = (unsigned long long)(lo >> 64), w0 = (unsigned long long)lo;
  unsigned long long top;
  bool sticky;
  int shift;  // value = top * 2^shift (+ sticky below)
  if (w2) {
    const int lz = __clzll(w2);
    top = lz ? (w2 << lz) | (w1 >> (64 - lz)) : w2;
    sticky = (lz ? (w1 << lz) != 0 : w1 != 0) || w0 != 0;
    shift = 128 - lz;
  } else if (w1) {
    const int lz = __clzll(w1);
    top = lz ? (w1 << lz) | (w0 >> (64 - lz)) : w1;
    sticky = lz ? (w0 << lz) != 0 : w0 != 0;
    shift = 64 - lz;
  } else {
    top = w0;
    sticky = false;
    shift = 0;
  }
  // fold the sticky bit into bit 0: the 11 discarded bits of `top` then round correctly
  const double m = __ull2double_rn(top | (sticky ? 1ull : 0ull));
  const double v = scale2(m, shift);
  return neg ? -v : v;
}

// round(p * 2^k) for a 128-bit p, rounding half up; k may be negative (right shift) or
// non-negative (left shift; the caller guarantees no overflow).
__device__ __forceinline__ long long round_shift(i128 p, int k) {
  if (k >= 0) return (long long)(p << k);
  const int s = -k;
  if (s >= 127) return 0;
  const i128 half = (i128)1 << (s - 1);
  return (long long)((p + half) >> s);
}

// The same arithmetic with the 128-bit words spelled out: 64 x 64 -> 128 products from the
// low and high halves of the multiply, sums as carry chains, and the rounding shift split on
// the (warp-uniform) shift amount. Results equal those of the i128 forms above bit for bit.
struct W128 {
  unsigned long long lo;
  long long hi;
};

__device__ __forceinline__ W128 smul128(long long a, long long b) {
  W128 r;
  r.lo = (unsigned long long)a * (unsigned long long)b;
  r.hi = __mul64hi(a, b);
  return r;
}

__device__ __forceinline__ W128 add128(const W128& a, const W128& b) {
  W128 r;
  asm("add.cc.u64 %0, %2, %4;\n\taddc.u64 %1, %3, %5;"
      : "=l"(r.lo), "=l"(r.hi)
      : "l"(a.lo), "l"(a.hi), "l"(b.lo), "l"(b.hi));
  return r;
}

// round_shift for a W128 value.
__device__ __forceinline__ long long round_shift128(const W128& p, int k) {
  if (k >= 0) return k >= 64 ? 0 : (long long)(p.lo << k);
  const int s = -k;
  if (s >= 127) return 0;
  if (s >= 64) {  // the half (2^(s-1)) reaches the high word only through bit 63 of the low one
    long long hi = p.hi;
    if (s == 64) {
      const unsigned long long l2 = p.lo + (1ull << 63);
      hi += (l2 < p.lo) ? 1 : 0;
    } else {
      hi += 1LL << (s - 65);
    }
    return hi >> (s - 64);
  }
  const unsigned long long l2 = p.lo + (1ull << (s - 1));
  const long long h2 = p.hi + ((l2 < p.lo) ? 1 : 0);
  return (long long)((l2 >> s) | ((unsigned long long)h2 << (64 - s)));
}

// 192-bit two's complement accumulator as three words (w2:w1:w0).
struct A192 {
  unsigned long long w0 = 0, w1 = 0, w2 = 0;
};

// a += x^2 with x = |v| < 2^64.
__device__ __forceinline__ void a192_add_sq(A192& a, unsigned long long x) {
  const unsigned long long lo = x * x, hi = __umul64hi(x, x);
  asm("add.cc.u64 %0, %0, %3;\n\taddc.cc.u64 %1, %1, %4;\n\taddc.u64 %2, %2, 0;"
      : "+l"(a.w0), "+l"(a.w1), "+l"(a.w2)
      : "l"(lo), "l"(hi));
}

// a += x y (signed).
__device__ __forceinline__ void a192_add_prod(A192& a, long long x, long long y) {
  const unsigned long long lo = (unsigned long long)x * (unsigned long long)y;
  const long long hi = __mul64hi(x, y);
  const unsigned long long ext = (unsigned long long)(hi >> 63);
  asm("add.cc.u64 %0, %0, %3;\n\taddc.cc.u64 %1, %1, %4;\n\taddc.u64 %2, %2, %5;"
      : "+l"(a.w0), "+l"(a.w1), "+l"(a.w2)
      : "l"(lo), "l"((unsigned long long)hi), "l"(ext));
}

__device__ __forceinline__ I192 a192_get(const A192& a) {
  I192 r;
  r.lo = ((u128)a.w1 << 64) | (u128)a.w0;
  r.hi = (long long)a.w2;
  return r;
}

__device__ __forceinline__ long long shift_signed(long long v, int sh) {
  if (sh >= 0) return v << sh;
  return round_shift((i128)v, sh);
}

// Element i of the random start vector as an integer: the top 53 bits of the (i+1)-th output of
// SplitMix64 (Steele, Lea & Flood 2014) seeded with `seed`, minus 2^52 (2 u - 1 = h 2^-52).
__device__ __forceinline__ long long start_int(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  return (long long)(z >> 11) - (1LL << 52);
}

// ------------------------------------------------------------------ reductions
// Block reduction of a 192-bit sum and a max; thread 0 writes out[0..3] =
// (lo bits 0..63, lo bits 64..127, hi, max).
__device__ __forceinline__ void fx_block_reduce(I192 v, long long mx, long long* out) {
  __shared__ unsigned long long sm[32][4];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const I192 w = i192_shfl_down(v, o);
    i192_add(v, w);
    mx = max(mx, (long long)__shfl_down_sync(0xffffffffu, mx, o));
  }
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) {
    sm[wid][0] = (unsigned long long)v.lo;
    sm[wid][1] = (unsigned long long)(v.lo >> 64);
    sm[wid][2] = (unsigned long long)v.hi;
    sm[wid][3] = (unsigned long long)mx;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    I192 a;
    i192_zero(a);
    long long m = 0;
    if (lane < nw) {
      a.lo = ((u128)sm[lane][1] << 64) | (u128)sm[lane][0];
      a.hi = (long long)sm[lane][2];
      m = (long long)sm[lane][3];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const I192 w = i192_shfl_down(a, o);
      i192_add(a, w);
      m = max(m, (long long)__shfl_down_sync(0xffffffffu, m, o));
    }
    if (lane == 0) {
      out[0] = (long long)(unsigned long long)a.lo;
      out[1] = (long long)(unsigned long long)(a.lo >> 64);
      out[2] = a.hi;
      out[3] = m;
    }
  }
  __syncthreads();
}

// Sum (exact) and max of n partial records of 4 words; every thread gets the result. They may
// come from other CTAs of the running launch: read from L2.
__device__ __forceinline__ void fx_sum_partials(const long long* __restrict__ p, int n, I192& sum,
                                                long long& mx) {
  __shared__ long long out[4];
  I192 v;
  i192_zero(v);
  long long m = 0;
  for (int i = threadIdx.x; i < n; i += 4 * blockDim.x) {  // four records in flight
    longlong2 r[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = i + k * (int)blockDim.x;
      const longlong2* w = reinterpret_cast<const longlong2*>(p + 4 * (int64_t)q);
      r[k][0] = q < n ? __ldcg(w) : make_longlong2(0, 0);
      r[k][1] = q < n ? __ldcg(w + 1) : make_longlong2(0, 0);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      I192 w;
      w.lo = ((u128)(unsigned long long)r[k][0].y << 64) | (u128)(unsigned long long)r[k][0].x;
      w.hi = r[k][1].x;
      i192_add(v, w);
      m = max(m, r[k][1].y);
    }
  }
  fx_block_reduce(v, m, out);
  sum.lo = ((u128)(unsigned long long)out[1] << 64) | (u128)(unsigned long long)out[0];
  sum.hi = out[2];
  mx = out[3];
  __syncthreads();
}

// End of a fixed-point H.v without a ticket: a CTA's sum of W X goes to the run's (no fence, no
// wait).
__device__ __forceinline__ void fx_hv_add(LzScalars* S, const I192& v) {
  __shared__ long long tot[4];
  fx_block_reduce(v, 0, tot);
  if (threadIdx.x < 6)
    atomicAdd(&S->fx_dot[threadIdx.x], (unsigned long long)reinterpret_cast<const uint32_t*>(tot)[threadIdx.x]);
}

// One thread: a_j from the sum of W X, and the update's integer coefficient (Q = W +
// round(d X 2^k2), d 2^k2 = -a_j s_cur / s_w, s_cur / s_w = 2^-r).
__device__ __forceinline__ double fx_alpha(const LzScalars* S, int cur, const I192& sum, long long& d, int& k2) {
  const double alpha = S->fx_sw * S->scale[cur] * i192_to_double(sum);
  const double D = scale2(-alpha, -S->fx_r);
  d = 0;
  k2 = -1;
  if (D != 0.0 && isfinite(D)) {
    k2 = exponent2(D) - 61;
    d = llrint(scale2(D, -k2));
  }
  return alpha;
}

// ... with a ticket: the last CTA records a_j and the coefficient.
__device__ __forceinline__ void fx_hv_finish(LzScalars* S, int cur, const I192& v, long long* part) {
  fx_block_reduce(v, 0, part + 4 * blockIdx.x);
  if (!last_cta(&S->tick_hv)) return;
  I192 sum;
  long long unused;
  fx_sum_partials(part, gridDim.x, sum, unused);
  if (threadIdx.x != 0) return;
  long long d;
  int k2;
  S->alpha[S->j + 1] = fx_alpha(S, cur, sum, d, k2);
  S->row_next = 0;
  S->fx_d = d;
  S->fx_k2 = k2;
}

// Either end, out of line: inlined, its registers cost the H.v's loops spills.
static __device__ __noinline__ void fx_hv_end(LzScalars* S, int cur, unsigned long long w0, unsigned long long w1,
                                              unsigned long long w2, long long* part, int ticket) {
  A192 a;
  a.w0 = w0;
  a.w1 = w1;
  a.w2 = w2;
  if (ticket) fx_hv_finish(S, cur, a192_get(a), part);
  else fx_hv_add(S, a192_get(a));
}

// The sum the H.v's CTAs added up.
__device__ __forceinline__ I192 fx_hv_dot(const LzScalars* S) {
  uint32_t w[6];
  unsigned long long c = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    c += S->fx_dot[i];
    w[i] = (uint32_t)c;
    c >>= 32;
  }
  I192 r;
  r.lo = ((u128)w[3] << 96) | ((u128)w[2] << 64) | ((u128)w[1] << 32) | (u128)w[0];
  r.hi = (long long)(((unsigned long long)w[5] << 32) | w[4]);
  return r;
}

}  // namespace ed
