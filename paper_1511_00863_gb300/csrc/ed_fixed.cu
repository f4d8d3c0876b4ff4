// FP64-accurate Lanczos (Sec. 2.2, Algorithm 1) with int64 fixed-point vectors.
//
// A vector is f = s * X (s: FP64 scale in LzScalars, X: int64, |X_i| <= 2^vb with
// vb = 62 - ceil(log2(hops + n_max + 2))), so that a hop sum of up to `hops` elements and
// the diagonal product n X never overflow. One step j on buffers cur (f_j) and prev
// (f_{j-1}):
//   plan   (1 thread, at the end of the step before): choose W's scale s_w = s_cur 2^r so that |W| <= 2^(vb-1), and the
//                       integer coefficients of  W = round((a S + b n X + c P) 2^k)  with
//                       a 2^k = -t 2^-r, b 2^k = U 2^-r, c 2^k = -b_j (s_prev/s_cur) 2^-r;
//   H.v    (fused):     S = exact int64 hop sum (Sec. 4 Eqs. 5-6), P = X_prev, W written
//                       over P; partial sums of W X_cur exact in 192 bits;
//   update:             a_j = s_w s_cur sum(W X_cur) (one FP64 rounding, one thread per CTA),
//                       Q = W + round(d X_cur 2^k2) with d 2^k2 = -a_j s_cur / s_w,
//                       exact partial sums of Q^2 and max |Q|;
//   finish (1 CTA):     b_{j+1} = s_w sqrt(sum Q^2), f_{j+1} = (s_w / b_{j+1}) Q.
// Every element of every vector is rounded once per pass, to a grid of 2^-vb of the
// vector's current maximum; sums and dot products are exact.
#include <cmath>

#include "ed_fixed.cuh"
#include "ed_internal.cuh"
#include "ed_lanczos_dev.cuh"

namespace ed {

constexpr int kFxThreads = 256;

FxRun fx_make(const ed_basis* b) {
  FxRun f;
  f.hops = b->up.maxhops + b->dn.maxhops;
  f.nmax = b->n_up < b->n_dn ? b->n_up : b->n_dn;
  const int need = f.hops + f.nmax + 2;
  int hb = 0;
  while ((1 << hb) < need) ++hb;
  f.vb = 62 - hb;
  return f;
}

__device__ __forceinline__ long long sgn_apply(long long v, uint32_t e) {
  const long long m = (long long)((int32_t)e >> 31);  // 0 or -1
  return (v ^ m) - m;
}

// ------------------------------------------------------------------ caller vectors
// Largest |f_i| as its IEEE bit pattern (sign cleared); a non-finite entry gives the
// pattern of infinity or NaN, which the host rejects.
__global__ void __launch_bounds__(kFxThreads)
fx_absmax_kernel(const double* __restrict__ f, int64_t n, unsigned long long* __restrict__ part) {
  __shared__ unsigned long long sm[32];
  unsigned long long m = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(f[i]) & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? sm[threadIdx.x] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) part[blockIdx.x] = m;
  }
}

__global__ void __launch_bounds__(kFxThreads)
fx_absmax_final(const unsigned long long* __restrict__ part, int n, unsigned long long* __restrict__ out) {
  __shared__ unsigned long long sm[32];
  unsigned long long m = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = max(m, part[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, sm[w]);
    *out = m;
  }
}

// f_1 = X / ||X||: scale[0] = 1 / sqrt(sum X^2), fx_max[0] = max |X|.
__global__ void __launch_bounds__(kFxThreads)
fx_init_kernel(LzScalars* S, const long long* __restrict__ part, int n) {
  I192 sum;
  long long mx;
  fx_sum_partials(part, n, sum, mx);
  if (threadIdx.x == 0) {
    const double q2 = i192_to_double(sum);
    S->scale[0] = q2 > 0.0 ? 1.0 / sqrt(q2) : 0.0;
    S->scale[1] = 0.0;
    S->fx_max[0] = mx;
    S->fx_max[1] = 0;
  }
}

// ------------------------------------------------------------------ one step
struct FxPlanArgs {
  double t, U;
  int hops, nmax, vb;
};

// One thread: the integer coefficients of the H.v of step S->j + 1 on buffer cur.
__device__ __forceinline__ void fx_plan_step(LzScalars* S, int cur, const FxPlanArgs& p) {
  const double t = p.t, U = p.U;
  const int hops = p.hops, nmax = p.nmax, vb = p.vb;
  const int j = S->j + 1;
  const double sc = S->scale[cur], sp = S->scale[1 - cur];
  const double mc = (double)S->fx_max[cur], mp = (double)S->fx_max[1 - cur];
  const double cp = sc != 0.0 ? S->beta[j] * sp / sc : 0.0;
  const double bound = (fabs(t) * hops + fabs(U) * nmax) * mc + fabs(cp) * mp;
  int r = 0;
  if (bound > 0.0 && isfinite(bound)) r = exponent2(bound) + 1 - (vb - 1);
  const double A = scale2(-t, -r), B = scale2(U, -r), C = scale2(-cp, -r);
  const double M = fmax(fabs(A), fmax(fabs(B), fabs(C)));
  int k = 0;
  long long a = 0, b = 0, c = 0;
  if (M > 0.0 && isfinite(M)) {
    k = exponent2(M) - 61;
    a = llrint(scale2(A, -k));
    b = llrint(scale2(B, -k));
    c = llrint(scale2(C, -k));
  }
  S->fx_a = a;
  S->fx_b = b;
  S->fx_c = c;
  S->fx_k = k;
  S->fx_r = r;
  S->fx_sw = scale2(sc, r);
}

__global__ void fx_plan_kernel(LzScalars* S, int cur, FxPlanArgs p) {
  if (threadIdx.x == 0 && S->status == 0) fx_plan_step(S, cur, p);
}

struct FxHvArgs {
  const uint32_t* __restrict__ up_bits;
  const uint32_t* __restrict__ dn_bits;
  const int32_t* __restrict__ hop_up;
  const int32_t* __restrict__ hop_dn;
  int64_t dim_up, dim_dn, ld;
  int maxhops_up, maxhops_dn;
};

// s += the signed values of a state's hop targets (integers: the order does not matter),
// four hops at a time with their table entries and values loaded before any is added, so a
// thread has more loads in flight. tab[k * stride] is hop k's entry; a target >= n is
// padding, and the rest of the state's list is padding too.
template <typename Load>
__device__ __forceinline__ void fx_add_hops(long long& s, const int32_t* tab, int64_t stride, int mh,
                                            int64_t n, Load load) {
  int k = 0;
  for (; k + 4 <= mh; k += 4) {
    uint32_t e[4];
    long long v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) e[q] = (uint32_t)tab[(int64_t)(k + q) * stride];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t tg = (int64_t)(e[q] & kTargetMask);
      v[q] = tg < n ? sgn_apply(load(tg), e[q]) : 0LL;
    }
    s += (v[0] + v[1]) + (v[2] + v[3]);
    if ((int64_t)(e[3] & kTargetMask) >= n) return;
  }
  for (; k < mh; ++k) {
    const uint32_t e = (uint32_t)tab[(int64_t)k * stride];
    const int64_t tg = (int64_t)(e & kTargetMask);
    if (tg >= n) return;
    s += sgn_apply(load(tg), e);
  }
}

// W = round((a S + b n X + c P) 2^k), written over P; partial sums of W X (exact).
// Row-staged like hv_staged_kernel: R up rows per CTA, interleaved in shared memory.
template <int R>
__global__ void __launch_bounds__(kFxThreads)
fx_hv_staged_kernel(FxHvArgs a, const long long* __restrict__ x, long long* __restrict__ y,
                    LzScalars* S) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (S->status != 0) return;
  const long long ca = S->fx_a, cb = S->fx_b, cc = S->fx_c;
  const int k = S->fx_k;
  const int dn = (int)a.dim_dn;
  long long* xs = reinterpret_cast<long long*>(smem);
  int32_t* ut = reinterpret_cast<int32_t*>(xs + (size_t)(dn + 1) * R);
  const int64_t u0 = (int64_t)blockIdx.x * R;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t u = u0 + r;
    const long long* xr = x + u * a.ld;
    for (int d = threadIdx.x; d < dn; d += blockDim.x) xs[d * R + r] = (u < a.dim_up) ? xr[d] : 0LL;
  }
  if (threadIdx.x < R) xs[(size_t)dn * R + threadIdx.x] = 0LL;
  for (int i = threadIdx.x; i < R * a.maxhops_up; i += blockDim.x) {
    const int r = i / a.maxhops_up, kk = i - r * a.maxhops_up;
    const int64_t u = u0 + r;
    ut[i] = (u < a.dim_up) ? a.hop_up[(int64_t)kk * a.dim_up + u] : (int32_t)a.dim_up;
  }
  uint32_t ub[R];
#pragma unroll
  for (int r = 0; r < R; ++r) ub[r] = (u0 + r < a.dim_up) ? a.up_bits[u0 + r] : 0u;
  __syncthreads();

  I192 dot;
  i192_zero(dot);
  for (int d = threadIdx.x; d < dn; d += blockDim.x) {
    const uint32_t db = a.dn_bits[d];
    long long hs[R];
#pragma unroll
    for (int r = 0; r < R; ++r) hs[r] = 0;
    for (int kk = 0; kk < a.maxhops_dn; ++kk) {
      const uint32_t e = (uint32_t)a.hop_dn[(int64_t)kk * dn + d];
      const int tg = (int)(e & kTargetMask);
#pragma unroll
      for (int r = 0; r < R; ++r) hs[r] += sgn_apply(xs[tg * R + r], e);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t u = u0 + r;
      if (u < a.dim_up) {
        fx_add_hops(hs[r], ut + r * a.maxhops_up, 1, a.maxhops_up, a.dim_up,
                    [&](int64_t tg) { return x[tg * a.ld + d]; });
        const long long xc = xs[d * R + r];
        const long long nx = xc * (long long)__popc(ub[r] & db);
        long long* yp = y + u * a.ld + d;
        const i128 p = (i128)ca * hs[r] + (i128)cb * nx + (i128)cc * (*yp);
        const long long w = round_shift(p, k);
        *yp = w;
        i192_add(dot, (i128)w * xc);
      }
    }
  }
  fx_hv_add(S, dot);
}

// Fallback when a row does not fit in shared memory.
__global__ void __launch_bounds__(kFxThreads)
fx_hv_global_kernel(FxHvArgs a, const long long* __restrict__ x, long long* __restrict__ y,
                    LzScalars* S) {
  if (S->status != 0) return;
  const long long ca = S->fx_a, cb = S->fx_b, cc = S->fx_c;
  const int k = S->fx_k;
  I192 dot;
  i192_zero(dot);
  const int64_t total = a.dim_up * a.dim_dn;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = g / a.dim_dn, d = g - u * a.dim_dn;
    const long long* xr = x + u * a.ld;
    long long hs = 0;
    fx_add_hops(hs, a.hop_dn + d, a.dim_dn, a.maxhops_dn, a.dim_dn, [&](int64_t tg) { return xr[tg]; });
    fx_add_hops(hs, a.hop_up + u, a.dim_up, a.maxhops_up, a.dim_up,
                [&](int64_t tg) { return x[tg * a.ld + d]; });
    const long long xc = xr[d];
    const long long nx = xc * (long long)__popc(a.up_bits[u] & a.dn_bits[d]);
    long long* yp = y + u * a.ld + d;
    const long long w = round_shift((i128)ca * hs + (i128)cb * nx + (i128)cc * (*yp), k);
    *yp = w;
    i192_add(dot, (i128)w * xc);
  }
  fx_hv_add(S, dot);
}

// Whole CTA: b_{j+1} and f_{j+1}'s scale from the n partial records of ||Q||^2, then the
// coefficients of the next H.v.
__device__ __forceinline__ void fx_finish_step(LzScalars* S, int cur, const long long* pb, int nb,
                                               const FxPlanArgs& p, const LzStore& store) {
  I192 sum;
  long long mx;
  fx_sum_partials(pb, nb, sum, mx);
  if (threadIdx.x < 6) S->fx_dot[threadIdx.x] = 0;
  if (threadIdx.x != 0) return;
  const int j = S->j + 1;
  const double sw = S->fx_sw;
  const double beta = sw * sqrt(i192_to_double(sum));
  if (finish_step(S, j, beta)) {
    S->scale[1 - cur] = sw / beta;
    S->fx_max[1 - cur] = mx;
    if (store.vscale) store.vscale[j] = sw / beta;
    if (store.vmax) store.vmax[j] = mx;
    fx_plan_step(S, 1 - cur, p);
  }
}

// kReady: the H.v left a_j finished (hv2_ticket), else its sum in S->fx_dot.
// finish: the last CTA ends the step (fx_finish_step); otherwise fx_finish_kernel does, after
// the reorthogonalisation. kKeep: Q goes to the step's slot of `store` too. The grid is 4 CTAs
// per SM: with more registers than that leaves (it takes 70 unbounded) a third of it ran as a
// second wave, 102 instead of 81 us on the 4x4 lattice.
template <bool kKeep, bool kReady>
__global__ void __launch_bounds__(kFxThreads, 4)
fx_update_kernel(LzScalars* S, int cur, const long long* __restrict__ xc, long long* __restrict__ xp,
                 int64_t n, long long* __restrict__ pb, int finish, FxPlanArgs plan, LzStore store) {
  if (S->status != 0) return;
  long long d;
  int k2;
  if constexpr (kReady) {
    d = S->fx_d;
    k2 = S->fx_k2;
  } else {
    __shared__ long long d_s;
    __shared__ int k2_s;
    if (threadIdx.x == 0) {
      const double alpha = fx_alpha(S, cur, fx_hv_dot(S), d_s, k2_s);
      if (blockIdx.x == 0) S->alpha[S->j + 1] = alpha;
    }
    __syncthreads();
    d = d_s;
    k2 = k2_s;
  }
  longlong2* const keep = kKeep ? (longlong2*)store.slots[S->j + 1] : nullptr;
  A192 q2;
  long long mx = 0;
  // n is even (rows are padded to 32 elements): pairs of elements, two pairs in flight
  const longlong2* c2 = reinterpret_cast<const longlong2*>(xc);
  longlong2* p2 = reinterpret_cast<longlong2*>(xp);
  const int64_t n2 = n / 2;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto upd = [&](long long w, long long c) {
    const long long q = w + round_shift128(smul128(d, c), k2);
    const unsigned long long aq = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
    a192_add_sq(q2, aq);
    mx = max(mx, (long long)aq);
    return q;
  };
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += 2 * stride) {
    const bool two = i + stride < n2;
    const longlong2 w0 = p2[i], c0 = c2[i];
    longlong2 w1 = make_longlong2(0, 0), c1 = make_longlong2(0, 0);
    if (two) {
      w1 = p2[i + stride];
      c1 = c2[i + stride];
    }
    const longlong2 r0 = make_longlong2(upd(w0.x, c0.x), upd(w0.y, c0.y));
    p2[i] = r0;
    if (kKeep && keep) __stcs(keep + i, r0);
    if (two) {
      const longlong2 r1 = make_longlong2(upd(w1.x, c1.x), upd(w1.y, c1.y));
      p2[i + stride] = r1;
      if (kKeep && keep) __stcs(keep + i + stride, r1);
    }
  }
  fx_block_reduce(a192_get(q2), mx, pb + 4 * blockIdx.x);
  if (finish && last_cta(&S->tick_upd)) fx_finish_step(S, cur, pb, gridDim.x, plan, store);
}

__global__ void __launch_bounds__(kRedThreads)
fx_finish_kernel(LzScalars* S, int cur, const long long* __restrict__ pb, int nb, FxPlanArgs plan) {
  if (S->status == 0) fx_finish_step(S, cur, pb, nb, plan, LzStore{nullptr, nullptr, nullptr});
}

// ------------------------------------------------------------------ ground-state vector
// psi = sum_j y_j f_j accumulated in int64 with psi = 2^-60 P (|psi_i| stays below 4):
// P_i += round(c X_i 2^k) with c 2^k = y_j s_cur 2^60. Also tracks the index of the
// largest |P| (ties: lowest index) for the sign gauge.
__global__ void __launch_bounds__(kFxThreads)
fx_psi_accum_kernel(const LzScalars* __restrict__ S, int cur, const double* __restrict__ y, int jstep,
                    const long long* __restrict__ X, int64_t rows, int64_t cols, int64_t ld,
                    const int32_t* __restrict__ colpos, long long* __restrict__ P) {
  const double c = y[jstep] * S->scale[cur] * 0x1.0p60;
  long long m = 0;
  int k = -1;
  if (c != 0.0 && isfinite(c)) {
    k = ilogb(c) - 61;
    m = llrint(ldexp(c, -k));
  }
  const int64_t n = rows * cols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols, cc = i - r * cols;
    P[i] += round_shift((i128)m * X[r * ld + (colpos ? colpos[cc] : cc)], k);
  }
}

// Partial records of max |P| with its lowest index and of ||P||^2 (exact).
__device__ __forceinline__ void fx_psi_records(long long bv, long long bi, const I192& nrm,
                                               long long* amax, long long* part) {
  __shared__ long long sv[32], si[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long v2 = __shfl_down_sync(0xffffffffu, bv, o), i2 = __shfl_down_sync(0xffffffffu, bi, o);
    if (v2 > bv || (v2 == bv && i2 < bi)) bv = v2, bi = i2;
  }
  if ((threadIdx.x & 31) == 0) sv[threadIdx.x >> 5] = bv, si[threadIdx.x >> 5] = bi;
  fx_block_reduce(nrm, 0, part + 4 * blockIdx.x);  // (a barrier in it covers sv, si)
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (sv[w] > bv || (sv[w] == bv && si[w] < bi)) bv = sv[w], bi = si[w];
    amax[2 * blockIdx.x] = bv;
    amax[2 * blockIdx.x + 1] = bi;
  }
}

// P = sum_k round(y_{k+1} s_k 2^60 X_k) over the m stored vectors, two columns per thread, and
// the records of P. Every vector is read once, coalesced, four of them in flight; the element goes
// to its rank (scattered within its row) once. Bound by the ALU (66%: a 128-bit product and a
// rounding shift per element and vector) before HBM (3.5 TB/s): 24 vectors of 95 MB take 0.66 ms.
// Against regenerating the vectors (a second run of the m H.v and update passes and a
// read-modify-write of P per step) the half-filled 14-site ring's 78 take 2.1 ms instead of 26.
__global__ void __launch_bounds__(kFxThreads)
fx_psi_sum_kernel(const double* __restrict__ y, int m, LzStore store, int64_t rows, int64_t cols,
                  int64_t ld, const int32_t* __restrict__ rank, long long* __restrict__ P,
                  long long* __restrict__ amax, long long* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char psi_smem[];
  long long* mant = reinterpret_cast<long long*>(psi_smem);
  const longlong2** vec = reinterpret_cast<const longlong2**>(mant + m);
  int* expo = reinterpret_cast<int*>(vec + m);
  for (int k = threadIdx.x; k < m; k += blockDim.x) {
    const double c = y[k + 1] * store.vscale[k] * 0x1.0p60;
    long long q = 0;
    int e = -1;
    if (c != 0.0 && isfinite(c)) {
      e = ilogb(c) - 61;
      q = llrint(ldexp(c, -e));
    }
    mant[k] = q;
    expo[k] = e;
    vec[k] = reinterpret_cast<const longlong2*>(store.slots[k]);
  }
  __syncthreads();
  const int64_t pairs = rows * (ld / 2);
  long long bv = -1, bi = 0;
  A192 nrm;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < pairs;
       i += (int64_t)gridDim.x * blockDim.x) {
    long long s0 = 0, s1 = 0;
    int k = 0;
    for (; k + 4 <= m; k += 4) {
      longlong2 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = __ldcs(vec[k + q] + i);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        s0 += round_shift128(smul128(mant[k + q], x[q].x), expo[k + q]);
        s1 += round_shift128(smul128(mant[k + q], x[q].y), expo[k + q]);
      }
    }
    for (; k < m; ++k) {
      const longlong2 x = __ldcs(vec[k] + i);
      s0 += round_shift128(smul128(mant[k], x.x), expo[k]);
      s1 += round_shift128(smul128(mant[k], x.y), expo[k]);
    }
    const int64_t r = i / (ld / 2), p = 2 * (i - r * (ld / 2));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int32_t d = rank[p + q];
      if (d < 0) continue;
      const long long v = q ? s1 : s0, e = r * cols + d;
      P[e] = v;
      const long long av = v < 0 ? -v : v;
      a192_add_sq(nrm, (unsigned long long)av);
      if (av > bv || (av == bv && e < bi)) bv = av, bi = e;
    }
  }
  fx_psi_records(bv, bi, a192_get(nrm), amax, part);
}

// The same records for a P in memory.
__global__ void __launch_bounds__(kFxThreads)
fx_psi_records_kernel(const long long* __restrict__ P, int64_t n, long long* __restrict__ amax,
                      long long* __restrict__ part) {
  long long bv = -1, bi = 0;
  A192 nrm;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const long long v = P[i], av = v < 0 ? -v : v;
    a192_add_sq(nrm, (unsigned long long)av);
    if (av > bv) bv = av, bi = i;
  }
  fx_psi_records(bv, bi, a192_get(nrm), amax, part);
}

// psi (FP64) = gauge * P 2^-60 / ||P 2^-60||, gauge making the largest entry positive. The
// factor g (one CTA): 2 x 608 records, a thread per record.
__global__ void __launch_bounds__(kFxThreads)
fx_psi_gauge_kernel(const long long* __restrict__ P, const long long* __restrict__ amax,
                    const long long* __restrict__ part, int n, double* __restrict__ g) {
  __shared__ long long sv[kFxThreads], si[kFxThreads];
  long long bv = -1, bi = 0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) {
    const long long v = amax[2 * b], i = amax[2 * b + 1];
    if (v > bv || (v == bv && i < bi)) bv = v, bi = i;
  }
  sv[threadIdx.x] = bv;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      const long long v2 = sv[threadIdx.x + o], i2 = si[threadIdx.x + o];
      if (v2 > sv[threadIdx.x] || (v2 == sv[threadIdx.x] && i2 < si[threadIdx.x])) {
        sv[threadIdx.x] = v2;
        si[threadIdx.x] = i2;
      }
    }
    __syncthreads();
  }
  I192 sum;
  long long unused;
  fx_sum_partials(part, n, sum, unused);
  if (threadIdx.x == 0) *g = (P[si[0]] < 0 ? -1.0 : 1.0) / sqrt(i192_to_double(sum));
}

// In place: the int64 P becomes the FP64 psi.
__global__ void __launch_bounds__(kFxThreads)
fx_psi_out_kernel(long long* __restrict__ P, int64_t n, const double* __restrict__ gauge) {
  const double g = *gauge;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    P[i] = __double_as_longlong((double)P[i] * g);
}

// ------------------------------------------------------------------ host side
static int fx_red_grid(int64_t n) {
  const int64_t want = (n + kFxThreads - 1) / kFxThreads;
  const int64_t cap = (int64_t)sm_count() * 4;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

static FxHvArgs fx_args(const ed_basis* b, int64_t ld) {
  FxHvArgs a;
  a.up_bits = b->up.bits;
  a.dn_bits = b->dn.bits;
  a.hop_up = b->up.hop;
  a.hop_dn = b->dn.hop;
  a.dim_up = b->up.dim;
  a.dim_dn = b->dn.dim;
  a.ld = ld;
  a.maxhops_up = b->up.maxhops;
  a.maxhops_dn = b->dn.maxhops;
  return a;
}

template <int R>
static size_t fx_smem(const ed_basis* b) {
  return (size_t)(b->dn.dim + 1) * R * 8 + (size_t)R * b->up.maxhops * 4;
}

static int smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return v;
}

static int fx_rows(const ed_basis* b) {
  if (b->up.dim < kMinRowsStaged) return 0;  // few rows: the element-parallel kernel
  const size_t lim = (size_t)smem_optin();
  if (fx_smem<2>(b) <= lim && b->up.dim >= 2) return 2;
  if (fx_smem<1>(b) <= lim) return 1;
  return 0;
}

ed_status fx_psi_accum(const ed_basis* b, const LzScalars* S, int cur, const double* y, int j,
                       const long long* X, int64_t ld, const int32_t* colpos, long long* P,
                       cudaStream_t s) {
  fx_psi_accum_kernel<<<fx_red_grid(b->dim), kFxThreads, 0, s>>>(S, cur, y, j, X, b->up.dim,
                                                                  b->dn.dim, ld, colpos, P);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

ed_status fx_psi_sum(const ed_basis* b, const double* y, int m, const LzStore& store, int64_t ld,
                     const int32_t* rank, long long* P, long long* part, cudaStream_t s) {
  const int g = fx_red_grid(b->dim);
  fx_psi_sum_kernel<<<g, kFxThreads, (size_t)m * 20, s>>>(y, m, store, b->up.dim, b->dn.dim, ld, rank,
                                                          P, part, part + 2 * g);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

ed_status fx_psi_finish(const ed_basis* b, long long* P, bool have_records, long long* part,
                        cudaStream_t s) {
  const int g = fx_red_grid(b->dim);
  if (!have_records) fx_psi_records_kernel<<<g, kFxThreads, 0, s>>>(P, b->dim, part, part + 2 * g);
  double* gauge = reinterpret_cast<double*>(part + 6 * g);
  fx_psi_gauge_kernel<<<1, kFxThreads, 0, s>>>(P, part, part + 2 * g, g, gauge);
  fx_psi_out_kernel<<<g, kFxThreads, 0, s>>>(P, b->dim, gauge);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

ed_status fx_prepare(const ed_basis* b) {
  const int R = fx_rows(b);
  if (R == 2)
    ED_TRY_CUDA(allow_max_smem(fx_hv_staged_kernel<2>));
  if (R == 1)
    ED_TRY_CUDA(allow_max_smem(fx_hv_staged_kernel<1>));
  return ED_OK;
}

ed_status fx_init(LzScalars* S, const long long* part, int n, cudaStream_t s) {
  fx_init_kernel<<<1, kFxThreads, 0, s>>>(S, part, n);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

ed_status fx_exponent(const ed_basis* b, const double* f1, long long* part, cudaStream_t s, int* E) {
  const int g = fx_red_grid(b->dim);
  unsigned long long* pm = reinterpret_cast<unsigned long long*>(part);
  fx_absmax_kernel<<<g, kFxThreads, 0, s>>>(f1, b->dim, pm);
  fx_absmax_final<<<1, kFxThreads, 0, s>>>(pm, g, pm + g);
  ED_TRY_CUDA(cudaGetLastError());
  unsigned long long mb = 0;
  ED_TRY_CUDA(cudaMemcpyAsync(&mb, pm + g, sizeof(mb), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  const int ef = (int)(mb >> 52);
  ED_CHECK_ARG(ef != 0x7FF, "f1 holds a non-finite value");
  ED_CHECK_ARG(mb != 0, "f1 is the zero vector");
  *E = ef ? ef - 1022 : -1022;  // |f1| < 2^E
  return ED_OK;
}

ed_status fx_plan(const FxRun& fx, double t, double U, int cur, LzScalars* S, cudaStream_t s) {
  fx_plan_kernel<<<1, 32, 0, s>>>(S, cur, FxPlanArgs{t, U, fx.hops, fx.nmax, fx.vb});
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

ed_status fx_step(const ed_basis* b, const FxRun& fx, double t, double U, long long* const B[2],
                  int cur, int64_t ld, LzScalars* S, long long* pa, long long* pb,
                  cudaStream_t s, cudaEvent_t ev0, cudaEvent_t ev1, const Hv2Plan* plan,
                  const LzStore& store, const Reorth* ro) {
  if (ev0) ED_TRY_CUDA(cudaEventRecord(ev0, s));
  const FxHvArgs a = fx_args(b, ld);
  const int R = plan ? -1 : fx_rows(b);
  if (plan) {
    ed_status r = hv2_launch(plan, b, t, U, B[cur], B[1 - cur], S, cur, pa, s);
    if (r != ED_OK) return r;
  } else if (R == 2) {
    const int grid = (int)((b->up.dim + 1) / 2);
    fx_hv_staged_kernel<2><<<grid, kFxThreads, fx_smem<2>(b), s>>>(a, B[cur], B[1 - cur], S);
  } else if (R == 1) {
    const int grid = (int)b->up.dim;
    fx_hv_staged_kernel<1><<<grid, kFxThreads, fx_smem<1>(b), s>>>(a, B[cur], B[1 - cur], S);
  } else {
    const int grid = fx_red_grid(b->dim) * 2;
    fx_hv_global_kernel<<<grid, kFxThreads, 0, s>>>(a, B[cur], B[1 - cur], S);
  }
  ED_TRY_CUDA(cudaGetLastError());
  if (ev1) ED_TRY_CUDA(cudaEventRecord(ev1, s));
  const int64_t n = b->up.dim * ld;
  const int ug = fx_red_grid(n);
  const FxPlanArgs next = {t, U, fx.hops, fx.nmax, fx.vb};
  const bool between = ro && ro_between(ro);  // passes between the update and the finish
  const bool ready = plan && hv2_ticket(plan);
  const auto update = store.slots ? (ready ? fx_update_kernel<true, true> : fx_update_kernel<true, false>)
                                  : (ready ? fx_update_kernel<false, true> : fx_update_kernel<false, false>);
  update<<<ug, kFxThreads, 0, s>>>(S, cur, B[cur], B[1 - cur], n, pb, !between, next, store);
  if (between) {
    const ed_status r = ro_apply(ro, S, B[1 - cur], pb, ug, s);
    if (r != ED_OK) return r;
    fx_finish_kernel<<<1, kRedThreads, 0, s>>>(S, cur, pb, ug, next);
  }
  ED_TRY_CUDA(cudaGetLastError());
  if (between) return ro_store(ro, S, 1 - cur, B[1 - cur], s);
  return ED_OK;
}

}  // namespace ed
