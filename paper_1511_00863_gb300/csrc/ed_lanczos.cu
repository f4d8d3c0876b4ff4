// Lanczos iteration (Sec. 2.2, Algorithm 1) on the device, the random start vector, and
// the lowest eigenvalue of the tridiagonal T by Sturm-sequence bisection in FP64.
//
// One step j is two launches on the run's stream:
//   1. fused H.v:  w = H f_j - b_j f_{j-1}, written over the f_{j-1} buffer, with per-CTA
//      partial sums of w . f_j  (ed_hv.cu, LzHvArgs);
//   2. update:     a_j = the sum of the partials (one warp of every CTA, in the same order, or
//      on long vectors the last CTA of the H.v: kTicketMin), q = w - a_j f_j in place, per-CTA partial sums of q . q; the last CTA sums them
//      (finish): b_{j+1} = sqrt(sum), breakdown test, f_{j+1} = q / b_{j+1} kept implicit
//      as a buffer scale.
// (Reorthogonalisation runs between the update and a finish launch of its own.)
// E0(j) = lambda_min(T_j) and the convergence test run beside the next steps, on a stream of
// their own (lz_check_kernel).
// Each buffer holds an unnormalised vector B with f = scale * B, so no pass rescales it.
// Once the run stops (breakdown, convergence, max_steps) every later kernel returns at
// entry; ed_lanczos_solve replays a captured CUDA graph of a few steps and reads the status of
// one batch of replays while the next one runs.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include "ed_fixed.cuh"
#include "ed_internal.cuh"
#include "ed_lanczos_dev.cuh"

namespace ed {

// ------------------------------------------------------------------ start vector
// Element i of the start vector is h_i 2^-52 / ||.||, h_i = (top 53 bits of the (i+1)-th
// SplitMix64 output) - 2^52 (start_int, ed_fixed.cuh). Everything per element is integer
// arithmetic: GB300's FP64 rate made the conversion, the product and the rounding of an element
// 15-17 ps and its share of the norm 7 ps (2.8 ms of a 166 M element FP32 start).

// Partial sums of x_i^2 = h_i^2 2^-104 over the raw start vector, exact per CTA.
__global__ void __launch_bounds__(kRedThreads)
start_norm_kernel(uint64_t seed, int64_t n, double* __restrict__ partial) {
  __shared__ long long tot[4];
  A192 acc;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const long long h = start_int(seed, (uint64_t)i);
    a192_add_sq(acc, (unsigned long long)(h < 0 ? -h : h));
  }
  fx_block_reduce(a192_get(acc), 0, tot);
  if (threadIdx.x == 0) {
    I192 v;
    v.lo = ((u128)(unsigned long long)tot[1] << 64) | (u128)(unsigned long long)tot[0];
    v.hi = tot[2];
    partial[blockIdx.x] = scale2(i192_to_double(v), -104);
  }
}

// RN(h 2^-52 inv) in FP64, then to T (both to nearest even): the product of the 52-bit h and
// inv's mantissa M 2^-63 (top bit set; inv = M 2^(e_inv - 63)) in integers.
template <typename T>
__device__ __forceinline__ T start_scaled(long long h, unsigned long long M, int e_inv) {
  if (h == 0) return T(0);
  const unsigned long long a = (unsigned long long)(h < 0 ? -h : h);
  const int lz = __clzll(a);
  const unsigned long long an = a << lz;
  unsigned long long hi = __umul64hi(an, M), lo = an * M;
  int e = e_inv - lz + 12;  // exponent of the product with hi's top bit set
  if (!(hi >> 63)) {
    hi = (hi << 1) | (lo >> 63);
    lo <<= 1;
    --e;
  }
  // 64 significant bits and a sticky remainder: to 53 bits
  unsigned long long m = hi >> 11, rem = (hi & 0x7FF) | (lo ? 1ull : 0ull);
  m += rem > 0x400 || (rem == 0x400 && (m & 1));
  if (m >> 53) {
    m >>= 1;
    ++e;
  }
  if constexpr (sizeof(T) == 8) {
    return __longlong_as_double((long long)((m & ((1ull << 52) - 1)) | ((unsigned long long)(e + 1023) << 52) |
                                            (h < 0 ? 1ull << 63 : 0ull)));
  } else {
    const unsigned r = (unsigned)(m & ((1u << 29) - 1));
    unsigned f = (unsigned)(m >> 29);
    f += r > (1u << 28) || (r == (1u << 28) && (f & 1u));
    // (a carry out of the 24 bits moves into the exponent field by itself)
    return __uint_as_float(f - (1u << 23) + ((unsigned)(e + 127) << 23) + (h < 0 ? 1u << 31 : 0u));
  }
}

// A vector in the library's layout: row r, scalar p of a row (cx = 2 scalars (re, im) per complex
// element) at out[r lds + p]; the element at column e = p / cx is the one of down rank
// rank[e] (-1: a pad, holds 0; rank NULL: rank e for e < cols). CTAs take runs of kRun scalars of
// a row and write them in column order, pads included.
constexpr int kRun = 2048;
struct RowRuns {
  int64_t rows, cols, lds, runs;  // cols in elements, lds in scalars, runs per row
  const int32_t* __restrict__ rank;
  int cx;
};

// f(i, o) for every scalar: i its index in the dense vector (-1: a pad), o its place.
template <typename F>
__device__ __forceinline__ void for_rows(const RowRuns& L, F f) {
  for (int64_t it = blockIdx.x; it < L.rows * L.runs; it += gridDim.x) {
    const int64_t r = it / L.runs, c0 = (it - r * L.runs) * kRun;
    const int64_t c1 = c0 + kRun < L.lds ? c0 + kRun : L.lds;
    for (int64_t p = c0 + threadIdx.x; p < c1; p += blockDim.x) {
      const int64_t e = L.cx == 2 ? p >> 1 : p;
      const int64_t d = L.rank ? (int64_t)L.rank[e] : (e < L.cols ? e : -1);
      f(d < 0 ? -1 : L.cx * (r * L.cols + d) + (L.cx == 2 ? p & 1 : 0), r * L.lds + p);
    }
  }
}

// raw_i / ||raw|| rounded to T, in the layout L.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
start_write_kernel(uint64_t seed, RowRuns L, const double* __restrict__ partial, int nparts, T* __restrict__ out) {
  __shared__ double red[33];
  const double inv = 1.0 / sqrt(block_sum_array(partial, nparts, red));
  const unsigned long long b = (unsigned long long)__double_as_longlong(inv);
  const unsigned long long M = (b << 11) | (1ull << 63);  // inv is positive and normal
  const int e_inv = (int)(b >> 52) - 1023;
  for_rows(L, [&](int64_t i, int64_t o) {
    out[o] = i < 0 ? T(0) : start_scaled<T>(start_int(seed, (uint64_t)i), M, e_inv);
  });
}

// Copy a dense caller vector into the layout L and accumulate its squared norm.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
copy_in_kernel(const T* __restrict__ src, RowRuns L, T* __restrict__ dst, double* __restrict__ partial) {
  __shared__ double red[33];
  DotAcc<T> acc;
  for_rows(L, [&](int64_t i, int64_t o) {
    const T v = i < 0 ? T(0) : src[i];
    dst[o] = v;
    acc.add(v, v);
  });
  const double v = block_sum(acc.get(), red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v;
}

// The same copies in fixed point (ed_fixed.cu): X_i = 2 h_i moved to the 2^vb range, and a
// caller's FP64 vector X_i = f_i 2^(vb - E), |f| < 2^E, by integer manipulation of the IEEE fields
// (round half up where bits fall off); records of sum X^2 (exact) and max |X|.
__global__ void __launch_bounds__(kRedThreads)
fx_start_kernel(uint64_t seed, RowRuns L, int vb, long long* __restrict__ X, long long* __restrict__ part) {
  A192 acc;
  long long mx = 0;
  for_rows(L, [&](int64_t i, int64_t o) {
    const long long v = i < 0 ? 0 : shift_signed(2 * start_int(seed, (uint64_t)i), vb - 53);
    X[o] = v;
    const long long av = v < 0 ? -v : v;
    a192_add_sq(acc, (unsigned long long)av);
    mx = max(mx, av);
  });
  fx_block_reduce(a192_get(acc), mx, part + 4 * blockIdx.x);
}

__global__ void __launch_bounds__(kRedThreads)
fx_copy_in_kernel(const double* __restrict__ f, RowRuns L, int vb, int E, long long* __restrict__ X,
                  long long* __restrict__ part) {
  A192 acc;
  long long mx = 0;
  for_rows(L, [&](int64_t i, int64_t o) {
    long long v = 0;
    if (i >= 0) {
      const unsigned long long bits = (unsigned long long)__double_as_longlong(f[i]);
      const int ef = (int)((bits >> 52) & 0x7FF);
      long long mant = (long long)(bits & 0xFFFFFFFFFFFFFull);
      int e2 = -1074;
      if (ef) {
        mant |= 1LL << 52;
        e2 = ef - 1075;
      }
      v = shift_signed(mant, e2 + vb - E);
      if (bits >> 63) v = -v;
    }
    X[o] = v;
    const long long av = v < 0 ? -v : v;
    a192_add_sq(acc, (unsigned long long)av);
    mx = max(mx, av);
  });
  fx_block_reduce(a192_get(acc), mx, part + 4 * blockIdx.x);
}

// The rank table of rank order: column p is rank p, -1 for a pad.
__global__ void rank_kernel(int64_t cols, int64_t ld, int32_t* __restrict__ rank) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ld; i += (int64_t)gridDim.x * blockDim.x)
    rank[i] = i < cols ? (int32_t)i : -1;
}

__global__ void init_scalars_kernel(LzScalars* S, const double* __restrict__ partial,
                                    int nparts, int use_partial) {
  __shared__ double red[33];
  double nrm2 = 1.0;
  if (use_partial) nrm2 = block_sum_array(partial, nparts, red);
  if (threadIdx.x == 0) S->scale[0] = 1.0 / sqrt(nrm2);
}

// ------------------------------------------------------------------ update
// Whole CTA: b_{j+1} and f_{j+1}'s scale from the nb partial sums of q . q.
__device__ __forceinline__ void lz_finish_step(LzScalars* S, int cur, const double* pb, int nb,
                                               double* red, double* vscale) {
  const double b2 = block_sum_array(pb, nb, red);
  if (threadIdx.x != 0) return;
  const double beta = sqrt(b2);
  const int j = S->j + 1;
  if (finish_step(S, j, beta)) {
    S->scale[1 - cur] = 1.0 / beta;
    if (vscale) vscale[j] = 1.0 / beta;
  }
}

// finish: the last CTA ends the step (lz_finish_step); otherwise lz_finish_kernel does, after
// the reorthogonalisation. kKeep: q goes to the step's slot of `store` too.
template <typename T, bool kKeep>
__global__ void __launch_bounds__(kRedThreads)
lz_update_kernel(LzScalars* S, int cur, const T* __restrict__ bcur, T* __restrict__ bprev,
                 int64_t n, const double* __restrict__ pa, int na, double* __restrict__ pb, int finish,
                 LzStore store) {
  __shared__ double red[33];
  __shared__ double alpha_s;
  if (S->status != 0) return;
  if (na == 0) {  // the H.v left a_j finished
    if (threadIdx.x == 0) alpha_s = S->alpha[S->j + 1];
  } else if (na <= 2048) {
    if (threadIdx.x < 32) {
      const double a = warp_sum_array(pa, na);
      if (threadIdx.x == 0) alpha_s = a;
    }
  } else {
    const double a = block_sum_array(pa, na, red);
    if (threadIdx.x == 0) alpha_s = a;
  }
  __syncthreads();
  if (na > 0 && blockIdx.x == 0 && threadIdx.x == 0) S->alpha[S->j + 1] = alpha_s;
  const T coef = (T)(alpha_s * S->scale[cur]);
  DotAcc<T> acc;
  // n is a multiple of 32 (padded rows): 16-byte vectors of 16 / sizeof(T) elements
  constexpr int VE = 16 / sizeof(T);
  typedef typename std::conditional<sizeof(T) == 4, float4, double2>::type Vec;
  const Vec* c4 = reinterpret_cast<const Vec*>(bcur);
  Vec* p4 = reinterpret_cast<Vec*>(bprev);
  Vec* const keep = kKeep ? (Vec*)store.slots[S->j + 1] : nullptr;
  const int64_t nv = n / VE;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nv;
       i += (int64_t)gridDim.x * blockDim.x) {
    Vec w = p4[i];
    const Vec c = c4[i];
    T* wv = reinterpret_cast<T*>(&w);
    const T* cv = reinterpret_cast<const T*>(&c);
#pragma unroll
    for (int e = 0; e < VE; ++e) {
      const T q = wv[e] - coef * cv[e];
      wv[e] = q;
      acc.add(q, q);
    }
    p4[i] = w;
    if (kKeep && keep) __stcs(keep + i, w);
  }
  const double v = block_sum(acc.get(), red);
  if (threadIdx.x == 0) pb[blockIdx.x] = v;
  if (finish && last_cta(&S->tick_upd)) lz_finish_step(S, cur, pb, gridDim.x, red, kKeep ? store.vscale : nullptr);
}

__global__ void __launch_bounds__(kRedThreads)
lz_finish_kernel(LzScalars* S, int cur, const double* __restrict__ pb, int nb) {
  __shared__ double red[33];
  if (S->status == 0) lz_finish_step(S, cur, pb, nb, red, nullptr);
}

__global__ void __launch_bounds__(kRedThreads)
lz_energy_kernel(const LzScalars* S, double* out) {
  const int j = S->j;
  if (j < 1) {
    if (threadIdx.x == 0) *out = NAN;
    return;
  }
  __shared__ double sturm_work[kSturmWork];
  const double E = sturm_lowest(S->alpha, S->beta, j, NAN, sturm_work);
  if (threadIdx.x == 0) *out = E;
}

// E0(i) = lambda_min(T_i) for i = 1 .. j, block i - 1 for step i (all != 0), or for i = j
// alone: the history of a run without convergence test. The steps' scalars are final, so the
// bisections run side by side on as many SMs instead of one after each step on one SM (FP64
// multisection: 4-9 rounds of ~9 us each on GB300).
__global__ void __launch_bounds__(kRedThreads)
lz_history_kernel(LzScalars* S, int all) {
  const int i = all ? (int)blockIdx.x + 1 : S->j;
  if (i < 1 || i > S->j) return;
  __shared__ double sturm_work[kSturmWork];
  const double E = sturm_lowest(S->alpha, S->beta, i, NAN, sturm_work);
  if (threadIdx.x == 0) S->E0[i] = E;
}

// The convergence test of the `gridDim.x` steps after S->chk, one CTA per step: E0(i) =
// lambda_min(T_i), then the last CTA to finish tests |E0(i) - E0(i-1)| in step order and
// records the first i that passes (conv_j; the next finish kernel stops the run). It needs a_i, b_i alone, which are final
// once step i is done, so it runs on a stream of its own beside the next steps' H.v: a
// bisection takes 35-50 us on one SM (the float-float and FP64 chains of sturm_lowest), which
// after every step was 41 of the 52 us of a step on the 12-site ring (48,400 states) and 51
// of 500 us on the 4x4 lattice (19 M). The steps enqueued meanwhile are not part of the
// result: everything a caller sees ends at conv_j.
// E0(chk), when known, bounds every later E0(i) from above (Cauchy interlacing).
__global__ void __launch_bounds__(kRedThreads)
lz_check_kernel(LzScalars* S) {
  __shared__ double sturm_work[kSturmWork];
  __shared__ int base_s, j_s, open_s, broke_s;
  if (threadIdx.x == 0) {  // once per CTA: the steps beside this kernel advance j
    base_s = S->chk;
    open_s = S->conv_j == 0;
    broke_s = *(volatile int*)&S->status == 1;  // then j is final
    __threadfence();
    j_s = *(volatile int*)&S->j;
  }
  __syncthreads();
  const int base = base_s;
  const int i = base + 1 + (int)blockIdx.x;
  // the steps up to base + gridDim.x are done, unless the run stopped before them
  if (open_s && i >= 1 && i <= j_s) {
    const double E = sturm_lowest(S->alpha, S->beta, i, base >= 1 ? S->E0[base] : NAN, sturm_work);
    if (threadIdx.x == 0) S->E0[i] = E;
  }
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(&S->tick_chk, 1u) != gridDim.x - 1) return;
  S->tick_chk = 0;
  __threadfence();
  if (open_s) {
    const int last = min(base + (int)gridDim.x, j_s);
    for (int k = max(base + 1, 2); k <= last; ++k) {
      const double E = __ldcg(&S->E0[k]), P = __ldcg(&S->E0[k - 1]);
      if (broke_s && k == j_s) break;  // a step that broke down ends the run by itself
      if (fabs(E - P) <= S->tol * fmax(fabs(E), 1.0)) {
        S->conv_j = k;
        break;
      }
    }
  }
  S->chk = base + (int)gridDim.x;
}

// Eigenvector y of T_m for its lowest eigenvalue lam (tridiag_ritz_vector): one thread's chain of
// dependent FP64 operations over arrays in shared memory (5 (m + 2) doubles; from global memory,
// 600 cycles a load instead of 30, m = 64 took 87 us).
__global__ void lz_ritz_kernel(const LzScalars* S, int m, double lam, double* y) {
  extern __shared__ double ritz_smem[];
  const int n = m + 2;
  double *a = ritz_smem, *b = a + n, *ys = b + n, *work = ys + n;
  for (int i = threadIdx.x; i < n; i += 32) a[i] = S->alpha[i], b[i] = S->beta[i];
  __syncwarp();
  if (threadIdx.x == 0) tridiag_ritz_vector(a, b, m, lam, ys, work);
  __syncwarp();
  for (int i = threadIdx.x; i < n; i += 32) y[i] = ys[i];
}

static RowRuns row_runs(int64_t rows, int64_t cols, int64_t ld, int cx, const int32_t* rank) {
  return RowRuns{rows, cols, cx * ld, (cx * ld + kRun - 1) / kRun, rank, cx};
}

static int red_grid(int64_t n) {
  const int64_t want = (n + kRedThreads - 1) / kRedThreads;
  const int64_t cap = (int64_t)sm_count() * 4;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace ed

using namespace ed;

struct ed_lanczos {
  const ed_basis* basis = nullptr;
  ed_opts opts{};
  int device = 0;
  cudaStream_t stream = nullptr;
  int64_t ld = 0;      // padded row stride (elements)
  int64_t n = 0;       // dim_up * ld
  size_t esize = 8;
  void* B[2] = {nullptr, nullptr};
  int cur = 0;         // buffer holding f_j
  LzScalars* S = nullptr;
  double* pa = nullptr;  // partials of the H.v pass
  double* pb = nullptr;  // partials of the update pass
  double* tmp = nullptr;
  int64_t npa = 0, npb = 0;
  int hv_grid = 0;
  bool stopped = false;
  double graph_t[4] = {}, graph_U[4] = {};  // parameters of the captured graphs
  bool fx = false;     // ED_F64: int64 fixed-point buffers (ed_fixed.cu)
  FxRun fxr{};
  Hv2Plan* plan = nullptr;  // fused H.v on the padded layout (ed_hv2.cu), if it fits
  Reorth* ro = nullptr;     // stored Lanczos vectors when opts.reorth != 0 (ed_reorth.cu)
  LzStore store{nullptr, nullptr, nullptr};  // where the update pass keeps the vectors
  cudaGraphExec_t graph[4] = {};  // without / with the convergence test, + 2: vectors kept in `slots`
  // ground-state vectors only: slot table, scales and maxima of the kept vectors, y of T_m with
  // the inverse iteration's work, ranks by column without a plan
  void** slots = nullptr;
  double* vscale = nullptr;
  long long* vmax = nullptr;
  double* ywork = nullptr;
  int32_t* rank = nullptr;
  // solves only (lz_iterate): the checks' stream, fork and join events of the capture, one event
  // per batch in flight and the host's copies of the run's scalars (pinned)
  cudaStream_t check_stream = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_batch[2] = {nullptr, nullptr};
  LzScalars* host = nullptr;  // [1] and the two batches' headers behind it
};

// Before the first step of a call: the fixed-point coefficients for these parameters.
static ed_status lz_plan(const ed_lanczos* st, const ed_params* p) {
  return st->fx ? fx_plan(st->fxr, p->t, p->U, st->cur, st->S, st->stream) : ED_OK;
}

static ed_status lz_launch_step(ed_lanczos* st, const ed_params* p, cudaStream_t s,
                                cudaEvent_t ev0 = nullptr, cudaEvent_t ev1 = nullptr) {
  const ed_basis* b = st->basis;
  const int c = st->cur;
  if (st->fx) {
    long long* const B[2] = {(long long*)st->B[0], (long long*)st->B[1]};
    ed_status r = fx_step(b, st->fxr, p->t, p->U, B, c, st->ld, st->S, (long long*)st->pa,
                          (long long*)st->pb, s, ev0, ev1, st->plan, st->store, st->ro);
    if (r == ED_OK) st->cur = 1 - c;
    return r;
  }
  LzHvArgs lz{st->S, c, st->pa};
  int grid = 0;
  ed_status r;
  if (ev0) ED_TRY_CUDA(cudaEventRecord(ev0, s));
  const ed_dtype dt = st->opts.dtype;
  if (st->plan) {
    grid = hv2_ticket(st->plan) ? 0 : hv2_grid(st->plan);  // (0: a_j is finished)
    r = hv2_launch(st->plan, b, p->t, p->U, st->B[c], st->B[1 - c], st->S, c, st->pa, s);
  } else if (dt == ED_C32) {
    r = launch_hvc<float>(b, p->t, p->U, st->B[c], st->B[1 - c], st->ld, s, &lz, &grid);
  } else if (dt == ED_C64) {
    r = launch_hvc<double>(b, p->t, p->U, st->B[c], st->B[1 - c], st->ld, s, &lz, &grid);
  } else if (dt == ED_F64_NATIVE)
    r = launch_hv<double>(b, p->t, p->U, (const double*)st->B[c], (double*)st->B[1 - c], st->ld,
                          s, &lz, &grid);
  else
    r = launch_hv<float>(b, p->t, p->U, (const float*)st->B[c], (float*)st->B[1 - c], st->ld,
                         s, &lz, &grid);
  if (r != ED_OK) return r;
  if (ev1) ED_TRY_CUDA(cudaEventRecord(ev1, s));
  // the update works on scalars: a complex vector is 2 n of them (a_j, b_j are real)
  const int64_t ns = is_complex(dt) ? 2 * st->n : st->n;
  const int ug = red_grid(ns);
  const bool between = st->ro && ro_between(st->ro);  // passes between the update and the finish
  const bool keep = st->store.slots != nullptr;
  if (dt == ED_F64_NATIVE || dt == ED_C64)  // (only FP32 and fixed-point runs keep their vectors here)
    lz_update_kernel<double, false><<<ug, kRedThreads, 0, s>>>(
        st->S, c, (const double*)st->B[c], (double*)st->B[1 - c], ns, st->pa, grid, st->pb, !between, st->store);
  else if (keep)
    lz_update_kernel<float, true><<<ug, kRedThreads, 0, s>>>(
        st->S, c, (const float*)st->B[c], (float*)st->B[1 - c], ns, st->pa, grid, st->pb, !between, st->store);
  else
    lz_update_kernel<float, false><<<ug, kRedThreads, 0, s>>>(
        st->S, c, (const float*)st->B[c], (float*)st->B[1 - c], ns, st->pa, grid, st->pb, !between, st->store);
  ED_TRY_CUDA(cudaGetLastError());
  if (between) {
    if ((r = ro_apply(st->ro, st->S, st->B[1 - c], st->pb, ug, s)) != ED_OK) return r;
    lz_finish_kernel<<<1, kRedThreads, 0, s>>>(st->S, c, st->pb, ug);
    ED_TRY_CUDA(cudaGetLastError());
  }
  if (between && (r = ro_store(st->ro, st->S, 1 - c, st->B[1 - c], s)) != ED_OK) return r;
  st->cur = 1 - c;
  return ED_OK;
}

// internal: also accept reorth = 3 (store the vectors without reorthogonalising; the FP32
// phase of ed_lanczos_solve_mixed)
static ed_status check_opts(const ed_opts* o, bool internal = false) {
  ED_CHECK_ARG(o != nullptr, "opts is NULL");
  ED_CHECK_ARG(o->max_steps >= 1 && o->max_steps <= ED_MAX_STEPS,
               "max_steps = %d outside [1, %d]", o->max_steps, ED_MAX_STEPS);
  ED_CHECK_ARG(o->dtype == ED_F64 || o->dtype == ED_F32 || o->dtype == ED_F64_NATIVE ||
                   is_complex(o->dtype),
               "unknown dtype %d", (int)o->dtype);
  ED_CHECK_ARG(o->reorth >= 0 && o->reorth <= (internal ? 3 : 2),
               "reorth = %d outside 0 (none), 1 (full), 2 (partial)", o->reorth);
  ED_CHECK_ARG(o->reorth == 0 || !is_complex(o->dtype),
               "reorthogonalisation is available for the real dtypes only");
  ED_CHECK_ARG(std::isfinite(o->tol), "tol is not finite");
  return ED_OK;
}

extern "C" ed_status ed_start_vector(int64_t dim, uint64_t seed, ed_dtype dtype, void* out,
                                     void* stream) {
  clear_error();
  ED_CHECK_ARG(dim >= 1, "ed_start_vector: dim < 1");
  ED_CHECK_ARG(out != nullptr && aligned16(out), "ed_start_vector: out NULL or not 16-byte aligned");
  ED_CHECK_ARG(dtype == ED_F64 || dtype == ED_F32 || dtype == ED_F64_NATIVE,
               "ed_start_vector: unknown dtype");
  cudaStream_t s = (cudaStream_t)stream;
  const int g = red_grid(dim);
  double* part = nullptr;
  ED_TRY_CUDA(cudaMallocAsync((void**)&part, g * sizeof(double), s));
  const RowRuns dense = row_runs(1, dim, dim, 1, nullptr);
  start_norm_kernel<<<g, kRedThreads, 0, s>>>(seed, dim, part);
  if (dtype != ED_F32)
    start_write_kernel<double><<<g, kRedThreads, 0, s>>>(seed, dense, part, g, (double*)out);
  else
    start_write_kernel<float><<<g, kRedThreads, 0, s>>>(seed, dense, part, g, (float*)out);
  cudaError_t e = cudaGetLastError();
  cudaFreeAsync(part, s);
  if (e != cudaSuccess) {
    set_error("ed_start_vector: %s", cudaGetErrorString(e));
    return ED_ERR_CUDA;
  }
  return ED_OK;
}

// ------------------------------------------------------------------ no-allocation variant
// Scratch of ed_start_vector_noalloc: the per-CTA partial sums of the squared norm. One
// copy per device that loads the library, kept until the process exits; every call shares
// it, so calls that overlap on the GPU race. Each call writes all the slots it reads, so
// nothing needs clearing between calls.
constexpr int kNoAllocPartials = 4096;
static __device__ __align__(256) double g_start_partials[kNoAllocPartials];

// Device address of g_start_partials on the current device (in host code the symbol names
// a host-side stand-in, not device memory). Resolved once per device, with that device
// current, on the first call there.
static ed_status noalloc_scratch(double** out) {
  static std::mutex mu;
  static double* addr[64] = {nullptr};
  int dev = 0;
  ED_TRY_CUDA(cudaGetDevice(&dev));
  ED_CHECK_ARG(dev >= 0 && dev < 64, "ed_start_vector_noalloc: device ordinal %d not supported", dev);
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_start_partials);
    if (e != cudaSuccess || p == nullptr) {
      set_error("ed_start_vector_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return ED_ERR_CUDA;
    }
    addr[dev] = (double*)p;
  }
  *out = addr[dev];
  return ED_OK;
}

extern "C" ed_status ed_start_vector_noalloc(int64_t dim, uint64_t seed, ed_dtype dtype, void* out,
                                             void* stream) {
  clear_error();
  ED_CHECK_ARG(dim >= 1, "ed_start_vector_noalloc: dim < 1");
  ED_CHECK_ARG(out != nullptr && aligned16(out),
               "ed_start_vector_noalloc: out NULL or not 16-byte aligned");
  ED_CHECK_ARG(dtype == ED_F64 || dtype == ED_F32 || dtype == ED_F64_NATIVE,
               "ed_start_vector_noalloc: unknown dtype");
  const int g = red_grid(dim);
  ED_CHECK_ARG(g <= kNoAllocPartials,
               "ed_start_vector_noalloc: needs %d partial sums, the static scratch holds %d", g,
               kNoAllocPartials);
  double* part = nullptr;
  const ed_status r = noalloc_scratch(&part);
  if (r != ED_OK) return r;
  cudaStream_t s = (cudaStream_t)stream;
  const RowRuns dense = row_runs(1, dim, dim, 1, nullptr);
  start_norm_kernel<<<g, kRedThreads, 0, s>>>(seed, dim, part);
  if (dtype != ED_F32)
    start_write_kernel<double><<<g, kRedThreads, 0, s>>>(seed, dense, part, g, (double*)out);
  else
    start_write_kernel<float><<<g, kRedThreads, 0, s>>>(seed, dense, part, g, (float*)out);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}

extern "C" void ed_lanczos_destroy(ed_lanczos* st) {
  if (!st) return;
  int prev = 0;
  cudaGetDevice(&prev);
  if (prev != st->device) cudaSetDevice(st->device);
  if (st->stream) cudaStreamSynchronize(st->stream);
  for (cudaGraphExec_t g : st->graph)
    if (g) cudaGraphExecDestroy(g);
  for (cudaEvent_t e : st->ev_batch)
    if (e) cudaEventDestroy(e);
  for (void* q : {(void*)st->slots, (void*)st->vscale, (void*)st->vmax, (void*)st->ywork, (void*)st->rank})
    if (q) cudaFree(q);
  if (st->ev_fork) cudaEventDestroy(st->ev_fork);
  if (st->ev_join) cudaEventDestroy(st->ev_join);
  if (st->check_stream) cudaStreamDestroy(st->check_stream);
  if (st->host) cudaFreeHost(st->host);
  if (st->plan) hv2_free(st->plan);
  if (st->ro) ro_free(st->ro);
  for (int i = 0; i < 2; ++i)
    if (st->B[i]) cudaFree(st->B[i]);
  if (st->S) cudaFree(st->S);
  if (st->pa) cudaFree(st->pa);
  if (st->pb) cudaFree(st->pb);
  if (st->tmp) cudaFree(st->tmp);
  if (prev != st->device) cudaSetDevice(prev);
  delete st;
}

// Bases below this many states use the default fused H.v variant order: timing every
// variant would cost more than their solves.
constexpr int64_t kAutotuneMinDim = (int64_t)1 << 22;

// The state's table of ranks by column: its plan's, or of rank order (built on first use).
static ed_status lz_rank(ed_lanczos* st, const int32_t** out) {
  if ((*out = hv2_rank(st->plan)) != nullptr || (*out = st->rank) != nullptr) return ED_OK;
  if (cudaMalloc((void**)&st->rank, (size_t)st->ld * sizeof(int32_t)) != cudaSuccess) {
    cudaGetLastError();
    st->rank = nullptr;
    set_error("Lanczos column ranks: out of device memory");
    return ED_ERR_OOM;
  }
  rank_kernel<<<red_grid(st->ld), kRedThreads, 0, st->stream>>>(st->basis->dn.dim, st->ld, st->rank);
  ED_TRY_CUDA(cudaGetLastError());
  *out = st->rank;
  return ED_OK;
}

static ed_status lz_alloc(const ed_basis* b, const ed_opts* o, cudaStream_t s, ed_lanczos** out) {
  *out = nullptr;
  ED_CHECK_ARG(b != nullptr, "basis is NULL");
  ed_status r = check_opts(o, true);
  if (r != ED_OK) return r;
  ED_CHECK_ARG(is_complex(o->dtype) || !b->has_tau(),
               "the lattice has complex amplitudes; use ED_C32 or ED_C64");
  ed_lanczos* st = new ed_lanczos();
  st->basis = b;
  st->opts = *o;
  cudaGetDevice(&st->device);
  st->stream = s;
  // bytes per element (a complex element is an (re, im) pair)
  st->esize = o->dtype == ED_F32 ? 4 : o->dtype == ED_C32 ? 8 : o->dtype == ED_C64 ? 16 : 8;
  st->fx = o->dtype == ED_F64;
  if (st->fx) st->fxr = fx_make(b);
  st->ld = (b->dn.dim + 31) / 32 * 32;
  bool split = false;  // the split-row kernel (its own row stride; no timing of variants)
  if (o->dtype == ED_F32 || o->dtype == ED_F64) {
    // rows longer than shared memory: the split-row fused H.v lays each row out as two
    // padded slices
    const int lds = hv2_split_ld(b, o->dtype == ED_F64 ? kHv2Fx : kHv2F32, o->schedule, s);
    if (lds > 0) {
      st->ld = lds;
      split = true;
    }
  }
  st->n = b->up.dim * st->ld;
  // partial sums: one double per CTA, or four int64 words per CTA on the fixed-point path
  st->npa = hv_max_grid(b) * (st->fx ? 4 : 1);
  st->npb = (int64_t)sm_count() * 4 * (st->fx ? 6 : 1) + 8;
  auto fail = [&](ed_status e) {
    ed_lanczos_destroy(st);
    return e;
  };
  for (int i = 0; i < 2; ++i) {
    if (cudaMalloc(&st->B[i], st->n * st->esize) != cudaSuccess) {
      set_error("Lanczos work vectors: out of device memory (%lld bytes each)",
                (long long)(st->n * st->esize));
      return fail(ED_ERR_OOM);
    }
  }
  if (o->reorth != 0) {
    const ed_status rr = ro_create(o->reorth, o->dtype, st->n, o->max_steps, b->dim, &st->ro);
    if (rr != ED_OK) return fail(rr);
    if (!ro_between(st->ro)) st->store = ro_slots(st->ro);  // mode 3
  }
  if (cudaMalloc((void**)&st->S, sizeof(LzScalars)) != cudaSuccess ||
      cudaMalloc((void**)&st->pa, st->npa * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&st->pb, st->npb * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&st->tmp, 64) != cudaSuccess) {
    set_error("Lanczos scalars: out of device memory");
    return fail(ED_ERR_OOM);
  }
  if (o->dtype == ED_F32 || o->dtype == ED_F64 || o->dtype == ED_C32) {
    const int mode = st->fx ? kHv2Fx : o->dtype == ED_C32 ? kHv2C32 : kHv2F32;
    int sched = o->schedule;
    if (split) sched = st->fx ? 30 : 31;
    if (sched < 0) {
      // autotune once per basis and dtype: time every variant on this run's zeroed buffers
      int& tuned = b->tuned_kind[(int)o->dtype];
      if (tuned == 0 && b->dim < kAutotuneMinDim) tuned = -1;  // default variant order
      if (tuned == 0) {
        ED_TRY_CUDA(cudaMemsetAsync(st->S, 0, sizeof(LzScalars), s));
        for (int i = 0; i < 2; ++i) ED_TRY_CUDA(cudaMemsetAsync(st->B[i], 0, st->n * st->esize, s));
        int k = 0;
        ed_status tr = hv2_autotune(b, mode, (int)st->ld, st->B[0], st->B[1], st->S, st->pa, s, &k);
        if (tr != ED_OK) return fail(tr);
        tuned = k > 0 ? k : -1;
      }
      sched = tuned > 0 ? tuned : -1;
    }
    ed_status pr = hv2_build(b, mode, (int)st->ld, sched, s, &st->plan);
    if (pr != ED_OK) return fail(pr);
  }
  // pads hold 0: lz_reset writes buffer 0 with its pads and clears buffer 1 in floating point; in
  // fixed point that stays cleared from here on (every pass writes 0 into pads or leaves them)
  if (st->fx && cudaMemsetAsync(st->B[1], 0, st->n * st->esize, s) != cudaSuccess) {
    set_error("Lanczos work vectors: clearing failed");
    return fail(ED_ERR_CUDA);
  }
  *out = st;
  return ED_OK;
}

// Steps tested per convergence check (and per CTA of it): enough that a check of 35-50 us
// hides behind as many later steps. A step takes about 10 us up to 2^18 states, 12-30 us up to
// 2^20, 25-60 us up to 2^22 (int64, rings to the 4x4 lattice).
static int check_stride(int64_t n) {
  return n < ((int64_t)1 << 18) ? 8 : n < ((int64_t)1 << 20) ? 4 : n < ((int64_t)1 << 22) ? 2 : 1;
}

// Start a run on an allocated state: load f_1 (caller vector or seeded start vector) with its pads
// and the run's scalars. The other buffer enters the first step with factor 0; it is cleared only
// in floating point, where what an earlier run left there may not be finite.
static ed_status lz_reset(ed_lanczos* st, const ed_opts* o, const void* f1) {
  const ed_basis* b = st->basis;
  cudaStream_t s = st->stream;
  ED_CHECK_ARG(f1 == nullptr || aligned16(f1), "f1 must be 16-byte aligned");
  st->opts = *o;
  st->stopped = false;
  if (!st->fx) ED_TRY_CUDA(cudaMemsetAsync(st->B[1], 0, st->n * st->esize, s));
  LzScalars h;
  memset(&h, 0, sizeof(h));
  h.max_steps = o->max_steps;
  h.tol = o->tol;
  h.chk = -check_stride(st->n);  // a graph's first check covers the steps before it: none yet
  h.scale[0] = 1.0;
  h.scale[1] = 0.0;
  for (int i = 0; i < ED_MAX_STEPS + 2; ++i) h.E0[i] = NAN;
  ED_TRY_CUDA(cudaMemcpyAsync(st->S, &h, sizeof(h), cudaMemcpyHostToDevice, s));
  // a complex vector is seen as scalars: dim (re, im) pairs = 2 dim scalars (for_rows)
  const int cx = is_complex(o->dtype) ? 2 : 1;
  const int64_t dim = cx * b->dim;
  const bool dbl = o->dtype == ED_F64_NATIVE || o->dtype == ED_C64;
  const int g = red_grid(dim);
  ED_CHECK_ARG((int64_t)g <= st->npb, "internal: partial buffer too small");
  st->cur = 0;
  // rank order (general kernels) without a plan
  const RowRuns L = row_runs(b->up.dim, b->dn.dim, st->ld, cx, hv2_rank(st->plan));
  if (st->fx) {
    long long* part = (long long*)st->pb;
    if (f1 == nullptr) {
      fx_start_kernel<<<g, kRedThreads, 0, s>>>(o->seed, L, st->fxr.vb, (long long*)st->B[0], part);
    } else {
      int E = 0;
      const ed_status r = fx_exponent(b, (const double*)f1, part, s, &E);
      if (r != ED_OK) return r;
      fx_copy_in_kernel<<<g, kRedThreads, 0, s>>>((const double*)f1, L, st->fxr.vb, E, (long long*)st->B[0], part);
    }
    const ed_status r = fx_init(st->S, part, g, s);
    if (r != ED_OK || !st->ro) return r;
    return ro_reset(st->ro, st->S, st->B[0], s);
  }
  if (f1 == nullptr) {
    start_norm_kernel<<<g, kRedThreads, 0, s>>>(o->seed, dim, st->pb);
    if (dbl)
      start_write_kernel<double><<<g, kRedThreads, 0, s>>>(o->seed, L, st->pb, g, (double*)st->B[0]);
    else
      start_write_kernel<float><<<g, kRedThreads, 0, s>>>(o->seed, L, st->pb, g, (float*)st->B[0]);
    init_scalars_kernel<<<1, 32, 0, s>>>(st->S, st->pb, g, 0);
  } else {
    if (dbl)
      copy_in_kernel<double><<<g, kRedThreads, 0, s>>>((const double*)f1, L, (double*)st->B[0], st->pb);
    else
      copy_in_kernel<float><<<g, kRedThreads, 0, s>>>((const float*)f1, L, (float*)st->B[0], st->pb);
    init_scalars_kernel<<<1, kRedThreads, 0, s>>>(st->S, st->pb, g, 1);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("Lanczos init: %s", cudaGetErrorString(e));
    return ED_ERR_CUDA;
  }
  if (st->ro) return ro_reset(st->ro, st->S, st->B[0], s);
  return ED_OK;
}

static ed_status lz_init(const ed_basis* b, const ed_opts* o, const void* f1, cudaStream_t s,
                         ed_lanczos** out) {
  ed_lanczos* st = nullptr;
  ed_status r = lz_alloc(b, o, s, &st);
  if (r != ED_OK) return r;
  if ((r = lz_reset(st, o, f1)) != ED_OK) {
    ed_lanczos_destroy(st);
    return r;
  }
  *out = st;
  return ED_OK;
}

extern "C" ed_status ed_lanczos_init(const ed_basis* b, const ed_opts* o, const void* f1,
                                     void* stream, ed_lanczos** out) {
  clear_error();
  ED_CHECK_ARG(out != nullptr, "ed_lanczos_init: out is NULL");
  *out = nullptr;
  {
    const ed_status rc = check_opts(o);
    if (rc != ED_OK) return rc;
  }
  ed_status r = lz_init(b, o, f1, (cudaStream_t)stream, out);
  if (r == ED_OK)
    r = o->dtype == ED_F64 ? fx_prepare(b)
        : is_complex(o->dtype) ? hvc_prepare(b, o->dtype)
                               : hv_prepare(b, o->dtype);
  if (r != ED_OK && *out) {
    ed_lanczos_destroy(*out);
    *out = nullptr;
  }
  return r;
}

extern "C" ed_status ed_lanczos_step(ed_lanczos* st, const ed_params* p, double* alpha_j,
                                     double* beta_j1) {
  clear_error();
  ED_CHECK_ARG(st != nullptr && p != nullptr, "ed_lanczos_step: state or params is NULL");
  ED_CHECK_ARG(!st->stopped, "ed_lanczos_step: the run has stopped (breakdown or max_steps)");
  ed_status r = lz_plan(st, p);
  if (r == ED_OK) r = lz_launch_step(st, p, st->stream);
  if (r != ED_OK) return r;
  // all scalars up to b_{m+1} in one copy: 16 KB take as long as 8 bytes, and three copies were 25 us
  // of a small basis' 65 us step
  LzScalars h;
  ED_TRY_CUDA(cudaMemcpyAsync(&h, st->S, offsetof(LzScalars, E0), cudaMemcpyDeviceToHost, st->stream));
  ED_TRY_CUDA(cudaStreamSynchronize(st->stream));
  if (alpha_j) *alpha_j = h.alpha[h.j];
  if (beta_j1) *beta_j1 = h.beta[h.j + 1];
  if (h.status != 0) st->stopped = true;
  return h.status == 1 ? ED_BREAKDOWN : ED_OK;
}

extern "C" ed_status ed_lanczos_run(ed_lanczos* st, const ed_params* p, int32_t nsteps,
                                    float* hv_ms) {
  clear_error();
  ED_CHECK_ARG(st != nullptr && p != nullptr, "ed_lanczos_run: state or params is NULL");
  ED_CHECK_ARG(nsteps >= 0 && nsteps <= ED_MAX_STEPS, "ed_lanczos_run: nsteps out of range");
  {
    const ed_status r = lz_plan(st, p);
    if (r != ED_OK) return r;
  }
  if (!hv_ms) {
    for (int i = 0; i < nsteps; ++i) {
      ed_status r = lz_launch_step(st, p, st->stream);
      if (r != ED_OK) return r;
    }
    return ED_OK;
  }
  std::vector<cudaEvent_t> ev(2 * (size_t)nsteps, nullptr);
  ed_status r = ED_OK;
  for (auto& e : ev)
    if (cudaEventCreate(&e) != cudaSuccess) {
      set_error("ed_lanczos_run: event creation failed");
      r = ED_ERR_CUDA;
      break;
    }
  for (int i = 0; r == ED_OK && i < nsteps; ++i) r = lz_launch_step(st, p, st->stream, ev[2 * i], ev[2 * i + 1]);
  float total = 0.f;
  if (r == ED_OK && cudaStreamSynchronize(st->stream) != cudaSuccess) {
    set_error("ed_lanczos_run: %s", cudaGetErrorString(cudaGetLastError()));
    r = ED_ERR_CUDA;
  }
  for (int i = 0; r == ED_OK && i < nsteps; ++i) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, ev[2 * i], ev[2 * i + 1]) != cudaSuccess) {
      set_error("ed_lanczos_run: event timing failed");
      r = ED_ERR_CUDA;
    }
    total += ms;
  }
  for (auto& e : ev)
    if (e) cudaEventDestroy(e);
  if (r == ED_OK) *hv_ms = total;
  return r;
}

extern "C" ed_status ed_lanczos_buffers(const ed_lanczos* st, const void** f_next,
                                       const void** f_cur, double* scale_next,
                                       double* scale_cur, int64_t* ld, const int32_t** colpos) {
  clear_error();
  ED_CHECK_ARG(st != nullptr, "ed_lanczos_buffers: state is NULL");
  // after step j the buffer `cur` holds f_{j+1} (scale S->scale[cur]) and the other f_j
  double sc[2] = {0.0, 0.0};
  ED_TRY_CUDA(cudaMemcpyAsync(sc, st->S->scale, sizeof(sc), cudaMemcpyDeviceToHost, st->stream));
  ED_TRY_CUDA(cudaStreamSynchronize(st->stream));
  if (f_next) *f_next = st->B[st->cur];
  if (f_cur) *f_cur = st->B[1 - st->cur];
  if (scale_next) *scale_next = sc[st->cur];
  if (scale_cur) *scale_cur = sc[1 - st->cur];
  if (ld) *ld = st->ld;
  if (colpos) *colpos = hv2_colpos(st->plan);
  return ED_OK;
}

extern "C" ed_status ed_lanczos_schedule(const ed_lanczos* st, int32_t* schedule) {
  clear_error();
  ED_CHECK_ARG(st != nullptr && schedule != nullptr, "ed_lanczos_schedule: NULL argument");
  *schedule = st->plan ? hv2_kind(st->plan) : 0;
  return ED_OK;
}

extern "C" ed_status ed_lanczos_energy(ed_lanczos* st, double* E0, int32_t* steps) {
  clear_error();
  ED_CHECK_ARG(st != nullptr, "ed_lanczos_energy: state is NULL");
  lz_energy_kernel<<<1, kRedThreads, 0, st->stream>>>(st->S, st->tmp);
  ED_TRY_CUDA(cudaGetLastError());
  double e = 0;
  int j = 0;
  ED_TRY_CUDA(cudaMemcpyAsync(&e, st->tmp, sizeof(double), cudaMemcpyDeviceToHost, st->stream));
  ED_TRY_CUDA(cudaMemcpyAsync(&j, &st->S->j, sizeof(int), cudaMemcpyDeviceToHost, st->stream));
  ED_TRY_CUDA(cudaStreamSynchronize(st->stream));
  if (E0) *E0 = e;
  if (steps) *steps = j;
  return ED_OK;
}

// ------------------------------------------------------------------ solve
// ed_lanczos_solve keeps, per basis, one allocated state per (dtype, schedule) and its
// instantiated graph of two to eight steps (lz_graph), so repeated solves skip allocation and capture; a solve that
// finds the cache busy (another thread) uses a private state instead.
struct SolveCache {
  std::mutex mu;
  cudaStream_t stream = nullptr;
  struct Entry {
    int dtype, schedule, reorth, slots;  // slots: stored vectors (reorth runs), else 0
    ed_lanczos* st;
  };
  std::vector<Entry> entries;
};
static std::mutex g_cache_mu;

namespace ed {
void lz_cache_free(const ed_basis* b) {
  SolveCache* C = (SolveCache*)b->solve_cache;
  if (!C) return;
  for (auto& e : C->entries) ed_lanczos_destroy(e.st);
  if (C->stream) cudaStreamDestroy(C->stream);
  delete C;
  b->solve_cache = nullptr;
}
}  // namespace ed

// The CUDA graph of a solve's steps (captured on first use per parameters): two steps, or
// with the convergence test max(2, K) steps, K = check_stride. The check of K steps is a
// branch beside the steps that follow: one opens the graph (the last K steps of the replay
// before, whose check would otherwise end it alone), the others follow their steps.
static int lz_graph_index(const ed_lanczos* st, bool check) {
  return (check ? 1 : 0) + (st->slots && st->store.slots == st->slots ? 2 : 0);
}

static ed_status lz_graph(ed_lanczos* st, const ed_params* p, bool check, int* steps) {
  cudaStream_t s = st->stream;
  const int K = check_stride(st->n);
  const int n = check ? std::max(2, K) : 2;
  *steps = n;
  const int gi = lz_graph_index(st, check);
  cudaGraphExec_t& exec = st->graph[gi];
  if (exec && st->graph_t[gi] == p->t && st->graph_U[gi] == p->U) return ED_OK;
  if (exec) cudaGraphExecDestroy(exec);
  exec = nullptr;
  if (!st->host) {
    int lo = 0, hi = 0;
    ED_TRY_CUDA(cudaDeviceGetStreamPriorityRange(&lo, &hi));
    if (!st->check_stream)
      ED_TRY_CUDA(cudaStreamCreateWithPriority(&st->check_stream, cudaStreamNonBlocking, hi));
    for (cudaEvent_t* e : {&st->ev_fork, &st->ev_join, &st->ev_batch[0], &st->ev_batch[1]})
      if (!*e) ED_TRY_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    ED_TRY_CUDA(cudaMallocHost((void**)&st->host, sizeof(LzScalars) + 2 * sizeof(int4)));
  }
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    set_error("ed_lanczos_solve: stream capture failed");
    return ED_ERR_CUDA;
  }
  ed_status r = ED_OK;
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < n && r == ED_OK && e == cudaSuccess; ++i) {
    if (check && i % K == 0) {
      e = cudaEventRecord(st->ev_fork, s);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(st->check_stream, st->ev_fork, 0);
      lz_check_kernel<<<K, kRedThreads, 0, st->check_stream>>>(st->S);
      if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e == cudaSuccess) r = lz_launch_step(st, p, s);
  }
  if (check) {  // the branch joins the steps again, also where the capture failed
    cudaEventRecord(st->ev_join, st->check_stream);
    cudaStreamWaitEvent(s, st->ev_join, 0);
  }
  const cudaError_t ce = cudaStreamEndCapture(s, &g);
  if (e == cudaSuccess) e = ce;
  if (r == ED_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, g, 0);
  if (g) cudaGraphDestroy(g);
  if (r != ED_OK || e != cudaSuccess) {
    exec = nullptr;
    cudaGetLastError();
    if (r != ED_OK) return r;
    set_error("ed_lanczos_solve: graph of the steps: %s", cudaGetErrorString(e));
    return ED_ERR_CUDA;
  }
  st->graph_t[gi] = p->t;
  st->graph_U[gi] = p->U;
  return ED_OK;
}

// Run a started state until it stops, and copy its scalars to st->host: m steps, status as in
// LzScalars. all_E0: E0 of every step, else of the last one (runs without convergence test).
// before(n): called before the steps up to n are enqueued.
template <typename Before>
static ed_status lz_iterate(ed_lanczos* st, const ed_params* p, const ed_opts* o, bool all_E0,
                            int* m, int* status, Before before) {
  cudaStream_t s = st->stream;
  const bool check = o->tol > 0.0;
  int n = 0;
  ed_status r = lz_graph(st, p, check, &n);
  if (r == ED_OK) r = lz_plan(st, p);
  if (r != ED_OK) return r;
  // batches of about 8 steps, the host one batch behind the device: it reads the status of a
  // batch while the next one runs (a stopped run's remaining kernels return at entry). Without a
  // convergence test only a breakdown ends a run early, and batches are of 16 steps: each copy of the
  // status holds the stream up for some 10 us, and 30 steps of the 10-site ring (63,504 states, native
  // FP64) took 745 us in four batches, 722 in two.
  int4* head = reinterpret_cast<int4*>(st->host + 1);
  const int per_batch = std::max(1, (check ? 8 : 16) / n);
  int launched = 0;
  const int gi = lz_graph_index(st, check);
  for (int batch = 0;; ++batch) {
    if ((r = before(std::min(launched + per_batch * n, o->max_steps))) != ED_OK) return r;
    for (int i = 0; i < per_batch && launched < o->max_steps; ++i, launched += n)
      ED_TRY_CUDA(cudaGraphLaunch(st->graph[gi], s));
    if (launched >= o->max_steps) break;
    ED_TRY_CUDA(cudaMemcpyAsync(&head[batch & 1], st->S, sizeof(int4), cudaMemcpyDeviceToHost, s));
    ED_TRY_CUDA(cudaEventRecord(st->ev_batch[batch & 1], s));
    if (batch == 0) continue;
    ED_TRY_CUDA(cudaEventSynchronize(st->ev_batch[(batch - 1) & 1]));
    if (head[(batch - 1) & 1].y != 0 || head[(batch - 1) & 1].z != 0) break;
  }
  if (check)
    lz_check_kernel<<<check_stride(st->n), kRedThreads, 0, s>>>(st->S);  // the last steps
  else
    lz_history_kernel<<<all_E0 ? o->max_steps : 1, kRedThreads, 0, s>>>(st->S, all_E0 ? 1 : 0);
  ED_TRY_CUDA(cudaGetLastError());
  ED_TRY_CUDA(cudaMemcpyAsync(st->host, st->S, sizeof(LzScalars), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  const LzScalars& h = *st->host;
  *m = h.conv_j ? h.conv_j : h.j;
  *status = h.conv_j ? 2 : h.status;
  return ED_OK;
}

static ed_status solve_on(ed_lanczos* st, const ed_basis* b, const ed_params* p, const ed_opts* o,
                          const void* f1, double* E0, int32_t* steps, double* alpha, double* beta,
                          double* E0_hist) {
  ed_status r = lz_reset(st, o, f1);
  if (r != ED_OK) return r;
  if ((r = (o->dtype == ED_F64 ? fx_prepare(b)
            : is_complex(o->dtype) ? hvc_prepare(b, o->dtype)
                                   : hv_prepare(b, o->dtype))) != ED_OK)
    return r;
  int j = 0, status = 0;
  if ((r = lz_iterate(st, p, o, E0_hist != nullptr, &j, &status, [](int) { return ED_OK; })) != ED_OK)
    return r;
  const LzScalars& h = *st->host;
  *E0 = j >= 1 ? h.E0[j] : NAN;
  if (steps) *steps = j;
  for (int i = 1; i <= j; ++i) {
    if (alpha) alpha[i - 1] = h.alpha[i];
    if (beta) beta[i - 1] = h.beta[i + 1];
    if (E0_hist) E0_hist[i - 1] = h.E0[i];
  }
  if (status == 1) return ED_BREAKDOWN;
  if (status == 3 && o->tol > 0.0) {
    set_error("ed_lanczos_solve: not converged after %d steps", j);
    return ED_ERR_NOT_CONVERGED;
  }
  return ED_OK;
}

// Run fn(st) on the basis's cached state for opts o (allocated on first use), or on a
// private state when another thread holds the cache; the work is ordered after the work
// already queued on the caller's stream. A state made by this call whose work vectors take more than
// keep_bytes is not kept.
template <typename Fn>
static ed_status with_state(const ed_basis* b, const ed_opts* o, cudaStream_t user, Fn fn,
                            double keep_bytes = INFINITY) {
  SolveCache* C = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    if (!b->solve_cache) {
      SolveCache* nc = new SolveCache();
      if (cudaStreamCreateWithFlags(&nc->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete nc;
        set_error("ed_lanczos_solve: stream creation failed");
        return ED_ERR_CUDA;
      }
      b->solve_cache = nc;
    }
    C = (SolveCache*)b->solve_cache;
  }
  std::unique_lock<std::mutex> lk(C->mu, std::try_to_lock);
  const bool cached = lk.owns_lock();
  cudaStream_t s = C->stream;
  if (!cached) ED_TRY_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  cudaEvent_t ev = nullptr;
  ED_TRY_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  cudaEventRecord(ev, user);
  cudaStreamWaitEvent(s, ev, 0);
  cudaEventDestroy(ev);
  ed_lanczos* st = nullptr;
  ed_status r;
  if (cached) {
    const int slots = o->reorth ? o->max_steps : 0;
    for (auto& e : C->entries)
      if (e.dtype == (int)o->dtype && e.schedule == o->schedule && e.reorth == o->reorth &&
          e.slots >= slots)
        st = e.st;
    if (!st) {
      if ((r = lz_alloc(b, o, s, &st)) != ED_OK) return r;
      if (2.0 * (double)st->n * (double)st->esize > keep_bytes) {
        r = fn(st);
        ed_lanczos_destroy(st);
        return r;
      }
      C->entries.push_back({(int)o->dtype, o->schedule, o->reorth, slots, st});
    }
    return fn(st);
  }
  if ((r = lz_alloc(b, o, s, &st)) != ED_OK) {
    cudaStreamDestroy(s);
    return r;
  }
  r = fn(st);
  ed_lanczos_destroy(st);
  cudaStreamDestroy(s);
  return r;
}

extern "C" ed_status ed_lanczos_solve(const ed_basis* b, const ed_params* p, const ed_opts* o,
                                      const void* f1, void* stream, double* E0, int32_t* steps,
                                      double* alpha, double* beta, double* E0_hist) {
  clear_error();
  ED_CHECK_ARG(b != nullptr && p != nullptr, "ed_lanczos_solve: basis or params is NULL");
  ED_CHECK_ARG(E0 != nullptr, "ed_lanczos_solve: E0 is NULL");
  ed_status r = check_opts(o);
  if (r != ED_OK) return r;
  return with_state(b, o, (cudaStream_t)stream, [&](ed_lanczos* st) {
    return solve_on(st, b, p, o, f1, E0, steps, alpha, beta, E0_hist);
  });
}

// ------------------------------------------------------------------ ground-state vector
namespace ed {
// Two memory pools per device, so that the next call does not map the same gigabytes again (0.75 ms
// per GB). psi: the vectors a ground-state call keeps and a batch's work; it holds at most kPsiKeep
// bytes while idle and gives them back when the last basis is destroyed. vstore: the FP32 vector
// stores of batched mixed solves (12 GB for 256 instances), kept in the process.
constexpr uint64_t kPsiKeep = 16ull << 30;
static std::mutex g_psi_mu;
static cudaMemPool_t g_psi_pool[64] = {}, g_vstore_pool[64] = {};
static int64_t g_psi_bases = 0;

static cudaMemPool_t lib_pool(cudaMemPool_t (&pools)[64], uint64_t keep) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(g_psi_mu);
  if (pools[dev]) return pools[dev];
  cudaMemPoolProps props = {};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
  return pools[dev] = pool;
}
cudaMemPool_t psi_pool() { return lib_pool(g_psi_pool, kPsiKeep); }
cudaMemPool_t vstore_pool() { return lib_pool(g_vstore_pool, UINT64_MAX); }

uint64_t pools_idle() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(g_psi_mu);
  uint64_t idle = 0;
  for (cudaMemPool_t p : {g_psi_pool[dev], g_vstore_pool[dev]}) {
    uint64_t reserved = 0, used = 0;
    if (p && cudaMemPoolGetAttribute(p, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
        cudaMemPoolGetAttribute(p, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess)
      idle += reserved - used;
  }
  return idle;
}

void psi_pool_basis(int delta) {
  std::lock_guard<std::mutex> lk(g_psi_mu);
  g_psi_bases += delta;
  if (g_psi_bases > 0) return;
  for (cudaMemPool_t p : g_psi_pool)
    if (p) cudaMemPoolTrimTo(p, 0);
}
}  // namespace ed

namespace {

// The Lanczos vectors of a ground-state call: blocks of up to 512 MB from the pool, taken as
// the run goes on (a run is far shorter than its step limit), at most half the free device
// memory and 96 GB in all. Returned to the pool on destruction, after the stream's work.
struct KeptVectors {
  ed_lanczos* st;
  size_t vbytes;
  int per_block, ready = 0;  // slots with memory
  double left;               // bytes still allowed
  bool complete = true;      // every slot asked for has memory
  cudaMemPool_t pool;
  std::vector<void*> blocks;

  explicit KeptVectors(ed_lanczos* state) : st(state), pool(ed::psi_pool()) {
    vbytes = (size_t)st->n * st->esize;
    per_block = (int)std::min<size_t>(std::max<size_t>((512ull << 20) / vbytes, 1), 64);
    size_t free_b = 0, total_b = 0;
    uint64_t reserved = 0, used = 0;
    if (!pool || cudaMemGetInfo(&free_b, &total_b) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
      cudaGetLastError();
      complete = false;
    }
    left = std::min(0.5 * ((double)free_b + (double)(reserved - used)), 96e9);
  }
  ~KeptVectors() {
    for (void* q : blocks) cudaFreeAsync(q, st->stream);
  }
  void* slot(int k) const { return (char*)blocks[k / per_block] + (size_t)(k % per_block) * vbytes; }
  // Slots 0 .. n - 1; from the first that does not fit on (complete false) the run keeps no more.
  ed_status grow(int n) {
    while (complete && ready < n) {
      const size_t bytes = (size_t)per_block * vbytes;
      void* q = nullptr;
      if ((double)bytes > left || cudaMallocFromPoolAsync(&q, bytes, pool, st->stream) != cudaSuccess) {
        cudaGetLastError();
        complete = false;
        break;
      }
      left -= (double)bytes;
      blocks.push_back(q);
      std::vector<void*> slot(std::min(per_block, ED_MAX_STEPS + 2 - ready));
      for (size_t k = 0; k < slot.size(); ++k) slot[k] = (char*)q + k * vbytes;
      ED_TRY_CUDA(cudaMemcpyAsync(st->slots + ready, slot.data(), slot.size() * sizeof(void*),
                                  cudaMemcpyHostToDevice, st->stream));
      ready += (int)slot.size();
    }
    return ED_OK;
  }
};

}  // namespace

// A ground-state call keeps its work vectors on the basis up to this size: larger ones leave the device
// as free as the call found it, and making them again is 1% of the call (2 GB: 3 of 330 ms).
constexpr double kGroundKeep = 1e9;

// The run of st, whose scalars are in st->host, from f_k on again: buffers and scalars from the kept
// vectors of f_{k-1} and f_k (k >= 2), the tridiagonal up to a_{k-1}, b_k from the first time.
static ed_status lz_resume(ed_lanczos* st, int k, size_t vbytes, void* const* slot) {
  cudaStream_t s = st->stream;
  LzScalars& h = *st->host;  // (pinned, and the stream has passed its last copy)
  h.j = k - 1;
  h.status = h.conv_j = h.row_next = 0;
  h.tick_chk = h.tick_hv = h.tick_upd = 0;
  memset(h.fx_dot, 0, sizeof(h.fx_dot));
  h.tscale = 0.0;
  for (int i = 1; i < k; ++i) h.tscale = std::max(h.tscale, std::fabs(h.alpha[i]) + h.beta[i]);
  ED_TRY_CUDA(cudaMemcpyAsync(st->S, &h, sizeof(h), cudaMemcpyHostToDevice, s));
  st->cur = 0;
  for (int i = 0; i < 2; ++i) {  // buffer 0: f_k, buffer 1: f_{k-1}
    ED_TRY_CUDA(cudaMemcpyAsync(st->B[i], slot[i], vbytes, cudaMemcpyDeviceToDevice, s));
    ED_TRY_CUDA(cudaMemcpyAsync(&st->S->scale[i], st->vscale + k - 1 - i, sizeof(double), cudaMemcpyDeviceToDevice, s));
    ED_TRY_CUDA(cudaMemcpyAsync(&st->S->fx_max[i], st->vmax + k - 1 - i, sizeof(long long), cudaMemcpyDeviceToDevice, s));
  }
  return ED_OK;
}

// psi on a started state: Algorithm 1 with its vectors kept where memory allows; one pass over
// them sums psi (the run itself is most of the time). Where memory ends before the run, the steps
// behind the last kept vector are made again from it, adding y_j f_j step by step, all of them when
// nothing fits. All sums are the same integers. Half-filled 16-site ring (1.3 GB a vector, 72 of
// them in the 96 GB): 622 ms; with all steps made again 909 ms, with nothing kept 839 ms.
static ed_status ground_on(ed_lanczos* st, const ed_basis* b, const ed_params* p, const ed_opts* o,
                           const void* f1, long long* P, double* E0, int32_t* steps) {
  cudaStream_t s = st->stream;
  if (!st->ywork) {
    if (cudaMalloc((void**)&st->slots, (ED_MAX_STEPS + 2) * sizeof(void*)) != cudaSuccess ||
        cudaMalloc((void**)&st->vscale, (ED_MAX_STEPS + 2) * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&st->vmax, (ED_MAX_STEPS + 2) * sizeof(long long)) != cudaSuccess ||
        cudaMalloc((void**)&st->ywork, 3 * (ED_MAX_STEPS + 4) * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      for (void* q : {(void*)st->slots, (void*)st->vscale, (void*)st->vmax})
        if (q) cudaFree(q);
      st->slots = nullptr, st->vscale = nullptr, st->vmax = nullptr;
      set_error("ed_lanczos_ground_state: out of device memory");
      return ED_ERR_OOM;
    }
  }
  const int32_t* rank = nullptr;
  ed_status r = lz_rank(st, &rank);
  if (r == ED_OK) r = lz_reset(st, o, f1);
  if (r != ED_OK) return r;
  if ((r = fx_prepare(b)) != ED_OK) return r;
  int m = 0, status = 0;
  double lam = NAN;
  double* y = st->ywork;
  int have = 0;  // psi holds the terms of f_1 .. f_have
  {
    struct Unset {  // later solves on the state keep no vectors
      ed_lanczos* st;
      ~Unset() { st->store = LzStore{nullptr, nullptr, nullptr}; }
    } unset{st};
    KeptVectors kept(st);
    const bool own = !st->ro;  // a reorthogonalising run keeps its vectors by itself
    if (own) {
      ED_TRY_CUDA(cudaMemsetAsync(st->slots, 0, (ED_MAX_STEPS + 2) * sizeof(void*), s));
      if ((r = kept.grow(1)) != ED_OK) return r;
      if (kept.complete) {
        ED_TRY_CUDA(cudaMemcpyAsync(kept.blocks[0], st->B[0], kept.vbytes, cudaMemcpyDeviceToDevice, s));
        ED_TRY_CUDA(cudaMemcpyAsync(st->vscale, &st->S->scale[0], sizeof(double), cudaMemcpyDeviceToDevice, s));
        ED_TRY_CUDA(cudaMemcpyAsync(st->vmax, &st->S->fx_max[0], sizeof(long long), cudaMemcpyDeviceToDevice, s));
        st->store = LzStore{st->slots, st->vscale, st->vmax};
      }
    }
    r = lz_iterate(st, p, o, false, &m, &status,
                   [&](int n) { return own ? kept.grow(n + 1) : ED_OK; });
    if (r != ED_OK) return r;
    if (m < 1) {
      set_error("ed_lanczos_ground_state: the run took no step");
      return ED_ERR_ARG;
    }
    lz_ritz_kernel<<<1, 32, 5 * (size_t)(m + 2) * sizeof(double), s>>>(st->S, m, st->host->E0[m], y);
    ED_TRY_CUDA(cudaGetLastError());
    lam = st->host->E0[m];
    have = own ? std::min(kept.ready, m) : m;
    if (have < std::min(m, 2)) have = 0;  // (a run goes on from two vectors)
    if (have > 0 &&
        (r = fx_psi_sum(b, y, have, own ? st->store : ro_slots(st->ro), st->ld, rank, P, (long long*)st->pb, s)) != ED_OK)
      return r;
    if (have > 0 && have < m) {
      void* const last[2] = {kept.slot(have - 1), kept.slot(have - 2)};
      if ((r = lz_resume(st, have, kept.vbytes, last)) != ED_OK) return r;
    }
  }
  const bool summed = have == m;
  if (!summed) {
    auto add = [&](int j) {  // the term of f_j, the running vector
      return fx_psi_accum(b, st->S, st->cur, y, j, (const long long*)st->B[st->cur], st->ld, hv2_colpos(st->plan), P, s);
    };
    if (have == 0) {
      if ((r = lz_reset(st, o, f1)) != ED_OK) return r;
      ED_TRY_CUDA(cudaMemsetAsync(P, 0, (size_t)b->dim * sizeof(long long), s));
      if ((r = add(++have)) != ED_OK) return r;
    }
    if ((r = lz_plan(st, p)) != ED_OK) return r;
    while (have < m) {
      if ((r = lz_launch_step(st, p, s)) != ED_OK) return r;
      if ((r = add(++have)) != ED_OK) return r;
    }
  }
  if ((r = fx_psi_finish(b, P, summed, (long long*)st->pb, s)) != ED_OK) return r;
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  *E0 = lam;
  if (steps) *steps = m;
  if (status == 3 && o->tol > 0.0) {
    set_error("ed_lanczos_ground_state: not converged after %d steps", m);
    return ED_ERR_NOT_CONVERGED;
  }
  return ED_OK;
}

extern "C" ed_status ed_lanczos_ground_state(const ed_basis* b, const ed_params* p,
                                             const ed_opts* o, const void* f1, void* stream,
                                             double* psi, double* E0, int32_t* steps) {
  clear_error();
  ED_CHECK_ARG(b && p && o && psi && E0, "ed_lanczos_ground_state: NULL argument");
  ED_CHECK_ARG(o->dtype == ED_F64, "ed_lanczos_ground_state: dtype must be ED_F64");
  {
    const ed_status rc = check_opts(o);
    if (rc != ED_OK) return rc;
  }
  ED_CHECK_ARG(aligned16(psi), "ed_lanczos_ground_state: psi must be 16-byte aligned");
  return with_state(b, o, (cudaStream_t)stream, [&](ed_lanczos* st) {
    return ground_on(st, b, p, o, f1, (long long*)psi, E0, steps);
  }, kGroundKeep);
}

extern "C" ed_status ed_lanczos_solve_mixed(const ed_basis* b, const ed_params* p,
                                            const ed_opts* o, const void* f1,
                                            int32_t refine_steps, double refine_tol, void* stream,
                                            double* E0, int32_t* steps32, double* E0_fp32,
                                            int32_t* steps64, double* residual) {
  clear_error();
  ED_CHECK_ARG(b != nullptr && p != nullptr && o != nullptr && E0 != nullptr,
               "ed_lanczos_solve_mixed: NULL argument");
  ed_status r = check_opts(o);
  if (r != ED_OK) return r;
  ED_CHECK_ARG(o->dtype == ED_F32, "ed_lanczos_solve_mixed: opts->dtype must be ED_F32");
  ED_CHECK_ARG(o->reorth == 0, "ed_lanczos_solve_mixed: opts->reorth must be 0");
  ED_CHECK_ARG(refine_steps >= 1 && refine_steps <= ED_MAX_STEPS,
               "ed_lanczos_solve_mixed: refine_steps = %d outside [1, %d]", refine_steps,
               ED_MAX_STEPS);
  ED_CHECK_ARG(std::isfinite(refine_tol), "ed_lanczos_solve_mixed: refine_tol is not finite");
  ED_CHECK_ARG(!b->has_tau(), "ed_lanczos_solve_mixed: real lattices only");
  cudaStream_t user = (cudaStream_t)stream;
  // ---- FP32 phase: Algorithm 1 with the vectors kept, then the Ritz vector in rank order
  ed_opts o32 = *o;
  o32.reorth = 3;
  {
    // the FP32 phase keeps at most as many vectors as fit in half the free device memory (and
    // of what the library's pools hold idle)
    // and in 96 GB; a shorter FP32 phase leaves more of the convergence to the refinement
    // steps
    size_t free_b = 0, total_b = 0;
    ED_TRY_CUDA(cudaMemGetInfo(&free_b, &total_b));
    const double vbytes = (double)b->up.dim * (double)((b->dn.dim + 31) / 32 * 32) * 4.0;
    const double budget = std::min(((double)free_b + (double)pools_idle()) / 2.0, 96e9);
    const int cap = (int)std::min(budget / vbytes - 1.0, (double)ED_MAX_STEPS);
    ED_CHECK_ARG(cap >= 2, "ed_lanczos_solve_mixed: device memory for FP32 vectors too small");
    if (o32.max_steps > cap) o32.max_steps = cap;
    // beyond dim steps the FP32 recurrence only adds rounding noise
    if ((int64_t)o32.max_steps > b->dim) o32.max_steps = (int)std::max<int64_t>(b->dim, 1);
  }
  double* psi = nullptr;
  double* y = nullptr;
  int m = 0;
  double e32 = NAN;
  r = with_state(b, &o32, user, [&](ed_lanczos* st) -> ed_status {
    cudaStream_t s = st->stream;
    ed_status rr = solve_on(st, b, p, &o32, f1, &e32, &m, nullptr, nullptr, nullptr);
    if (rr < 0 && rr != ED_ERR_NOT_CONVERGED) return rr;
    if (m < 1) {
      set_error("ed_lanczos_solve_mixed: the FP32 phase took no step");
      return ED_ERR_ARG;
    }
    if (cudaMallocAsync((void**)&y, (size_t)3 * (m + 2) * sizeof(double), s) != cudaSuccess ||
        cudaMallocAsync((void**)&psi, (size_t)b->dim * sizeof(double), s) != cudaSuccess) {
      set_error("ed_lanczos_solve_mixed: out of device memory");
      return ED_ERR_OOM;
    }
    lz_ritz_kernel<<<1, 32, 5 * (size_t)(m + 2) * sizeof(double), s>>>(st->S, m, e32, y);
    ED_TRY_CUDA(cudaGetLastError());
    rr = ro_ritz_vector(st->ro, y, m, b->dim, b->dn.dim, st->ld, hv2_colpos(st->plan), psi, s);
    if (rr != ED_OK) return rr;
    ED_TRY_CUDA(cudaStreamSynchronize(s));
    return ED_OK;
  });
  auto release = [&](ed_status e) {
    if (y) cudaFreeAsync(y, user);
    if (psi) cudaFreeAsync(psi, user);
    return e;
  };
  if (r != ED_OK) return release(r);
  if (steps32) *steps32 = m;
  if (E0_fp32) *E0_fp32 = e32;
  // ---- FP64-accurate phase from psi: a_1 = psi.H psi (the Rayleigh quotient), b_2 = the
  // residual norm, E0 = lambda_min of the refined T
  ed_opts o64 = *o;
  o64.dtype = ED_F64;
  o64.max_steps = refine_steps;
  o64.tol = refine_tol;
  o64.schedule = -1;
  std::vector<double> a(refine_steps), bt(refine_steps);
  int32_t k = 0;
  r = with_state(b, &o64, user, [&](ed_lanczos* st) {
    return solve_on(st, b, p, &o64, psi, E0, &k, a.data(), bt.data(), nullptr);
  });
  if (r == ED_BREAKDOWN) r = ED_OK;
  if (steps64) *steps64 = k;
  if ((r == ED_OK || r == ED_ERR_NOT_CONVERGED) && residual) *residual = bt[0];
  return release(r);
}
