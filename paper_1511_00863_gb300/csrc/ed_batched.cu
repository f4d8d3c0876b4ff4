// Batched Lanczos (Sec. 2.2, Algorithm 1) over many independent (lattice, filling, U)
// instances in ONE persistent cooperative kernel launch.
//
// Instances are packed onto groups of co-resident CTAs by a schedule (kScheds): an instance
// whose dimension reaches a threshold gets a group of several CTAs, smaller instances run
// one after another inside single-CTA groups (only __syncthreads needed there). Groups
// with several CTAs synchronise through a global-memory barrier whose spin is bounded:
// when it runs out the kernel records ED_ERR_TIMEOUT for the batch and returns.
// Per instance and step (FP32 or FP64 vectors, FP64 scalars, as the single-instance ED_F32 /
// ED_F64_NATIVE paths):
//   phase 1: w = s_c H B_c - b_j s_p B_p (written over B_p), partial sums of w . f_j
//   phase 2: a_j, q = w - a_j f_j, partial sums of q . q
//   phase 3: b_{j+1}, scale of f_{j+1}, every `check` steps E0(j) = lambda_min(T_j) by
//            Sturm bisection (leader CTA), convergence / breakdown / max_steps.
// The H.v phase stages blocks of up rows in shared memory (down-hop gathers there) and reads
// up-neighbour rows coalesced; vectors of the batch stay in L2. Instances with tables of the
// row-ordered H.v (ed_rows.cu) take 32 columns of equal hop counts per warp, one table entry for
// two rows, and read neighbour rows in 16-byte loads; the others go element by element.
// ed_lanczos_solve_batched_mixed carries the FP32 batch to FP64 accuracy: the FP32 run keeps
// its vectors, a Ritz vector is assembled per instance and FP64 steps refine it
// (batched_ritz_kernel and the `refine` form of the FP64 kernel, below).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <map>
#include <mutex>
#include <queue>
#include <string>
#include <vector>

#include "ed_internal.cuh"
#include "ed_lanczos_dev.cuh"

namespace ed {

constexpr int kBThreads = 256;
// CTAs per SM the register bound allows: the batch is bound by latency across many small
// instances, and 6 CTAs per SM (40 registers, a few words spilled) ran the FP32 batch in 56
// ms against 72 ms with 4 (64 registers). The FP64 kernel keeps 4 (its 64-bit arithmetic
// spills more at 40 registers: 204 ms against 191 ms).
constexpr int kBCtasPerSm = 6;
template <typename T>
constexpr int bctas_per_sm() { return sizeof(T) == 4 ? kBCtasPerSm : 4; }
// Staging area of the H.v phase (a block of up rows, at most kBRowFloats * 4 bytes); the same
// shared buffer holds the leader CTA's bisection workspace at another time.
constexpr int kBRowFloats = 4096;
constexpr int kBLists = 128;  // up-hop list entries in it (row-ordered H.v)
// Dynamic shared memory of the batched kernels: the row-block staging area, or the bisection
// workspace of T_m for m <= max_steps, whichever is larger (sized per run, so short runs keep
// the L1 data cache that the hop tables are read through).
static size_t bsmem_bytes(int max_steps) {
  const size_t sturm = (size_t)sturm_work_doubles(max_steps + 2) * sizeof(double);
  return sturm > (size_t)kBRowFloats * 4 ? sturm : (size_t)kBRowFloats * 4;
}

// ... of batched_ritz_kernel: a, b, y and the two arrays of the inverse iteration.
static size_t ritz_bytes(int max_steps) { return 5 * (size_t)(max_steps + 2) * sizeof(double); }

struct BInst {
  const uint32_t* upb;
  const uint32_t* dnb;
  const int32_t* hu;
  const int32_t* hd;
  int dim_up, dim_dn, mhu, mhd;
  int ld;  // row stride of the vectors: dim_dn, or rounded up to 4 where the tables below serve
  // tables of the row-ordered H.v (ed_rows.cu: columns by hop count, one class), or tab NULL
  const int32_t* perm;
  const int32_t* base;
  const uint8_t* kc;
  const uint16_t* tab;
  void* B0;  // two work vectors of the instance (FP32 or FP64 elements)
  void* B1;
  double t, U;
  // mixed solves only: the FP32 phase's Lanczos vectors (raw, [max_steps][dpad]) and the
  // FP64 refinement's two work vectors
  float* V;
  double* D0;
  double* D1;
  int dpad;
};

// Per-instance results and Lanczos scalars (1-based a_j, b_j like LzScalars).
struct BState {
  int j, status;
  double scale[2];
  double last_E0, last_lo;  // bracket of E0(last_E0_step), the last tested step's
  int last_E0_step;
  int pad_;
};

struct BGroup {
  int first_cta, ncta;
  int inst_begin, inst_end;  // range in the instance order list
};

struct BArgs {
  const BInst* inst;
  BState* st;
  double* alpha;  // [n_inst][max_steps + 2]
  double* beta;   // [n_inst][max_steps + 2]
  double* E0;     // [n_inst][max_steps + 2]
  const int* order;
  const BGroup* groups;
  const int* group_of_cta;
  double* part_a;  // [grid]
  double* part_b;  // [grid]
  unsigned* bar_count;  // [n_groups]
  unsigned* bar_gen;    // [n_groups]
  int* error;
  int max_steps, check;
  double tol;
  uint64_t seed;
  long long max_spin;
  // mixed solves only (batched_ritz_kernel and the refinement): per instance the FP32
  // vectors' scales, y and the inverse iteration's workspace ([n_inst][4 (max_steps + 2)]:
  // vscale | y | 2 (max_steps + 2) of work), the refinement's state and scalars
  BState* st2;
  double* rwork;
  double* alpha2;  // [n_inst][refine_steps + 2]
  double* beta2;
  double* E02;
  int refine_steps;
  double refine_tol;
  int refine;  // batched_lanczos_kernel<double>: run the refinement of a mixed solve
  int store;   // batched_lanczos_kernel<float>: keep the Lanczos vectors (mixed solves)
};

// acc += the signed values of a state's hop targets, hop by hop in table order (so the
// rounding is that of a one-at-a-time loop), taking the table entries and gathered values
// of Q hops before adding any: more loads in flight. tab[k * stride] is hop k's entry; a
// target >= n is padding, and the rest of the state's list is padding too. FP32 takes 4 at
// a time (the 256-instance batch: 51.8 -> 44.3 ms); FP64 one (4 at a time spilled more and
// took 212 against 191 ms).
template <typename T, typename Load>
__device__ __forceinline__ void add_hops(T& acc, const int32_t* tab, int64_t stride, int mh, uint32_t n,
                                         Load load) {
  constexpr int Q = sizeof(T) == 4 ? 4 : 1;
  int k = 0;
  for (; Q > 1 && k + Q <= mh; k += Q) {
    uint32_t en[Q];
    T v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) en[q] = (uint32_t)tab[(int64_t)(k + q) * stride];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const uint32_t tg = en[q] & kTargetMask;
      v[q] = tg < n ? load(tg) : T(0);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if ((en[q] & kTargetMask) < n) acc += (en[q] & kSignBit) ? -v[q] : v[q];
    if ((en[Q - 1] & kTargetMask) >= n) return;
  }
  for (; k < mh; ++k) {
    const uint32_t en = (uint32_t)tab[(int64_t)k * stride];
    const uint32_t tg = en & kTargetMask;
    if (tg >= n) return;
    const T v = load(tg);
    acc += (en & kSignBit) ? -v : v;
  }
}

// One instance's run of Algorithm 1, for the CTAs of its group.
struct RunSpec {
  BState* S;
  double* al;
  double* be;
  double* e0;
  void* B0;
  void* B1;
  const double* f1;   // FP64 start vector (unnormalised) or NULL for the seeded one
  float* V;           // store the raw FP32 vector of every step here ([max_steps][dpad]), or NULL
  double* vscale;     // with V: the scale of the stored vector of step j at vscale[j]
  int dpad;
  int max_steps, check;
  double tol;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier of the `g` CTAs of one group. The wait is bounded by `max_spin` nanoseconds of
// the global timer; on expiry (or when another group already failed) it sets *error and
// returns false, and the caller returns from the kernel.
__device__ bool group_barrier(unsigned* count, unsigned* gen, int g, long long max_spin, int* error) {
  __shared__ int ok_s;
  __syncthreads();
  if (g > 1) {
    if (threadIdx.x == 0) {
      int ok = 1;
      const unsigned my_gen = atomicAdd(gen, 0u);
      __threadfence();
      const unsigned arrived = atomicAdd(count, 1u);
      if (arrived == (unsigned)g - 1u) {
        atomicExch(count, 0u);
        __threadfence();
        atomicAdd(gen, 1u);
      } else {
        const unsigned long long t0 = global_ns();
        const long long max_iter = (max_spin >> 6) + 1000000;  // backstop if the timer stalls
        long long it = 0;
        while (atomicAdd(gen, 0u) == my_gen) {
          if ((long long)(global_ns() - t0) > max_spin || ++it > max_iter ||
              *(volatile int*)error != 0) {
            ok = 0;
            atomicExch(error, 1);
            break;
          }
          __nanosleep(128);
        }
      }
      __threadfence();
      ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
  }
  return true;
}

// Loads of data that other CTAs of the group wrote during this launch go to L2 (the L1 of
// this SM is not coherent with their stores).
template <typename T>
__device__ __forceinline__ T ld_shared_f(const T* p, bool multi) { return multi ? __ldcg(p) : *p; }

// ---- H.v of a block of up rows through the row-ordered tables
template <typename T> struct BWide;
template <> struct BWide<float> { typedef float4 V; static constexpr int kRows = 2; };
template <> struct BWide<double> { typedef double2 V; static constexpr int kRows = 1; };
template <typename T, int N>
struct alignas(sizeof(T) * N) BPack {
  T v[N];
};
template <typename T>
__device__ __forceinline__ T b_sign(T x, uint32_t s) {  // s: 0 or the sign bit in bit 31
  if constexpr (sizeof(T) == 4) return __uint_as_float(__float_as_uint(x) ^ s);
  else return __hiloint2double(__double2hiint(x) ^ (int)s, __double2loint(x));
}
// 16-byte load; from L2 when other CTAs of the group wrote the data
template <typename V>
__device__ __forceinline__ V b_ld16(const V* p, bool multi) { return multi ? __ldcg(p) : *p; }

// Row packs (kRows rows each) per block of a CTA: what the staging area holds, but no more than
// leaves every CTA of the group four blocks.
template <typename T>
__device__ __forceinline__ int b_packs(const BInst& I, int g) {
  constexpr int R = BWide<T>::kRows;
  const int fit = (kBRowFloats * 4 - 4 * kBLists) / ((2 * I.ld + 1) * R * (int)sizeof(T));
  const int share = I.dim_up / (4 * R * g);
  return max(1, min(min(fit, share), min(kBLists / max(1, R * I.mhu), 2048 / (R * I.ld))));
}

template <typename T>
__device__ __forceinline__ void hv_block(const BInst& I, const T* xc, T* xp, float* vj, int u0, int packs,
                                         bool multi, T sc, T bsp, DotAcc<T>& dot, unsigned char* bsm) {
  constexpr int R = BWide<T>::kRows, W = 16 / (int)sizeof(T);
  typedef typename BWide<T>::V V;
  const int dn = I.dim_dn, ld = I.ld, MH = I.mhu;
  BPack<T, R>* xs = reinterpret_cast<BPack<T, R>*>(bsm);               // [packs][ld + 1]
  T* ys = reinterpret_cast<T*>(xs + packs * (ld + 1));                 // [packs * R][ld]
  uint32_t* ue = reinterpret_cast<uint32_t*>(ys + (packs * R) * ld);   // [packs * R][MH]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T tt = (T)I.t, UU = (T)I.U;
  __syncthreads();
  for (int b = 0; b < packs; ++b)
    for (int d = threadIdx.x; d <= ld; d += blockDim.x) {
      BPack<T, R> p;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int u = u0 + b * R + r;
        p.v[r] = d < ld && u < I.dim_up ? ld_shared_f(xc + (int64_t)u * ld + d, multi) : T(0);
      }
      xs[b * (ld + 1) + d] = p;
    }
  for (int i = threadIdx.x; i < packs * R * MH; i += blockDim.x) {
    const int r = i / MH, k = i - r * MH;
    ue[i] = u0 + r < I.dim_up ? (uint32_t)I.hu[(int64_t)k * I.dim_up + u0 + r] : (uint32_t)I.dim_up;
  }
  __syncthreads();
  // ---- down part: 32 columns of (nearly) equal hop counts per warp and pack
  const int nch = (dn + 31) >> 5;
  for (int task = warp; task < nch * packs; task += kBThreads / 32) {
    const int b = task / nch, ch = task - b * nch;
    const int p = I.perm[32 * ch + lane], n = I.kc[ch];
    const uint16_t* tp = I.tab + I.base[ch] + lane;
    const BPack<T, R>* xb = xs + b * (ld + 1);
    T acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = T(0);
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      const uint32_t e = tp[32 * k];  // target (dim_dn: a zero column) | sign << 15
      const BPack<T, R> q = xb[e & 0x7FFFu];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] += b_sign(q.v[r], (e & 0x8000u) << 16);
    }
    if (p >= 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) ys[(b * R + r) * ld + p] = acc[r];
    }
  }
  __syncthreads();
  // ---- up part, diagonal and the Lanczos update: 16 bytes of a row per thread (pads hold 0)
  const int per_row = ld / W;
  for (int q = threadIdx.x; q < packs * R * per_row; q += blockDim.x) {
    const int r = q / per_row, d0 = (q - r * per_row) * W, u = u0 + r;
    if (u >= I.dim_up) break;
    const uint32_t* ul = ue + r * MH;
    T acc[W];
#pragma unroll
    for (int v = 0; v < W; ++v) acc[v] = d0 + v < dn ? ys[r * ld + d0 + v] : T(0);
    const T* xd = xc + d0;
#pragma unroll 2
    for (int k = 0; k < MH; ++k) {
      const uint32_t e = ul[k];
      const int tg = (int)(e & kTargetMask);
      if (tg >= I.dim_up) break;
      const V x4 = b_ld16(reinterpret_cast<const V*>(xd + (int64_t)tg * ld), multi);
      const T* xv = reinterpret_cast<const T*>(&x4);
#pragma unroll
      for (int v = 0; v < W; ++v) acc[v] += b_sign(xv[v], e & kSignBit);
    }
    const int64_t e0 = (int64_t)u * ld + d0;
    const V P4 = b_ld16(reinterpret_cast<const V*>(xp + e0), multi);
    const T* P = reinterpret_cast<const T*>(&P4);
    const uint32_t ub = I.upb[u];
    V w4, x4;
    T* w = reinterpret_cast<T*>(&w4);
    T* xo = reinterpret_cast<T*>(&x4);
#pragma unroll
    for (int v = 0; v < W; ++v) {
      const T xv = xs[(r / R) * (ld + 1) + d0 + v].v[r % R];
      const uint32_t db = d0 + v < dn ? I.dnb[d0 + v] : 0u;
      const T hx = fma(-tt, acc[v], UU * (T)__popc(ub & db) * xv);
      w[v] = fma(sc, hx, -bsp * P[v]);
      xo[v] = xv;
      dot.add(w[v], sc * xv);
    }
    *reinterpret_cast<V*>(xp + e0) = w4;
    if constexpr (sizeof(T) == 4) {
      if (vj) __stcs(reinterpret_cast<V*>(vj + e0), x4);
    }
  }
}

__device__ __forceinline__ double bstart_element(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  return 2.0 * ((double)(z >> 11) * 0x1.0p-53) - 1.0;
}

// Group-wide sum of the group's CTA partials (fixed order), every thread gets it.
__device__ __forceinline__ double group_sum(const double* part, int first, int g, double* red) {
  double v = 0.0;
  for (int i = threadIdx.x; i < g; i += blockDim.x) v += __ldcg(part + first + i);
  v = block_sum(v, red);
  if (threadIdx.x == 0) red[32] = v;
  __syncthreads();
  v = red[32];
  __syncthreads();
  return v;
}

// sturm_lowest out of line: inlined three times it cost the kernel's loops 700 bytes of spills.
__device__ __noinline__ double group_sturm(const double* al, const double* be, int m, double hint, double* work,
                                           int cap, double* rough_lo) {
  return sturm_lowest(al, be, m, hint, work, cap, rough_lo);
}

// The stop test of step j (whole leader CTA; st: 1 after a breakdown): the new status. It compares
// E0(j) with the last tested step's, but away from convergence a rough bracket of each decides it
// for a quarter of the time (two float-float rounds instead of those and the FP64 ones): while the
// brackets lie further apart than tol, the test fails whatever the exact values are. Otherwise, and
// at the last step, both are computed exactly.
__device__ __noinline__ int group_stop_test(BState* S, const RunSpec& R, const double* al, const double* be, double* e0, int j,
                               int st, double* work) {
  const int cap = R.max_steps + 2;
  const bool last = st != 0 || j >= R.max_steps;
  const int prev = S->last_E0_step;
  const double plo = S->last_lo, phi = S->last_E0;  // [plo, phi] holds E0(prev); plo == phi: exact
  __syncthreads();
  double E, lo;
  if (prev > 0 && !last) {
    E = group_sturm(al, be, j, phi, work, cap, &lo);
    const double mag = fmax(fmax(fabs(lo), fabs(E)), 1.0);
    if (plo - E > 1.001 * R.tol * mag) {
      __syncthreads();
      if (threadIdx.x == 0) {
        S->last_lo = lo;
        S->last_E0 = E;
        S->last_E0_step = j;
      }
      return 0;
    }
    __syncthreads();
  }
  double P = phi;
  if (prev > 0 && st == 0 && R.tol > 0.0 && plo != phi) {
    P = group_sturm(al, be, prev, phi, work, cap, nullptr);
    __syncthreads();
  }
  E = group_sturm(al, be, j, prev > 0 ? P : NAN, work, cap, nullptr);
  __syncthreads();
  if (threadIdx.x == 0) {
    e0[j] = E;
    S->last_lo = E;
    S->last_E0 = E;
    S->last_E0_step = j;
  }
  if (st == 0 && R.tol > 0.0 && prev > 0 && fabs(E - P) <= R.tol * fmax(fabs(E), 1.0)) return 2;
  return st == 0 && j >= R.max_steps ? 3 : st;
}

// T = float (ED_F32) or double (ED_F64_NATIVE): vector elements and H.v arithmetic; the
// scalars are FP64 either way.
// Algorithm 1 for instance I on its group (CTA c of g, leader = c == 0), FP32 or FP64
// vectors T, as specified by R. Returns false when a group barrier's bounded wait ran out.
template <typename T>
__device__ bool run_instance(const BArgs& a, const BInst& I, const RunSpec& R, int c, int g,
                             int first_cta, unsigned* bc, unsigned* bg, double* red, int* stop_s,
                             unsigned char* bsm) {
  constexpr int kRowElems = kBRowFloats * 4 / (int)sizeof(T);  // staged elements of a row block
  T* xsm = reinterpret_cast<T*>(bsm);
  const bool leader = c == 0;
  const bool multi = g > 1;
  BState* S = R.S;
  double* al = R.al;
  double* be = R.be;
  double* e0 = R.e0;
  const int dim = I.dim_up * I.ld;  // elements of a vector, pads included
  const int64_t gt = (int64_t)g * blockDim.x;
  const int64_t t0 = (int64_t)c * blockDim.x + threadIdx.x;
  // element e of the seeded start vector (0 in a pad)
  auto start = [&](int64_t e) {
    if (I.ld == I.dim_dn) return bstart_element(a.seed, (uint64_t)e);
    const int r = (int)e / I.ld, d = (int)e - r * I.ld;
    return d < I.dim_dn ? bstart_element(a.seed, (uint64_t)((int64_t)r * I.dim_dn + d)) : 0.0;
  };
  // the scalars of the running step, one copy per CTA (all CTAs compute the same)
  __shared__ struct {
    double scale, scale_prev, beta, tscale;  // of f_j and f_{j-1}; b_j
  } run_s;
  if (threadIdx.x == 0) {
    run_s.scale = 1.0;
    run_s.scale_prev = run_s.beta = run_s.tscale = 0.0;
  }
  __syncthreads();
  // ---- start vector: raw values (SplitMix64 or the given FP64 vector), FP64 norm,
  // normalised then rounded
  {
    double v = 0.0;
    for (int64_t e = t0; e < dim; e += gt) {
      const double x = R.f1 ? ld_shared_f(R.f1 + e, multi) : start(e);
      v = fma(x, x, v);
    }
    v = block_sum(v, red);
    if (threadIdx.x == 0) a.part_a[blockIdx.x] = v;
    if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return false;
    const double inv = 1.0 / sqrt(group_sum(a.part_a, first_cta, g, red));
    for (int64_t e = t0; e < dim; e += gt) {
      const double x = R.f1 ? ld_shared_f(R.f1 + e, multi) : start(e);
      ((T*)R.B0)[e] = (T)(x * inv);
      ((T*)R.B1)[e] = T(0);
    }
    if (leader && threadIdx.x == 0) {
      S->j = 0;
      S->status = 0;
      S->scale[0] = 1.0;
      S->scale[1] = 0.0;
      S->last_E0_step = 0;
      S->last_E0 = S->last_lo = 0.0;
      be[1] = 0.0;
    }
    if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return false;
  }
  int cur = 0;
  for (int j = 1; j <= R.max_steps; ++j) {
    T* xc = (T*)(cur ? R.B1 : R.B0);
    T* xp = (T*)(cur ? R.B0 : R.B1);
    float* vj = R.V ? R.V + (size_t)(j - 1) * R.dpad : nullptr;
    if (vj && leader && threadIdx.x == 0) R.vscale[j] = run_s.scale;
    // ---- phase 1: fused H.v
    const T sc = (T)run_s.scale;
    const T bsp = (T)(run_s.beta * run_s.scale_prev);
    const T tt = (T)I.t, UU = (T)I.U;
    DotAcc<T> dot;
    if (I.tab) {
      const int packs = b_packs<T>(I, g), rows = packs * BWide<T>::kRows;
      for (int u0 = c * rows; u0 < I.dim_up; u0 += g * rows)
        hv_block<T>(I, xc, xp, vj, u0, packs, multi, sc, bsp, dot, bsm);
    } else if (I.dim_dn <= kRowElems) {
      // blocks of BR consecutive up rows staged in shared memory (coalesced loads; from L2
      // when other CTAs of the group wrote them): down-hop gathers read shared memory,
      // up-hop gathers read whole neighbour rows coalesced
      const int BR = max(1, min(kRowElems, 2048) / I.dim_dn);
      const int nblk = (I.dim_up + BR - 1) / BR;
      for (int blk = c; blk < nblk; blk += g) {
        const int u0 = blk * BR;
        const int nr = min(BR, I.dim_up - u0);
        const int nel = nr * I.dim_dn;
        const T* xb = xc + (int64_t)u0 * I.dim_dn;
        for (int i = threadIdx.x; i < nel; i += blockDim.x) xsm[i] = ld_shared_f(xb + i, multi);
        __syncthreads();
        // (row, column) of element i carried from one iteration to the next: i advances by
        // blockDim.x = sr rows and sd columns
        int r = threadIdx.x / I.dim_dn, d = threadIdx.x - r * I.dim_dn;
        const int sr = blockDim.x / I.dim_dn, sd = blockDim.x - sr * I.dim_dn;
        for (int i = threadIdx.x; i < nel; i += blockDim.x) {
          const int u = u0 + r;
          const T* xr = xsm + r * I.dim_dn;
          T acc = T(0);
          add_hops(acc, I.hd + d, I.dim_dn, I.mhd, (uint32_t)I.dim_dn, [&](uint32_t tg) { return xr[tg]; });
          add_hops(acc, I.hu + u, I.dim_up, I.mhu, (uint32_t)I.dim_up, [&](uint32_t tg) {
            return ld_shared_f(xc + (int64_t)tg * I.dim_dn + d, multi);
          });
          const T xv = xsm[i];
          const int64_t e = (int64_t)u0 * I.dim_dn + i;
          const T hx = fma(-tt, acc, UU * (T)__popc(I.upb[u] & I.dnb[d]) * xv);
          const T w = fma(sc, hx, -bsp * ld_shared_f(xp + e, multi));
          xp[e] = w;
          if (vj) vj[e] = (float)xv;
          dot.add(w, sc * xv);
          r += sr;
          d += sd;
          if (d >= I.dim_dn) {
            d -= I.dim_dn;
            ++r;
          }
        }
        __syncthreads();
      }
    } else {
      // (row, column) of element e carried from one iteration to the next (e < 2^31)
      int u = (int)t0 / I.dim_dn, d = (int)t0 - u * I.dim_dn;
      const int su = (int)gt / I.dim_dn, sdd = (int)gt - su * I.dim_dn;
      for (int64_t e = t0; e < dim; e += gt, u += su, d += sdd) {
        if (d >= I.dim_dn) {
          d -= I.dim_dn;
          ++u;
        }
        const T* xr = xc + (int64_t)u * I.dim_dn;
        T acc = T(0);
        add_hops(acc, I.hd + d, I.dim_dn, I.mhd, (uint32_t)I.dim_dn,
                 [&](uint32_t tg) { return ld_shared_f(xr + tg, multi); });
        add_hops(acc, I.hu + u, I.dim_up, I.mhu, (uint32_t)I.dim_up, [&](uint32_t tg) {
          return ld_shared_f(xc + (int64_t)tg * I.dim_dn + d, multi);
        });
        const T xv = ld_shared_f(xr + d, multi);
        const T hx = fma(-tt, acc, UU * (T)__popc(I.upb[u] & I.dnb[d]) * xv);
        const T w = fma(sc, hx, -bsp * ld_shared_f(xp + e, multi));
        xp[e] = w;
        if (vj) vj[e] = (float)xv;
        dot.add(w, sc * xv);
      }
    }
    {
      const double v = block_sum(dot.get(), red);
      if (threadIdx.x == 0) a.part_a[blockIdx.x] = v;
    }
    if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return false;
    // ---- phase 2: a_j, update
    const double alpha = group_sum(a.part_a, first_cta, g, red);
    if (leader && threadIdx.x == 0) al[j] = alpha;
    const T coef = (T)(alpha * run_s.scale);
    DotAcc<T> q2;
    // (phase 1 wrote w by row blocks: other CTAs' values are read from L2)
    if (I.tab) {  // (rows of a multiple of 16 bytes)
      typedef typename BWide<T>::V V;
      constexpr int W = 16 / (int)sizeof(T);
      for (int64_t e = t0; e < dim / W; e += gt) {
        V w4 = b_ld16(reinterpret_cast<const V*>(xp) + e, multi);
        const V c4 = b_ld16(reinterpret_cast<const V*>(xc) + e, multi);
        T* w = reinterpret_cast<T*>(&w4);
        const T* x = reinterpret_cast<const T*>(&c4);
#pragma unroll
        for (int v = 0; v < W; ++v) {
          w[v] = w[v] - coef * x[v];
          q2.add(w[v], w[v]);
        }
        reinterpret_cast<V*>(xp)[e] = w4;
      }
    } else {
      for (int64_t e = t0; e < dim; e += gt) {
        const T q = ld_shared_f(xp + e, multi) - coef * ld_shared_f(xc + e, multi);
        xp[e] = q;
        q2.add(q, q);
      }
    }
    {
      const double v = block_sum(q2.get(), red);
      if (threadIdx.x == 0) a.part_b[blockIdx.x] = v;
    }
    if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return false;
    // ---- phase 3: b_{j+1} (every CTA, from the same partials); the stop test when due: E0(j) by
    // the leader, then everyone reads the status
    const double b2 = group_sum(a.part_b, first_cta, g, red);
    if (threadIdx.x == 0) {
      const double beta = sqrt(b2);
      const double ts = fmax(run_s.tscale, fabs(alpha) + run_s.beta);
      const int st = (beta > kBreakdownRel * fmax(1.0, ts)) ? 0 : 1;
      run_s.tscale = ts;
      run_s.beta = beta;
      run_s.scale_prev = run_s.scale;
      run_s.scale = st == 0 ? 1.0 / beta : 0.0;
      if (leader) {
        be[j + 1] = beta;
        S->j = j;
        if (st == 0) S->scale[1 - cur] = run_s.scale;
      }
      *stop_s = st;
    }
    __syncthreads();
    int st = *stop_s;
    if (st != 0 || j >= R.max_steps || (R.tol > 0.0 && j % R.check == 0)) {
      if (leader) {
        st = group_stop_test(S, R, al, be, e0, j, st, reinterpret_cast<double*>(bsm));
        if (threadIdx.x == 0) {
          S->status = st;
          __threadfence();
        }
      }
      if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return false;
      if (__ldcg(&S->status) != 0) break;
    }
    cur = 1 - cur;
  }
  return true;
}

template <typename T>
__global__ void __launch_bounds__(kBThreads, bctas_per_sm<T>())
batched_lanczos_kernel(BArgs a) {
  __shared__ double red[33];
  __shared__ int stop_s;
  extern __shared__ __align__(16) unsigned char bsm[];
  const int gi = a.group_of_cta[blockIdx.x];
  const BGroup G = a.groups[gi];
  const int c = blockIdx.x - G.first_cta, g = G.ncta;
  const int stride = a.refine ? a.refine_steps + 2 : a.max_steps + 2;
  for (int oi = G.inst_begin; oi < G.inst_end; ++oi) {
    const int id = a.order[oi];
    const BInst I = a.inst[id];
    RunSpec R;
    if (a.refine) {
      // the FP64 refinement of a mixed solve: from psi, which batched_ritz_kernel left in D1
      R.S = a.st2 + id;
      R.al = a.alpha2 + (size_t)id * stride;
      R.be = a.beta2 + (size_t)id * stride;
      R.e0 = a.E02 + (size_t)id * stride;
      R.B0 = I.D0;
      R.B1 = I.D1;
      R.f1 = I.D1;
      R.max_steps = a.refine_steps;
      R.check = 1;
      R.tol = a.refine_tol;
    } else {
      R.S = a.st + id;
      R.al = a.alpha + (size_t)id * stride;
      R.be = a.beta + (size_t)id * stride;
      R.e0 = a.E0 + (size_t)id * stride;
      R.B0 = I.B0;
      R.B1 = I.B1;
      R.f1 = nullptr;
      R.max_steps = a.max_steps;
      R.check = a.check;
      R.tol = a.tol;
    }
    // mixed solves: the FP32 phase keeps its vectors and their scales (rwork: vscale | y | work)
    R.V = a.store ? I.V : nullptr;
    R.vscale = a.store ? a.rwork + (size_t)id * 4 * stride : nullptr;
    R.dpad = I.dpad;
    if (!run_instance<T>(a, I, R, c, g, G.first_cta, a.bar_count + gi, a.bar_gen + gi, red, &stop_s, bsm))
      return;
  }
}

// Mixed precision per instance (the batched form of ed_lanczos_solve_mixed) in three
// cooperative launches (the first over a plan sized for its kernel's residency, the other two
// over one sized for theirs; all state between them is per instance):
// batched_lanczos_kernel<float> with `store` runs Algorithm 1 in FP32 and keeps its Lanczos
// vectors; batched_ritz_kernel computes the
// eigenvector y of T_m for its lowest eigenvalue (inverse iteration, leader thread) and
// assembles the Ritz vector psi = sum_j y_j f_j into D1; batched_lanczos_kernel<double> with
// `refine` runs Algorithm 1 in FP64 from psi, with E0 checked every step, until the
// refinement's convergence test passes.
__global__ void __launch_bounds__(kBThreads, kBCtasPerSm)
batched_ritz_kernel(BArgs a) {
  __shared__ __align__(16) float coef[ED_MAX_STEPS + 2];  // y_j times the stored vector's scale
  extern __shared__ __align__(16) unsigned char bsm[];    // the leader's T_m, y and work
  const int gi = a.group_of_cta[blockIdx.x];
  const BGroup G = a.groups[gi];
  const int c = blockIdx.x - G.first_cta, g = G.ncta;
  const bool multi = g > 1;
  const int stride = a.max_steps + 2;
  unsigned* bc = a.bar_count + gi;
  unsigned* bg = a.bar_gen + gi;
  for (int oi = G.inst_begin; oi < G.inst_end; ++oi) {
    const int id = a.order[oi];
    const BInst I = a.inst[id];
    double* rw = a.rwork + (size_t)id * 4 * stride;  // vscale | y | inverse-iteration work (2 strides)
    const double* al = a.alpha + (size_t)id * stride;
    const double* be = a.beta + (size_t)id * stride;
    const int m = __ldcg(&a.st[id].j);
    double* y = rw + stride;
    if (c == 0) {  // in shared memory: one thread's chain of dependent operations
      double *as = reinterpret_cast<double*>(bsm), *bs = as + stride, *ys = bs + stride, *work = ys + stride;
      for (int i = threadIdx.x; i < m + 2 && m >= 1; i += blockDim.x) as[i] = al[i], bs[i] = be[i];
      __syncthreads();
      if (threadIdx.x == 0 && m >= 1)
        tridiag_ritz_vector(as, bs, m, __ldcg(&a.E0[(size_t)id * stride + m]), ys, work);
      __syncthreads();
      for (int i = threadIdx.x; i < m + 2 && m >= 1; i += blockDim.x) y[i] = ys[i];
      __threadfence();
    }
    if (!group_barrier(bc, bg, g, a.max_spin, a.error)) return;
    // psi in FP32 arithmetic: it only starts the FP64 refinement, and the FP32 vectors already
    // bound its accuracy far above the FP32 rounding of the sum (GB300's FP64 rate would make
    // this the slowest part of the solve)
    for (int j = 1 + threadIdx.x; j <= m; j += blockDim.x)
      coef[j] = (float)(__ldcg(&y[j]) * __ldcg(&rw[j]));
    __syncthreads();
    const int dim = I.dim_up * I.ld;
    for (int64_t e = (int64_t)c * blockDim.x + threadIdx.x; e < dim; e += (int64_t)g * blockDim.x) {
      float p = 0.f;
      for (int j = 1; j <= m; ++j) p = fmaf(coef[j], ld_shared_f(I.V + (size_t)(j - 1) * I.dpad + e, multi), p);
      I.D1[e] = (double)p;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ schedules
// A schedule maps instances to CTA groups: instances with dim >= big get `gbig` CTAs,
// with dim >= mid get `gmid` CTAs, the rest are queued on single-CTA groups; queues are
// balanced by estimated work (dim x hops x 1), longest first.
// Schedules 5 and 6 instead size groups in proportion to a weight, the work per step (5) or that
// times log2 dim (6), an estimate of the steps growing with the dimension (a random start overlaps
// the ground state by about dim^-1/2): with the smallest load t per CTA that fits, an instance of
// at least 4096 states and weight w > t gets ceil(w / t) CTAs, the rest are queued, largest first,
// on queues of load t. (With round(w / T) from w = 1.5 T on, T = total / CTAs, the instances just
// below took twice the step time of the average and ended the batch: 27.4 ms, CTAs busy 44%.)
struct Sched {
  int big, gbig, mid, gmid;
  int weight;  // proportional schedules: 0 work, 1 work x log2 dim
};
static const Sched kScheds[] = {
    {1 << 30, 1, 1 << 30, 1, 0},  // 0: one CTA per queue, everything queued
    {200000, 8, 20000, 2, 0},     // 1
    {100000, 16, 10000, 4, 0},    // 2
    {400000, 32, 40000, 4, 0},    // 3
    {50000, 8, 5000, 2, 0},       // 4
    {0, 0, 0, 0, 0},              // 5: proportional to work
    {0, 0, 0, 0, 1},              // 6: proportional to work x log2 dim
};
constexpr int kNumScheds = (int)(sizeof(kScheds) / sizeof(kScheds[0]));

struct Plan {
  std::vector<BGroup> groups;
  std::vector<int> group_of_cta;
  std::vector<int> order;
  int grid = 0;
};

static Plan make_plan(const std::vector<long long>& work_in, const std::vector<int>& dims,
                      const Sched& sc, int max_ctas) {
  const int n = (int)dims.size();
  std::vector<long long> work(work_in);
  if (sc.gbig == 0 && sc.weight == 1)
    for (int i = 0; i < n; ++i)
      work[i] = (long long)((double)work_in[i] * std::log2(std::max(2, dims[i])));
  std::vector<int> idx(n);
  for (int i = 0; i < n; ++i) idx[i] = i;
  std::sort(idx.begin(), idx.end(), [&](int a, int b) { return work[a] != work[b] ? work[a] > work[b] : a < b; });
  Plan p;
  int ctas = 0;
  std::vector<int> big_ids, small_ids;
  const bool prop = sc.gbig == 0;
  std::vector<int> gprop(n, 1);
  if (prop) {
    // the smallest t by bisection: groups for w > t, the others on queues of load <= t
    auto fits = [&](double t) {
      long long used = 0;
      for (int i : idx)
        if (dims[i] >= 4096 && (double)work[i] > t) used += (long long)std::ceil((double)work[i] / t);
      const long long left = max_ctas - used;
      std::priority_queue<double, std::vector<double>, std::greater<double>> load;
      for (int i : idx) {
        if (dims[i] >= 4096 && (double)work[i] > t) continue;
        if (left < 1) return false;
        double l = (double)work[i];
        if ((long long)load.size() >= left) {
          l += load.top();
          load.pop();
          if (l > t) return false;
        }
        load.push(l);
      }
      return used <= max_ctas;
    };
    double lo = 0.0, hi = 1.0;
    for (int i = 0; i < n; ++i) hi += (double)work[i];
    lo = hi / (2.0 * max_ctas);
    for (int it = 0; it < 20 && hi > 1.01 * lo; ++it) {
      const double t = std::sqrt(lo * hi);
      if (fits(t)) hi = t;
      else lo = t;
    }
    for (int i = 0; i < n; ++i)
      if (dims[i] >= 4096 && (double)work[i] > hi) gprop[i] = (int)std::ceil((double)work[i] / hi);
  }
  for (int i : idx) {
    int gsz = dims[i] >= sc.big ? sc.gbig : (dims[i] >= sc.mid ? sc.gmid : 1);
    if (prop) gsz = gprop[i];
    const int cap = prop ? max_ctas : max_ctas / 2;
    if (gsz > 1 && ctas + gsz <= cap) {
      BGroup G{ctas, gsz, (int)p.order.size(), (int)p.order.size() + 1};
      p.order.push_back(i);
      p.groups.push_back(G);
      ctas += gsz;
    } else {
      small_ids.push_back(i);
    }
  }
  // single-CTA queues for the rest: as many queues as CTAs remain, longest-processing-first
  int nq = std::max(1, std::min((int)small_ids.size(), max_ctas - ctas));
  std::vector<std::vector<int>> q(nq);
  std::vector<long long> load(nq, 0);
  for (int i : small_ids) {
    int best = 0;
    for (int k = 1; k < nq; ++k)
      if (load[k] < load[best]) best = k;
    q[best].push_back(i);
    load[best] += work[i];
  }
  for (int k = 0; k < nq; ++k) {
    if (q[k].empty()) continue;
    BGroup G{ctas, 1, (int)p.order.size(), (int)p.order.size() + (int)q[k].size()};
    for (int i : q[k]) p.order.push_back(i);
    p.groups.push_back(G);
    ctas += 1;
  }
  p.grid = ctas;
  p.group_of_cta.resize(ctas);
  for (int gi = 0; gi < (int)p.groups.size(); ++gi)
    for (int c = 0; c < p.groups[gi].ncta; ++c) p.group_of_cta[p.groups[gi].first_cta + c] = gi;
  return p;
}

// Autotuned schedule per batch signature (dims and hop counts), cached per process.
static std::mutex g_tune_mu;
static std::map<std::string, int> g_tune_cache;

}  // namespace ed

using namespace ed;

namespace {

// Layout of an instance's vectors: the row-ordered H.v where the basis has its tables (one hop
// class) and a block of rows and its up-hop lists fit the staging area, with rows padded to 4
// elements; else dense rows. Rows shorter than 96 columns leave most warps of the down part idle.
bool blayout_rows(const ed_basis* b) {
  const int64_t ld = (b->dn.dim + 3) / 4 * 4;
  return b->rows.C == 1 && b->rows.ucnt == nullptr && b->up.maxhops * 2 <= kBLists &&
         (2 * ld + 1) * 8 + 4 * kBLists <= kBRowFloats * 4;
}
int blayout_ld(const ed_basis* b) { return blayout_rows(b) ? (int)((b->dn.dim + 3) / 4 * 4) : (int)b->dn.dim; }
size_t blayout_elems(const ed_basis* b) { return ((size_t)b->up.dim * blayout_ld(b) + 3) / 4 * 4; }

struct BatchRun {
  int n = 0;
  cudaStream_t stream = nullptr;  // frees the pooled memory
  std::vector<BInst> hinst;
  std::vector<int> dims;
  std::vector<long long> work;
  std::vector<BState> hs, hs2;  // the instances' final states of the two phases
  int max_ctas = 0, max_ctas2 = 0;
  void* mem = nullptr;        // one block from the library's bounded pool for all but the store:
  void* vec = nullptr;        //   work vectors
  BInst* d_inst = nullptr;
  BState* d_state = nullptr;
  double* d_scal = nullptr;   //   alpha | beta | E0
  int* d_misc = nullptr;      //   error flag
  void* d_plan = nullptr;     //   the launches' plans
  void* d_plan2 = nullptr;
  // mixed solves
  bool mixed = false;
  int refine_steps = 0;
  double refine_tol = 0.0;
  void* vstore = nullptr;     // FP32 Lanczos vectors of every instance
  bool pooled = false;
  void* dvec = nullptr;       //   FP64 refinement vectors
  double* d_rwork = nullptr;
  BState* d_state2 = nullptr;
  double* d_scal2 = nullptr;  //   alpha | beta | E0 of the refinement
  ~BatchRun() {
    if (mem) cudaFreeAsync(mem, stream);
    if (vstore && pooled) cudaFreeAsync(vstore, stream);
    if (vstore && !pooled) cudaFree(vstore);
  }
};

// Device copy of a plan on at most max_ctas CTAs, in one block.
size_t plan_bytes(int max_ctas, int n) {
  return (size_t)max_ctas * (sizeof(BGroup) + sizeof(int) + 2 * sizeof(double) + 2 * sizeof(unsigned)) +
         (size_t)n * sizeof(int) + 64;
}

// The batch's plan for max_ctas CTAs, uploaded to `mem`; sets the plan's fields of a and the grid.
ed_status upload_plan(const BatchRun& R, int sched, int max_ctas, void* mem, BArgs& a, int* grid, cudaStream_t s) {
  const Plan p = make_plan(R.work, R.dims, kScheds[sched], max_ctas);
  double* part = (double*)mem;
  BGroup* groups = (BGroup*)(part + 2 * (size_t)max_ctas);
  int* goc = (int*)(groups + max_ctas);
  int* order = goc + max_ctas;
  unsigned* bar = (unsigned*)(order + R.n);
  ED_TRY_CUDA(cudaMemcpyAsync(groups, p.groups.data(), p.groups.size() * sizeof(BGroup), cudaMemcpyHostToDevice, s));
  ED_TRY_CUDA(cudaMemcpyAsync(goc, p.group_of_cta.data(), p.group_of_cta.size() * sizeof(int), cudaMemcpyHostToDevice, s));
  ED_TRY_CUDA(cudaMemcpyAsync(order, p.order.data(), p.order.size() * sizeof(int), cudaMemcpyHostToDevice, s));
  ED_TRY_CUDA(cudaMemsetAsync(bar, 0, 2 * (size_t)max_ctas * sizeof(unsigned), s));
  // (the plan's host arrays may go: copies from pageable memory are staged when the call returns,
  // and the caller synchronises the stream before the block is freed)
  a.order = order;
  a.groups = groups;
  a.group_of_cta = goc;
  a.part_a = part;
  a.part_b = part + max_ctas;
  a.bar_count = bar;
  a.bar_gen = bar + max_ctas;
  *grid = p.grid;
  return ED_OK;
}

// The whole batch: Algorithm 1 in one cooperative launch and, for a mixed solve, the Ritz vectors
// and the refinement in one each, over a plan for their kernels' residency (all state between the
// launches is per instance).
ed_status run_batch(BatchRun& R, int sched, const ed_opts* o, int check, cudaStream_t s, float* ms_out) {
  const void* kernel = o->dtype == ED_F64_NATIVE ? (const void*)batched_lanczos_kernel<double>
                                                 : (const void*)batched_lanczos_kernel<float>;
  ED_TRY_CUDA(cudaMemsetAsync(R.d_misc, 0, sizeof(int), s));
  BArgs a = {};
  a.inst = R.d_inst;
  a.st = R.d_state;
  const size_t stride = (size_t)o->max_steps + 2;
  a.alpha = R.d_scal;
  a.beta = R.d_scal + stride * R.n;
  a.E0 = R.d_scal + 2 * stride * R.n;
  a.error = R.d_misc;
  a.max_steps = o->max_steps;
  a.check = check;
  a.tol = o->tol;
  a.seed = o->seed;
  a.max_spin = 1000000000LL;  // a group barrier waits at most 1 s
  a.st2 = R.d_state2;
  a.rwork = R.d_rwork;
  const size_t stride2 = (size_t)R.refine_steps + 2;
  a.alpha2 = R.d_scal2;
  a.beta2 = R.d_scal2 ? R.d_scal2 + stride2 * R.n : nullptr;
  a.E02 = R.d_scal2 ? R.d_scal2 + 2 * stride2 * R.n : nullptr;
  a.refine_steps = R.refine_steps;
  a.refine_tol = R.refine_tol;
  a.store = R.mixed ? 1 : 0;
  const auto t0 = std::chrono::steady_clock::now();
  int grid = 0;
  ed_status r = upload_plan(R, sched, R.max_ctas, R.d_plan, a, &grid, s);
  if (r != ED_OK) return r;
  void* args[] = {&a};
  ED_TRY_CUDA(cudaLaunchCooperativeKernel(kernel, grid, kBThreads, args, bsmem_bytes(o->max_steps), s));
  if (R.mixed) {
    BArgs b = a;
    b.store = 0;
    if ((r = upload_plan(R, sched, R.max_ctas2, R.d_plan2, b, &grid, s)) != ED_OK) return r;
    void* args2[] = {&b};
    ED_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)batched_ritz_kernel, grid, kBThreads, args2,
                                            ritz_bytes(o->max_steps), s));
    b.refine = 1;  // (a launch copies its arguments)
    ED_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)batched_lanczos_kernel<double>, grid, kBThreads, args2,
                                            bsmem_bytes(R.refine_steps), s));
    R.hs2.resize(R.n);
    ED_TRY_CUDA(cudaMemcpyAsync(R.hs2.data(), R.d_state2, R.n * sizeof(BState), cudaMemcpyDeviceToHost, s));
  }
  int err = 0;
  R.hs.resize(R.n);
  ED_TRY_CUDA(cudaMemcpyAsync(R.hs.data(), R.d_state, R.n * sizeof(BState), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaMemcpyAsync(&err, R.d_misc, sizeof(int), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  if (err) {
    set_error("batched Lanczos: a group barrier timed out");
    return ED_ERR_TIMEOUT;
  }
  if (ms_out) *ms_out = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
  return ED_OK;
}

}  // namespace

namespace ed {
// Self-test kernel of the bounded group barrier: CTA `absent` never arrives, so the other
// CTAs of the group must give up after `limit_ns` and flag the error.
__global__ void barrier_selftest_kernel(unsigned* bar, int* error, int absent, long long limit_ns) {
  if ((int)blockIdx.x == absent) return;
  group_barrier(bar, bar + 1, gridDim.x, limit_ns, error);
}
}  // namespace ed

extern "C" ed_status ed_selftest_barrier_timeout(int32_t ctas, int32_t timeout_ms, void* stream) {
  clear_error();
  ED_CHECK_ARG(ctas >= 2 && ctas <= 64 && timeout_ms >= 1 && timeout_ms <= 5000,
               "ed_selftest_barrier_timeout: ctas in [2, 64], timeout_ms in [1, 5000]");
  cudaStream_t s = (cudaStream_t)stream;
  unsigned* bar = nullptr;
  int* err = nullptr;
  struct ReleaseOnReturn {  // frees the scratch on every return path, error returns included
    cudaStream_t s;
    unsigned*& bar;
    int*& err;
    ~ReleaseOnReturn() {
      if (bar) cudaFreeAsync(bar, s);
      if (err) cudaFreeAsync(err, s);
    }
  } release{s, bar, err};
  ED_TRY_CUDA(cudaMallocAsync((void**)&bar, 2 * sizeof(unsigned), s));
  ED_TRY_CUDA(cudaMallocAsync((void**)&err, sizeof(int), s));
  ED_TRY_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s));
  ED_TRY_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
  int absent = ctas - 1;
  long long limit = (long long)timeout_ms * 1000000LL;
  void* args[] = {&bar, &err, &absent, &limit};
  ED_TRY_CUDA(cudaLaunchCooperativeKernel((const void*)barrier_selftest_kernel, ctas, 32, args, 0, s));
  int h = 0;
  ED_TRY_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  if (h) {
    set_error("group barrier wait ran out after %d ms (as the self-test intends)", timeout_ms);
    return ED_ERR_TIMEOUT;
  }
  return ED_OK;
}

static ed_status solve_batched(int32_t n, const ed_basis* const* bases, const ed_params* params,
                               const ed_opts* o, bool mixed, int32_t refine_steps, double refine_tol,
                               void* stream, double* E0, int32_t* steps, int32_t* steps64,
                               int32_t* status, int32_t* schedule_used) {
  const char* fn = mixed ? "ed_lanczos_solve_batched_mixed" : "ed_lanczos_solve_batched";
  ED_CHECK_ARG(n >= 1 && bases && params && o && E0, "%s: bad arguments", fn);
  if (mixed)
    ED_CHECK_ARG(o->dtype == ED_F32, "%s: dtype must be ED_F32 (the phase before refinement)", fn);
  else
    ED_CHECK_ARG(o->dtype == ED_F32 || o->dtype == ED_F64_NATIVE,
                 "%s: dtype must be ED_F32 or ED_F64_NATIVE", fn);
  ED_CHECK_ARG(o->reorth == 0, "%s: reorth must be 0 (none)", fn);
  ED_CHECK_ARG(o->max_steps >= 1 && o->max_steps <= ED_MAX_STEPS, "max_steps out of range");
  ED_CHECK_ARG(!mixed || (refine_steps >= 1 && refine_steps <= ED_MAX_STEPS),
               "%s: refine_steps out of range", fn);
  ED_CHECK_ARG(o->schedule >= -1 && o->schedule < kNumScheds, "schedule %d out of range", o->schedule);
  cudaStream_t user = (cudaStream_t)stream;
  cudaStream_t s = nullptr;
  ED_TRY_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
  struct StreamGuard {
    cudaStream_t s;
    ~StreamGuard() { cudaStreamDestroy(s); }
  } guard{s};
  {
    cudaEvent_t ev;
    ED_TRY_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    cudaEventRecord(ev, user);
    cudaStreamWaitEvent(s, ev, 0);
    cudaEventDestroy(ev);
  }
  BatchRun R;
  R.n = n;
  R.hinst.resize(n);
  R.dims.resize(n);
  R.work.resize(n);
  size_t total = 0;
  for (int i = 0; i < n; ++i) {
    const ed_basis* b = bases[i];
    ED_CHECK_ARG(b != nullptr, "%s: basis %d is NULL", fn, i);
    ED_CHECK_ARG(!b->has_tau(), "%s: basis %d has complex amplitudes", fn, i);
    ED_CHECK_ARG(b->dim < (1LL << 31), "%s: instance %d too large", fn, i);
    R.dims[i] = (int)b->dim;
    // (the element-by-element H.v takes about 1.4 times as long as the row-ordered one)
    R.work[i] = (long long)b->dim * (b->up.maxhops + b->dn.maxhops + 4) * (blayout_rows(b) ? 5 : 7);
    ED_CHECK_ARG(b->up.dim * (int64_t)blayout_ld(b) < (1LL << 31), "%s: instance %d too large", fn, i);
    total += blayout_elems(b);
  }
  const size_t esize = o->dtype == ED_F64_NATIVE ? 8 : 4;
  const size_t stride = (size_t)o->max_steps + 2, stride2 = (size_t)refine_steps + 2;
  R.stream = s;
  // a cooperative launch needs every CTA resident: grids of (resident CTAs per SM) x SMs
  int per_sm = 0, per_sm2 = 0;
  if (o->dtype == ED_F64_NATIVE)
    ED_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_lanczos_kernel<double>,
                                                              kBThreads, bsmem_bytes(o->max_steps)));
  else
    ED_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_lanczos_kernel<float>,
                                                              kBThreads, bsmem_bytes(o->max_steps)));
  if (mixed) {  // the Ritz and refinement launches share a limit
    int pm = 0, pd = 0;
    ED_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pm, batched_ritz_kernel, kBThreads,
                                                              ritz_bytes(o->max_steps)));
    ED_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pd, batched_lanczos_kernel<double>,
                                                              kBThreads, bsmem_bytes(refine_steps)));
    per_sm2 = std::min(pm, pd);
  }
  ED_CHECK_ARG(per_sm >= 1 && (!mixed || per_sm2 >= 1), "%s: the batched kernels do not fit an SM", fn);
  R.max_ctas = sm_count() * std::min(per_sm, o->dtype == ED_F64_NATIVE
                                                 ? bctas_per_sm<double>() : bctas_per_sm<float>());
  R.max_ctas2 = sm_count() * std::min(std::max(per_sm2, 1), kBCtasPerSm);
  // ---- one block for the work vectors, states, scalars and plans
  {
    size_t at = 0;
    auto place = [&](size_t bytes) {
      const size_t o0 = at;
      at += (bytes + 255) / 256 * 256;
      return o0;
    };
    const size_t o_vec = place(2 * total * esize), o_inst = place(n * sizeof(BInst)), o_st = place(n * sizeof(BState)),
                 o_misc = place(sizeof(int)), o_plan = place(plan_bytes(R.max_ctas, n)),
                 o_plan2 = place(mixed ? plan_bytes(R.max_ctas2, n) : 0),
                 o_dvec = place(mixed ? 2 * total * sizeof(double) : 0), o_st2 = place(mixed ? n * sizeof(BState) : 0),
                 o_zero = at, o_scal = place(3 * stride * n * sizeof(double)),
                 o_scal2 = place(mixed ? 3 * stride2 * n * sizeof(double) : 0),
                 o_rw = place(mixed ? 4 * stride * n * sizeof(double) : 0);
    cudaMemPool_t pool = psi_pool();
    const cudaError_t e = pool ? cudaMallocFromPoolAsync(&R.mem, at, pool, s) : cudaMallocAsync(&R.mem, at, s);
    if (e != cudaSuccess) {
      cudaGetLastError();
      R.mem = nullptr;
      set_error("%s: %zu bytes of device memory are not available", fn, at);
      return e == cudaErrorMemoryAllocation ? ED_ERR_OOM : ED_ERR_CUDA;
    }
    char* m = (char*)R.mem;
    R.vec = m + o_vec;
    R.d_inst = (BInst*)(m + o_inst);
    R.d_state = (BState*)(m + o_st);
    R.d_misc = (int*)(m + o_misc);
    R.d_plan = m + o_plan;
    R.d_plan2 = m + o_plan2;
    R.d_scal = (double*)(m + o_scal);
    if (mixed) {
      R.dvec = m + o_dvec;
      R.d_state2 = (BState*)(m + o_st2);
      R.d_scal2 = (double*)(m + o_scal2);
      R.d_rwork = (double*)(m + o_rw);
    }
    ED_TRY_CUDA(cudaMemsetAsync(m + o_zero, 0, at - o_zero, s));
  }
  if (mixed) {
    R.mixed = true;
    R.refine_steps = refine_steps;
    R.refine_tol = refine_tol;
    const size_t vbytes = total * (size_t)o->max_steps * sizeof(float);
    cudaMemPool_t pool = vstore_pool();
    const cudaError_t ve = pool ? cudaMallocFromPoolAsync(&R.vstore, vbytes, pool, s) : cudaMalloc(&R.vstore, vbytes);
    if (ve != cudaSuccess) {
      cudaGetLastError();
      R.vstore = nullptr;
      set_error("%s: %zu bytes for the FP32 Lanczos vectors are not available", fn, vbytes);
      return ED_ERR_OOM;
    }
    R.pooled = pool != nullptr;
  }
  size_t off = 0;
  for (int i = 0; i < n; ++i) {
    const ed_basis* b = bases[i];
    BInst& I = R.hinst[i];
    I.upb = b->up.bits;
    I.dnb = b->dn.bits;
    I.hu = b->up.hop;
    I.hd = b->dn.hop;
    I.dim_up = (int)b->up.dim;
    I.dim_dn = (int)b->dn.dim;
    I.mhu = b->up.maxhops;
    I.mhd = b->dn.maxhops;
    const bool rows = blayout_rows(b);
    I.ld = blayout_ld(b);
    I.perm = b->rows.perm;
    I.base = b->rows.base;
    I.kc = b->rows.kc;
    I.tab = rows ? b->rows.tab : nullptr;
    const size_t dpad = blayout_elems(b);
    I.dpad = (int)dpad;
    // the two work vectors of an instance side by side (per instance: B0, B1; D0, D1)
    I.B0 = (char*)R.vec + 2 * off * esize;
    I.B1 = (char*)R.vec + (2 * off + dpad) * esize;
    I.V = mixed ? (float*)R.vstore + off * (size_t)o->max_steps : nullptr;
    I.D0 = mixed ? (double*)R.dvec + 2 * off : nullptr;
    I.D1 = mixed ? (double*)R.dvec + 2 * off + dpad : nullptr;
    off += dpad;
    I.t = params[i].t;
    I.U = params[i].U;
  }
  ED_TRY_CUDA(cudaMemcpyAsync(R.d_inst, R.hinst.data(), n * sizeof(BInst), cudaMemcpyHostToDevice, s));
  const int check = 4;  // E0(j) every 4 steps (and at the stop step)
  int sched = o->schedule;
  if (sched < 0) {
    // autotune: time every candidate schedule on this batch with a short plain run (the
    // schedules pack the same H.v work in both forms), keep the best
    std::string key;
    for (int i = 0; i < n; ++i) key += std::to_string(R.work[i]) + ",";
    key += std::to_string(R.max_ctas) + "/" + std::to_string((int)o->dtype);
    {
      std::lock_guard<std::mutex> lk(g_tune_mu);
      auto it = g_tune_cache.find(key);
      if (it != g_tune_cache.end()) sched = it->second;
    }
    if (sched < 0) {
      // the real solve (its tolerance, at most 200 steps): how instances converge decides
      // the batch's tail as much as the work per step does
      ed_opts ot = *o;
      ot.max_steps = std::min(o->max_steps, 200);
      const bool was_mixed = R.mixed;
      R.mixed = false;
      float best = 1e30f;
      for (int k = 0; k < kNumScheds; ++k) {
        float ms = 0.f;
        ed_status r = run_batch(R, k, &ot, check, s, &ms);
        if (r != ED_OK) return r;
        if (ms < best) best = ms, sched = k;
      }
      R.mixed = was_mixed;
      std::lock_guard<std::mutex> lk(g_tune_mu);
      g_tune_cache[key] = sched;
    }
  }
  ed_status r = run_batch(R, sched, o, check, s, nullptr);
  if (r != ED_OK) return r;
  const std::vector<BState>&hs = R.hs, &hs2 = R.hs2;
  const size_t stride_out = mixed ? stride2 : stride;
  std::vector<double> hE(stride_out * n);
  ED_TRY_CUDA(cudaMemcpyAsync(hE.data(), mixed ? R.d_scal2 + 2 * stride2 * n : R.d_scal + 2 * stride * n,
                              stride_out * n * sizeof(double), cudaMemcpyDeviceToHost, s));
  ED_TRY_CUDA(cudaStreamSynchronize(s));
  bool all_conv = true;
  for (int i = 0; i < n; ++i) {
    const BState& F = mixed ? hs2[i] : hs[i];
    const int j = F.j;
    E0[i] = j >= 1 ? hE[(size_t)i * stride_out + j] : NAN;
    if (steps) steps[i] = hs[i].j;
    if (steps64) steps64[i] = mixed ? hs2[i].j : 0;
    if (status) status[i] = F.status;
    if (F.status == 3 && (mixed ? refine_tol : o->tol) > 0.0) all_conv = false;
  }
  if (schedule_used) *schedule_used = sched;
  if (!all_conv) {
    set_error("%s: some instances reached max_steps before converging", fn);
    return ED_ERR_NOT_CONVERGED;
  }
  return ED_OK;
}

extern "C" ed_status ed_lanczos_solve_batched(int32_t n, const ed_basis* const* bases,
                                              const ed_params* params, const ed_opts* o,
                                              void* stream, double* E0, int32_t* steps,
                                              int32_t* status, int32_t* schedule_used) {
  clear_error();
  return solve_batched(n, bases, params, o, false, 0, 0.0, stream, E0, steps, nullptr, status,
                       schedule_used);
}

extern "C" ed_status ed_lanczos_solve_batched_mixed(int32_t n, const ed_basis* const* bases,
                                                    const ed_params* params, const ed_opts* o,
                                                    int32_t refine_steps, double refine_tol,
                                                    void* stream, double* E0, int32_t* steps32,
                                                    int32_t* steps64, int32_t* status,
                                                    int32_t* schedule_used) {
  clear_error();
  return solve_batched(n, bases, params, o, true, refine_steps, refine_tol, stream, E0, steps32,
                       steps64, status, schedule_used);
}
