// Row-ordered H.v: y = H x on caller vectors (every dtype) and the Lanczos-fused form of the
// FP64 and complex FP64 runs (Sec. 4, Eqs. 5-6), for rows that fit in shared memory twice.
//
//   y[u,d] = U popc(up & dn) x[u,d] + sum_c A_c ( sum of s x[u,tgt] over the down hops of class c
//                                              + sum of s x[tgt,d] over the up hops of class c )
//
// A class is one hopping amplitude up to sign (one class without per-bond amplitudes): hops are
// summed with their signs alone and the sum is multiplied once per class, two additions per
// complex hop instead of four multiply-adds. That is what bounds the FP64 forms: GB300 issues a
// warp-wide FP64 instruction every 16-19 cycles per SM.
//
// A CTA stages R up rows in shared memory (xs, interleaved by row, a zero column at dim_dn).
//  * Down part: a warp takes 32 columns with (nearly) equal hop counts per class (perm: columns
//    sorted by their counts; rank order would make a warp run to the largest count of 32
//    unrelated states, and a table of constant row length to the largest of the basis: 20
//    instead of 14.7 hops on the 4x4 lattice at 5/5) and leaves the sums in shared memory (ys).
//  * Up part: consecutive columns per thread, so neighbour rows are read in wide coalesced
//    loads, four in flight; then the diagonal and the store (or the Lanczos epilogue).
// The grid is one resident wave; a CTA takes every grid-th row group (in the order that keeps
// neighbours in L2).
// Measured against the row-staged kernels with one padded list length per basis (ed_hv.cu,
// ed_hvc.cu), which stay for rows too long or too short for this one (rows_usable): FP32, 14-site
// ring 7/7: 178 -> 103 us; FP64, 4x4 5/5: 1664 -> 1107 us; complex FP64 on the 4x4 checkerboard-type
// lattice (73 hops per state, 4 classes): 18.9 -> 6.6 ms.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <numeric>
#include <type_traits>
#include <vector>

#include "ed_internal.cuh"

namespace ed {

// ------------------------------------------------------------------ tables
// f(class, entry with the amplitude's flip in its sign) for the hops of state s in table order (cls:
// class | flip << 7 of an amplitude number; NULL: class 0), four loaded before the first is taken: one
// state's list is a chain of dependent loads otherwise, 1 us a hop.
template <typename F>
__device__ __forceinline__ void for_hops(const int32_t* __restrict__ hop, const int32_t* __restrict__ hopa,
                                         const uint8_t* __restrict__ cls, int64_t dim, int maxhops, int64_t s, F f) {
  for (int k = 0; k < maxhops; k += 4) {
    uint32_t e[4], m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = k + i < maxhops ? (uint32_t)hop[(int64_t)(k + i) * dim + s] : (uint32_t)dim;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      m[i] = cls && (int64_t)(e[i] & kTargetMask) < dim ? cls[hopa[(int64_t)(k + i) * dim + s]] : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if ((int64_t)(e[i] & kTargetMask) >= dim) return;
      f((int)(m[i] & 0x7F), e[i] ^ (m[i] >> 7 << 31));
    }
  }
}

constexpr int kRowsThreads = 128;

// counts[s * C + c] = hops of state s in class c.
__global__ void __launch_bounds__(kRowsThreads)
rows_count_kernel(const int32_t* __restrict__ hop, const int32_t* __restrict__ hopa, const uint8_t* __restrict__ cls,
                  int64_t dim, int maxhops, int C, uint8_t* __restrict__ counts) {
  __shared__ uint8_t n[kMaxClasses][kRowsThreads];
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < dim; s += (int64_t)gridDim.x * blockDim.x) {
    for (int c = 0; c < C; ++c) n[c][threadIdx.x] = 0;
    for_hops(hop, hopa, cls, dim, maxhops, s, [&](int c, uint32_t) { ++n[c][threadIdx.x]; });
    for (int c = 0; c < C; ++c) counts[s * C + c] = n[c][threadIdx.x];
  }
}

// Down table: per chunk of 32 columns and class the hops of perm's columns, kc[chunk * C + c] rows
// of 32 entries (target, sign in bit 15; the zero column dim pads short lists).
__global__ void __launch_bounds__(kRowsThreads)
rows_down_kernel(const int32_t* __restrict__ hop, const int32_t* __restrict__ hopa, const uint8_t* __restrict__ cls,
                 int64_t dim, int maxhops, int C, const int32_t* __restrict__ perm, const int32_t* __restrict__ base,
                 const uint8_t* __restrict__ kc, int nchunks, uint16_t* __restrict__ tab) {
  __shared__ uint16_t at[kMaxClasses][kRowsThreads];  // the class's next row
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 32 * nchunks; i += gridDim.x * blockDim.x) {
    const int ch = i >> 5, d = perm[i];
    uint16_t* t = tab + base[ch] + (i & 31);
    for (int c = 0, row = 0; c < C; row += kc[ch * C + c], ++c) at[c][threadIdx.x] = (uint16_t)row;
    if (d >= 0)
      for_hops(hop, hopa, cls, dim, maxhops, d, [&](int c, uint32_t e) {
        t[32 * at[c][threadIdx.x]++] = (uint16_t)((e & kTargetMask) | (e >> 31 << 15));
      });
    for (int c = 0, end = 0; c < C; ++c) {
      end += kc[ch * C + c];
      for (int row = at[c][threadIdx.x]; row < end; ++row) t[32 * row] = (uint16_t)dim;
    }
  }
}

// Exclusive sum of v over the CTA's threads (kSortThreads of them; sm: 32 words).
constexpr int kSortThreads = 1024;
__device__ __forceinline__ int block_scan(int v, int* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int in = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int w = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) in += w;
  }
  if (lane == 31) sm[warp] = in;
  __syncthreads();
  int pre = lane < warp ? sm[lane] : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xffffffffu, pre, o);
  __syncthreads();
  return pre + in - v;
}

// Columns by their hop counts, descending, class 0 first, ties by rank (perm, -1 pads), then a
// chunk's rows per class (kc) and start in the table (base). One CTA: a stable counting sort per class,
// the last class first; a warp takes a run of columns, 32 at a time, ranked by __match_any_sync.
__global__ void __launch_bounds__(kSortThreads)
rows_sort_kernel(const uint8_t* __restrict__ counts, int nd, int C, int nchunks, int32_t* __restrict__ perm,
                 int32_t* __restrict__ tmp, uint8_t* __restrict__ kc, int32_t* __restrict__ base) {
  __shared__ int place[256][32];  // [255 - count][warp]: columns, then where the next one goes
  __shared__ int sm[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int run = (nd + 32 * 32 - 1) / (32 * 32) * 32, i0 = warp * run, i1 = min(nd, i0 + run);
  int* flat = &place[0][0];
  for (int c = C - 1; c >= 0; --c) {
    const int32_t* src = c & 1 ? perm : tmp;  // the last sort (class 0) writes perm
    int32_t* dst = c & 1 ? tmp : perm;
    for (int i = threadIdx.x; i < 256 * 32; i += kSortThreads) flat[i] = 0;
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      for (int i = i0; i < i1; i += 32) {
        const int q = i + lane;
        const int d = q < i1 ? (c == C - 1 ? q : src[q]) : 0;
        const int key = q < i1 ? 255 - counts[(int64_t)d * C + c] : 256;
        const unsigned same = __match_any_sync(0xffffffffu, key);
        int* p = key < 256 ? &place[key][warp] : nullptr;
        if (pass && p) dst[*p + __popc(same & ((1u << lane) - 1u))] = d;
        __syncwarp();
        if (p && lane == __ffs(same) - 1) *p += __popc(same);
        __syncwarp();
      }
      __syncthreads();
      if (pass) continue;
      int v[8], sum = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) sum += v[k] = flat[8 * threadIdx.x + k];
      int at = block_scan(sum, sm);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        flat[8 * threadIdx.x + k] = at;
        at += v[k];
      }
      __syncthreads();
    }
  }
  for (int i = nd + threadIdx.x; i < 32 * nchunks; i += kSortThreads) perm[i] = -1;
  __syncthreads();
  for (int ch = warp; ch < nchunks; ch += 32) {
    const int d = perm[32 * ch + lane];
    int rows = 0;
    for (int c = 0; c < C; ++c) {
      const unsigned n = __reduce_max_sync(0xffffffffu, d >= 0 ? (unsigned)counts[(int64_t)d * C + c] : 0u);
      if (lane == 0) kc[ch * C + c] = (uint8_t)n;
      rows += (int)n;
    }
    if (lane == 0) base[ch] = 32 * rows;
  }
  __syncthreads();
  const int t = threadIdx.x, n = t < nchunks ? base[t] : 0;  // (nchunks <= 1,024: rows below 32,767 columns)
  const int at = block_scan(n, sm);
  if (t < nchunks) base[t] = at;
}

// Up table with per-bond amplitudes: the hops of a row class by class, sign flips applied.
__global__ void __launch_bounds__(kRowsThreads)
rows_up_kernel(const int32_t* __restrict__ hop, const int32_t* __restrict__ hopa, const uint8_t* __restrict__ cls,
               int64_t dim, int maxhops, int C, const uint8_t* __restrict__ counts, int32_t* __restrict__ out) {
  __shared__ uint16_t at[kMaxClasses][kRowsThreads];
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < dim; s += (int64_t)gridDim.x * blockDim.x) {
    for (int c = 0, n = 0; c < C; n += counts[s * C + c], ++c) at[c][threadIdx.x] = (uint16_t)n;
    for_hops(hop, hopa, cls, dim, maxhops, s,
             [&](int c, uint32_t e) { out[(int64_t)at[c][threadIdx.x]++ * dim + s] = (int32_t)e; });
  }
}

void rows_free(ed_basis* b) {
  if (b->rows.mem) cudaFree(b->rows.mem);
  b->rows = HvRows();
}

// Classes: distinct amplitudes up to sign (amplitude number 2 q: tau_q, 2 q + 1: its conjugate, the
// gather amplitudes over -t). p.C = 0: no tables for this basis.
void rows_plan(int n_sites, int n_up, int n_dn, const double* t_bond, int n_bonds, RowsPlan& p) {
  if (t_bond) {
    p.cls.resize(2 * (size_t)n_bonds);
    for (size_t i = 0; i < p.cls.size(); ++i) {
      const double re = t_bond[2 * (i / 2)], im = (i & 1) ? -t_bond[2 * (i / 2) + 1] : t_bond[2 * (i / 2) + 1];
      size_t c = 0;
      while (c < p.amp.size() && !(p.amp[c].x == re && p.amp[c].y == im) && !(p.amp[c].x == -re && p.amp[c].y == -im))
        ++c;
      if (c == p.amp.size()) p.amp.push_back(make_double2(re, im));
      p.cls[i] = (uint8_t)(c | (p.amp[c].x == re && p.amp[c].y == im ? 0 : 0x80));
      if (p.amp.size() > kMaxClasses) return;  // too many to pay: the plain kernels
    }
    // per element: 2 additions per hop and 4 multiply-adds per class and species, against 4
    // multiply-adds per hop of the plain kernels: taken while the classes cost no more than the
    // additions save (4 classes for 73 hops on the checkerboard-type lattice). A bond's ends are
    // occupied differently, so it hops, in 2 n (L - n) / (L (L - 1)) of a species' states.
    const double L = n_sites, pairs = L > 1 ? L * (L - 1) : 1;
    const double hops = 2.0 * n_bonds * (n_up * (L - n_up) + n_dn * (L - n_dn)) / pairs;
    if (8.0 * (double)p.amp.size() > 2.0 * hops && !p.amp.empty()) return;
  }
  if (p.amp.empty()) p.amp.push_back(make_double2(1.0, 0.0));
  p.C = (int)p.amp.size();
}

// Enqueue the tables: five launches and a copy at most, no wait (p and t_bond's classes stay until s
// has passed them). Sorted on the host, with the counts' way there and back, they made ed_build_basis
// 4-8% longer, 20% with amplitudes; so they are made beside the host's work on the row order.
ed_status rows_build(ed_basis* b, RowsPlan& p, cudaStream_t s) {
  const int64_t nd = b->dn.dim, nu = b->up.dim;
  if (p.C == 0 || nu < kMinRowsStaged || nd < kMinRowCols || nd >= 0x7FFF || b->dn.maxhops > 255 || b->up.maxhops > 255)
    return ED_OK;
  const int C = p.C, nch = (int)((nd + 31) / 32);
  const bool amps = !p.cls.empty();
  // one allocation: amplitudes and classes (from the host), the counts and the sort's second buffer,
  // the tables. A chunk has as many rows of a class as one of its columns has hops in it: one per bond
  // at most, or two where the two directions of a bond are of different classes (complex amplitudes:
  // columns that hop one way and columns that hop the other can share a chunk).
  HvRows& r = b->rows;
  auto up16 = [](size_t n) { return (n + 15) / 16 * 16; };
  int chunk_rows = b->dn.maxhops;
  if (amps) {
    int n = 0;
    for (size_t q = 0; q < p.cls.size(); q += 2) n += (p.cls[q] & 0x7F) == (p.cls[q + 1] & 0x7F) ? 1 : 2;
    chunk_rows = std::min(C * b->dn.maxhops, n);
  }
  const size_t rows = (size_t)nch * chunk_rows;
  const size_t o_cls = up16(C * sizeof(double2)), o_cnt = up16(o_cls + p.cls.size()), o_ucnt = up16(o_cnt + nd * C),
               o_tmp = up16(o_ucnt + (amps ? nu * C : 0)), o_perm = up16(o_tmp + nd * 4),
               o_base = up16(o_perm + 32 * (size_t)nch * 4), o_kc = up16(o_base + nch * 4),
               o_tab = up16(o_kc + (size_t)nch * C), o_up = up16(o_tab + rows * 64),
               bytes = o_up + (amps ? (size_t)b->up.maxhops * nu * 4 : 0);
  const cudaError_t e = cudaMalloc(&r.mem, bytes + 16);
  if (e == cudaErrorMemoryAllocation) {  // the basis goes without (the row-staged kernels serve it)
    cudaGetLastError();
    r.mem = nullptr;
    return ED_OK;
  }
  ED_TRY_CUDA(e);
  char* m = (char*)r.mem;
  uint8_t* cls = amps ? (uint8_t*)(m + o_cls) : nullptr;
  uint8_t* cnt = (uint8_t*)(m + o_cnt);
  r.amp = (double2*)m;
  r.ucnt = amps ? (uint8_t*)(m + o_ucnt) : nullptr;
  r.perm = (int32_t*)(m + o_perm);
  r.base = (int32_t*)(m + o_base);
  r.kc = (uint8_t*)(m + o_kc);
  r.tab = (uint16_t*)(m + o_tab);
  r.up = amps ? (int32_t*)(m + o_up) : b->up.hop;
  r.nchunks = nch;
  p.host.resize(o_cnt);
  memcpy(p.host.data(), p.amp.data(), C * sizeof(double2));
  if (amps) memcpy(&p.host[o_cls], p.cls.data(), p.cls.size());
  ED_TRY_CUDA(cudaMemcpyAsync(m, p.host.data(), o_cnt, cudaMemcpyHostToDevice, s));
  auto grid = [](int64_t n) { return (unsigned)std::min<int64_t>((n + kRowsThreads - 1) / kRowsThreads, 1024); };
  rows_count_kernel<<<grid(nd), kRowsThreads, 0, s>>>(b->dn.hop, b->dn.hopa, cls, nd, b->dn.maxhops, C, cnt);
  rows_sort_kernel<<<1, kSortThreads, 0, s>>>(cnt, (int)nd, C, nch, r.perm, (int32_t*)(m + o_tmp), r.kc, r.base);
  rows_down_kernel<<<grid(32 * (int64_t)nch), kRowsThreads, 0, s>>>(b->dn.hop, b->dn.hopa, cls, nd, b->dn.maxhops, C,
                                                                    r.perm, r.base, r.kc, nch, r.tab);
  if (amps) {
    rows_count_kernel<<<grid(nu), kRowsThreads, 0, s>>>(b->up.hop, b->up.hopa, cls, nu, b->up.maxhops, C, r.ucnt);
    rows_up_kernel<<<grid(nu), kRowsThreads, 0, s>>>(b->up.hop, b->up.hopa, cls, nu, b->up.maxhops, C, r.ucnt, r.up);
  }
  ED_TRY_CUDA(cudaGetLastError());
  r.C = C;
  return ED_OK;
}

// ------------------------------------------------------------------ the product
struct RowsArgs {
  const uint32_t* __restrict__ up_bits;
  const uint32_t* __restrict__ dn_bits;
  const int32_t* __restrict__ order;  // up-row visit order (NULL = rank order)
  const int32_t* __restrict__ up;     // [maxhops_up][dim_up], class by class
  const uint8_t* __restrict__ ucnt;   // [dim_up][C] (NULL: one class, the list ends at its padding)
  const int32_t* __restrict__ perm;
  const int32_t* __restrict__ base;
  const uint8_t* __restrict__ kc;
  const uint16_t* __restrict__ tab;
  const double2* __restrict__ amp;
  int64_t dim_up, ld;
  int dim_dn, nchunks, C, maxhops_up;
  double t, U;
};

template <typename E> struct RowElem;
template <> struct RowElem<float> { typedef float T; static constexpr int kWide = 4; };
template <> struct RowElem<double> { typedef double T; static constexpr int kWide = 2; };
template <> struct RowElem<float2> { typedef float T; static constexpr int kWide = 2; };
template <> struct RowElem<double2> { typedef double T; static constexpr int kWide = 1; };

template <typename T> __device__ __forceinline__ void row_mad(T& a, T c, T x) { a = fma(c, x, a); }
__device__ __forceinline__ void row_mad(float2& a, float c, float2 x) { a.x = fma(c, x.x, a.x), a.y = fma(c, x.y, a.y); }
__device__ __forceinline__ void row_mad(double2& a, double c, double2 x) { a.x = fma(c, x.x, a.x), a.y = fma(c, x.y, a.y); }
// a += A s for the amplitude A = (re, im) of a class (real vectors: re alone)
template <typename T> __device__ __forceinline__ void row_amp(T& a, T re, T, T s) { a = fma(re, s, a); }
template <typename T, typename V> __device__ __forceinline__ void row_amp2(V& a, T re, T im, V s) {
  a.x = fma(re, s.x, a.x);
  a.y = fma(re, s.y, a.y);
  if (im != T(0)) {  // the same for all threads
    a.x = fma(-im, s.y, a.x);
    a.y = fma(im, s.x, a.y);
  }
}
__device__ __forceinline__ void row_amp(float2& a, float re, float im, float2 s) { row_amp2(a, re, im, s); }
__device__ __forceinline__ void row_amp(double2& a, double re, double im, double2 s) { row_amp2(a, re, im, s); }

template <typename E, int N>
struct alignas(sizeof(E) * N) RowPack {
  E v[N];
};

// w = sc h - bsp P and the dot product with sc x
template <typename T> __device__ __forceinline__ T row_lz(T sc, T bsp, T h, T P, T x, DotAcc<T>& dot) {
  const T w = sc * h - bsp * P;
  dot.add(w, sc * x);
  return w;
}
template <typename T, typename V>
__device__ __forceinline__ V row_lz2(T sc, T bsp, V h, V P, V x, DotAcc<T>& dot) {
  V w;
  w.x = row_lz(sc, bsp, h.x, P.x, x.x, dot);
  w.y = row_lz(sc, bsp, h.y, P.y, x.y, dot);
  return w;
}
__device__ __forceinline__ float2 row_lz(float sc, float bsp, float2 h, float2 P, float2 x, DotAcc<float>& d) {
  return row_lz2(sc, bsp, h, P, x, d);
}
__device__ __forceinline__ double2 row_lz(double sc, double bsp, double2 h, double2 P, double2 x, DotAcc<double>& d) {
  return row_lz2(sc, bsp, h, P, x, d);
}

template <typename E, int R, int T, int MB, bool kLz>
__global__ void __launch_bounds__(T, MB)
hv_rows_kernel(RowsArgs a, const E* __restrict__ x, E* __restrict__ y, LzHvArgs lz, int wide) {
  typedef typename RowElem<E>::T F;
  constexpr int W = RowElem<E>::kWide;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[33];
  __shared__ F diag[kMaxSites + 1];              // U n
  __shared__ F amp[2 * kMaxClasses];             // -t tau of each class
  __shared__ int ubound[R][kMaxClasses + 1];     // up-hop list bounds of each class
  F sc = F(1), bsp = F(0);
  if (kLz) {
    if (lz.S->status != 0) return;
    sc = (F)lz.S->scale[lz.cur];
    bsp = (F)(lz.S->beta[lz.S->j + 1] * lz.S->scale[1 - lz.cur]);
  }
  const int dn = a.dim_dn, C = a.C;
  RowPack<E, R>* xs = reinterpret_cast<RowPack<E, R>*>(smem);  // [dn + 1]
  E* ys = reinterpret_cast<E*>(xs + dn + 1);                   // [R][dn]
  uint32_t* ue = reinterpret_cast<uint32_t*>(ys + (size_t)R * dn);  // [R][maxhops_up]
  if (threadIdx.x <= kMaxSites) diag[threadIdx.x] = (F)(a.U * (double)threadIdx.x);
  if (threadIdx.x < C) {
    amp[2 * threadIdx.x] = (F)(-a.t * a.amp[threadIdx.x].x);
    amp[2 * threadIdx.x + 1] = (F)(-a.t * a.amp[threadIdx.x].y);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  DotAcc<F> dot;
  const int ngroups = (int)((a.dim_up + R - 1) / R);
  for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
    int64_t urow[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t q = (int64_t)g * R + r;
      urow[r] = q < a.dim_up ? (a.order ? (int64_t)a.order[q] : q) : a.dim_up;  // dim_up = none
    }
    __syncthreads();  // the rows before are done with xs and the lists
    // ---- stage the rows, their up-hop lists and the lists' class bounds
    for (int d = threadIdx.x; d <= dn; d += T) {
      RowPack<E, R> p;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        p.v[r] = E();
        if (d < dn && urow[r] < a.dim_up) p.v[r] = x[urow[r] * a.ld + d];
      }
      xs[d] = p;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (warp != r) continue;
      const int64_t u = urow[r];
      int n = 0;
      for (int k0 = 0; k0 < a.maxhops_up; k0 += 32) {
        const int k = k0 + lane;
        const uint32_t e = k < a.maxhops_up && u < a.dim_up ? (uint32_t)a.up[(int64_t)k * a.dim_up + u]
                                                            : (uint32_t)a.dim_up;
        if (k < a.maxhops_up) ue[r * a.maxhops_up + k] = e;
        if (!a.ucnt) n += __popc(__ballot_sync(0xffffffffu, (int64_t)(e & kTargetMask) < a.dim_up));
      }
      if (lane == 0) {
        ubound[r][0] = 0;
        for (int c = 0; c < C; ++c)
          ubound[r][c + 1] = a.ucnt ? ubound[r][c] + (u < a.dim_up ? a.ucnt[u * C + c] : 0) : n;
      }
    }
    __syncthreads();
    // ---- down part, 32 columns of equal hop counts per warp
    for (int ch = warp; ch < a.nchunks; ch += T / 32) {
      const int p = a.perm[32 * ch + lane];
      const uint16_t* tp = a.tab + a.base[ch] + lane;
      E out[R];
#pragma unroll
      for (int r = 0; r < R; ++r) out[r] = E();
      for (int c = 0; c < C; ++c) {
        const int n = a.kc[ch * C + c];
        E acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = E();
        int k = 0;
        for (; k + 4 <= n; k += 4) {
          uint32_t e[4];
          RowPack<E, R> q[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i] = tp[32 * (k + i)];
#pragma unroll
          for (int i = 0; i < 4; ++i) q[i] = xs[e[i] & 0x7FFFu];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int r = 0; r < R; ++r) row_mad(acc[r], sign_one(e[i] << 16, F()), q[i].v[r]);
        }
        for (; k < n; ++k) {
          const uint32_t e = tp[32 * k];
          const RowPack<E, R> q = xs[e & 0x7FFFu];
#pragma unroll
          for (int r = 0; r < R; ++r) row_mad(acc[r], sign_one(e << 16, F()), q.v[r]);
        }
        tp += 32 * n;
#pragma unroll
        for (int r = 0; r < R; ++r) row_amp(out[r], amp[2 * c], amp[2 * c + 1], acc[r]);
      }
      if (p >= 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) ys[r * dn + p] = out[r];
      }
    }
    __syncthreads();
    // ---- up part, diagonal and result: W consecutive columns per thread where rows are
    // aligned for it, else one
    auto columns = [&](auto width, int d0) {
      constexpr int N = decltype(width)::value;
      uint32_t db[N];
#pragma unroll
      for (int v = 0; v < N; ++v) db[v] = a.dn_bits[d0 + v];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int64_t u = urow[r];
        if (u >= a.dim_up) continue;
        const uint32_t* ul = ue + r * a.maxhops_up;
        const E* xb = x + d0;
        E out[N];
#pragma unroll
        for (int v = 0; v < N; ++v) out[v] = ys[r * dn + d0 + v];
        int k = 0;
        for (int c = 0; c < C; ++c) {
          const int end = ubound[r][c + 1];
          E acc[N];
#pragma unroll
          for (int v = 0; v < N; ++v) acc[v] = E();
          for (; k + 4 <= end; k += 4) {
            RowPack<E, N> q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              q[i] = *reinterpret_cast<const RowPack<E, N>*>(xb + (int64_t)(ul[k + i] & kTargetMask) * a.ld);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int v = 0; v < N; ++v) row_mad(acc[v], sign_one(ul[k + i], F()), q[i].v[v]);
          }
          for (; k < end; ++k) {
            const RowPack<E, N> q = *reinterpret_cast<const RowPack<E, N>*>(xb + (int64_t)(ul[k] & kTargetMask) * a.ld);
#pragma unroll
            for (int v = 0; v < N; ++v) row_mad(acc[v], sign_one(ul[k], F()), q.v[v]);
          }
#pragma unroll
          for (int v = 0; v < N; ++v) row_amp(out[v], amp[2 * c], amp[2 * c + 1], acc[v]);
        }
        const uint32_t ub = a.up_bits[u];
        RowPack<E, N>* yp = reinterpret_cast<RowPack<E, N>*>(y + u * a.ld + d0);
        RowPack<E, N> P, w;
        if (kLz) P = *yp;
#pragma unroll
        for (int v = 0; v < N; ++v) {
          const E xc = xs[d0 + v].v[r];
          row_mad(out[v], diag[__popc(ub & db[v])], xc);
          w.v[v] = kLz ? row_lz(sc, bsp, out[v], P.v[v], xc, dot) : out[v];
        }
        *yp = w;
      }
    };
    const int dw = wide ? dn / W * W : 0;
    for (int d0 = threadIdx.x * W; d0 < dw; d0 += T * W) columns(std::integral_constant<int, W>(), d0);
    for (int d0 = dw + threadIdx.x; d0 < dn; d0 += T) columns(std::integral_constant<int, 1>(), d0);
  }
  if (kLz) {
    const double v = block_sum(dot.get(), red);
    if (threadIdx.x == 0) lz.partial[blockIdx.x] = v;
  }
}

// ------------------------------------------------------------------ host side
template <typename E, int R>
static size_t rows_smem(const ed_basis* b) {
  return ((size_t)(b->dn.dim + 1) + (size_t)b->dn.dim) * R * sizeof(E) + (size_t)R * b->up.maxhops * 4;
}

// Shared-memory limit and resident CTAs of one kernel on the current device, looked up once per
// device and shared-memory size.
template <typename K>
static ed_status rows_wave(K kernel, int threads, size_t smem, int64_t want, std::atomic<uint64_t>* cache, int* grid) {
  int dev = 0;
  ED_TRY_CUDA(cudaGetDevice(&dev));
  const uint64_t key = ((uint64_t)(dev + 1) << 40) | ((uint64_t)smem << 8);
  uint64_t have = cache->load(std::memory_order_acquire);
  if ((have & ~(uint64_t)0xFF) != key) {
    ED_TRY_CUDA(allow_max_smem(kernel));
    int per_sm = 0;
    ED_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
    ED_CHECK_ARG(per_sm >= 1 && per_sm < 256, "H.v rows: the kernel does not fit an SM");
    have = key | (uint64_t)per_sm;
    cache->store(have, std::memory_order_release);
  }
  *grid = (int)std::min<int64_t>(want, (int64_t)(have & 0xFF) * sm_count());
  return ED_OK;
}

template <typename E, int R, int T, int MB, bool kLz>
static ed_status rows_launch(const ed_basis* b, const RowsArgs& a, const E* x, E* y, cudaStream_t s,
                             const LzHvArgs& lz, int* grid_out) {
  static std::atomic<uint64_t> cache{0};
  const size_t smem = rows_smem<E, R>(b);
  int grid = 0;
  const ed_status r = rows_wave(hv_rows_kernel<E, R, T, MB, kLz>, T, smem, (b->up.dim + R - 1) / R, &cache, &grid);
  if (r != ED_OK) return r;
  const int wide = a.ld % RowElem<E>::kWide == 0;
  hv_rows_kernel<E, R, T, MB, kLz><<<grid, T, smem, s>>>(a, x, y, lz, wide);
  ED_TRY_CUDA(cudaGetLastError());
  if (grid_out) *grid_out = grid;
  return ED_OK;
}

// Whether this kernel takes the basis. Its rows fit in shared memory twice, and they are long enough
// to occupy a CTA: a row of 120 columns is four warps' work in the down part and one in the up part
// of 12, while the row-staged kernel (ed_hv.cu, ed_hvc.cu) keeps eight small CTAs of two rows on an SM.
// The lines, with both kernels' times of one ed_hv call (row-staged / this kernel, us) on either side:
//  * FP32: 12,870 rows x 120 columns 23 / 50, 6,435 x 455 37 / 45, 1,001 x 2,002 31 / 35; but 8,008 x
//    560 54 / 46, 12,870 x 1,820 265 / 181. Rows of a multiple of 4 columns (16-byte loads) from 500 on,
//    others from 1,200 on where rows come in pairs (launch_hv_rows) or from 5,000 on. With few rows
//    (four CTAs per SM or fewer) the down part's length counts: 120 x 252 5.0 / 4.5, 462 x 330 8.8 / 5.6.
//  * FP64: 12,870 x 120 65 / 92, 3,003 x 105 17 / 23, 18,564 x 153 120 / 122, 495 x 220 7.4 / 8.9;
//    1,716 x 286 28 / 22. With few rows 330 x 165 6.1 / 5.5, 165 x 165 5.3 / 4.9, 153 x 153 3.9 / 4.3, 462 x 165 6.5 / 7.4; in the
//    Lanczos-fused form the row-staged kernel takes 2-4% less.
//  * complex FP32: 6,435 x 455 50 / 65, 924 x 495 14.5 / 16, 38,760 x 190 127 / 232; 1,287 x 286 11.3 /
//    10.4, 12,870 x 560 126 / 116. Few rows: 330 x 165 5.1 / 4.4, 455 x 105 4.6 / 4.3, 462 x 165 5.5 / 6.2.
//  * complex FP64: 3,003 x 105 34 / 66, 12,870 x 120 142 / 275 (8,568 x 153 183 / 186 and 462 x 165
//    20 / 15.5 while the row-staged kernel multiplied at every hop); with amplitude classes (fewer multiply-adds, the bound) 12,870 x 120 already 1,090 / 855.
template <typename E>
bool rows_usable(const ed_basis* b, bool lz) {
  const int64_t nd = b->dn.dim, nu = b->up.dim, sms = sm_count();
  if (b->rows.C == 0 || rows_smem<E, 1>(b) + 4096 > (size_t)smem_optin_max()) return false;
  if constexpr (std::is_same<E, float>::value)
    return nd % 4 == 0 ? nd >= 500 || (nd >= 240 && nu <= 4 * sms)
                       : nd >= 5000 || (nd >= 1200 && nu >= 8 * sms) || (nd >= 240 && nu <= 4 * sms);
  else if constexpr (std::is_same<E, double>::value)
    return nd >= 240 || (nd >= 160 && nu <= 3 * sms && !lz);
  else if constexpr (std::is_same<E, float2>::value)
    return nu <= 3 * sms || nd >= 1000 || (nd >= 280 && (nd % 2 == 0 || nu <= 4 * sms));
  else
    return nd >= 160 || nu <= 2 * sms || b->rows.C > 1;
}

template <typename E>
ed_status launch_hv_rows(const ed_basis* b, double t, double U, const E* x, E* y, int64_t ld, cudaStream_t s,
                         const LzHvArgs* lz, int* grid_out) {
  const HvRows& r = b->rows;
  RowsArgs a;
  a.up_bits = b->up.bits;
  a.dn_bits = b->dn.bits;
  a.order = b->up_order;
  a.up = r.up;
  a.ucnt = r.ucnt;
  a.perm = r.perm;
  a.base = r.base;
  a.kc = r.kc;
  a.tab = r.tab;
  a.amp = r.amp;
  a.dim_up = b->up.dim;
  a.ld = ld;
  a.dim_dn = (int)b->dn.dim;
  a.nchunks = r.nchunks;
  a.C = r.C;
  a.maxhops_up = b->up.maxhops;
  a.t = t;
  a.U = U;
  const LzHvArgs none{nullptr, 0, nullptr};
  if constexpr (sizeof(E) == 4) {
    // two rows per CTA share the table reads where two such CTAs fit an SM and there are rows for
    // every SM
    if (2 * rows_smem<E, 2>(b) + 8192 <= (size_t)smem_optin_max() && b->up.dim >= 8 * (int64_t)sm_count())
      return lz ? rows_launch<E, 2, 384, 4, true>(b, a, x, y, s, *lz, grid_out)
                : rows_launch<E, 2, 384, 4, false>(b, a, x, y, s, none, grid_out);
    return lz ? rows_launch<E, 1, 384, 4, true>(b, a, x, y, s, *lz, grid_out)
              : rows_launch<E, 1, 384, 4, false>(b, a, x, y, s, none, grid_out);
  } else if constexpr (sizeof(E) == 8) {
    return lz ? rows_launch<E, 1, 384, 3, true>(b, a, x, y, s, *lz, grid_out)
              : rows_launch<E, 1, 384, 3, false>(b, a, x, y, s, none, grid_out);
  } else {
    return lz ? rows_launch<E, 1, 512, 1, true>(b, a, x, y, s, *lz, grid_out)
              : rows_launch<E, 1, 512, 1, false>(b, a, x, y, s, none, grid_out);
  }
}

#define ROWS_INST(E)                                                                              \
  template bool rows_usable<E>(const ed_basis*, bool);                                            \
  template ed_status launch_hv_rows<E>(const ed_basis*, double, double, const E*, E*, int64_t,    \
                                       cudaStream_t, const LzHvArgs*, int*);
ROWS_INST(float)
ROWS_INST(double)
ROWS_INST(float2)
ROWS_INST(double2)

}  // namespace ed
