#pragma once
// Lanczos-fused H.v for rows longer than shared memory (split rows): the same product and
// epilogue as hv2_kernel (Sec. 4, Eqs. 5-6; w = s_cur H B_cur - b_j s_prev B_prev written
// over B_prev, per-CTA partial sums of w . f_j), for bases whose down row (dim_dn elements)
// does not fit in one CTA's shared memory, e.g. the FP64-accurate 18-site 9/9 basis (389 KB
// rows of int64).
//
// The down states are cut in two slices by the occupation of one site (SplitTables): a hop
// changes that occupation only when it moves a particle onto or off the site, so most down
// hops stay inside their slice. One CTA owns one up row and processes it slice by slice. A
// slice is laid out and staged exactly like a whole row of hv2_kernel (R = 1): column order
// by hop count, slot map (p & ~(G-1)) | lo[p] against bank conflicts, zero slots ld_s ..
// ld_s + G - 1, per-lane hop order chosen by the host. The in-slice down hops gather from
// shared memory; the few cross-slice ones have table rows of their own and read the row in
// global memory (it is L2-resident while the CTA works on it); the up part streams the
// neighbour rows' columns of the slice; the epilogue is hv2_kernel's.
#include "ed_hv2_kernel.cuh"

namespace ed {

struct Hv2sArgs {
  const uint32_t* __restrict__ up_bits;
  const uint32_t* __restrict__ dn_bits;  // by column, padded (pads 0)
  const uint16_t* __restrict__ dtab;     // [rows][ld]: slot of the target inside the slice
  const uint16_t* __restrict__ xtab;     // [xrows][ld]: target column inside the other slice
  const uchar4* __restrict__ kpn;        // per chunk of 32 V columns: in +, in -, cross +, cross -
  const uint8_t* __restrict__ slot_lo;   // [ld] slot of column p within its group of G
  const int32_t* __restrict__ hop_up;    // basis table [maxhops_up][dim_up]
  const int32_t* __restrict__ order;     // up-row visit order (NULL = rank order)
  int64_t dim_up;
  int ld, maxhops_up, nslots;            // nslots: longest slice + G
  int cstart0, cstart1, cstart2;         // slices [cstart0, cstart1), [cstart1, cstart2)
  float t, U;                            // FP32 variant
};

template <typename E, int V, int T, int MB>
__global__ void __launch_bounds__(T, MB)
hv2s_kernel(Hv2sArgs a, const E* __restrict__ x, E* __restrict__ y,
            LzScalars* S, int cur, void* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int npos_s, nneg_s;
  __shared__ double red[33];
  if (S->status != 0) return;
  const int ld = a.ld;
  constexpr int G = hv2_group<E, 1>();
  E* xs = reinterpret_cast<E*>(smem);
  int64_t* upoff = reinterpret_cast<int64_t*>(smem + ((size_t)a.nslots * sizeof(E) + 15) / 16 * 16);
  float sc = 1.f, bsp = 0.f;
  long long ca = 0, cb = 0, cc = 0;
  int ck = 0;
  if constexpr (sizeof(E) == 4) {
    const int j = S->j + 1;
    sc = (float)S->scale[cur];
    bsp = (float)(S->beta[j] * S->scale[1 - cur]);
  } else {
    ca = S->fx_a;
    cb = S->fx_b;
    cc = S->fx_c;
    ck = S->fx_k;
  }
  DotAcc<float> dotf;
  A192 dota;
  // One CTA per row: its reduction is 1% of its 100-180 us, and as the hardware starts CTAs in order
  // the rows in flight stay neighbours, whose rows L2 then holds. One resident wave over every
  // grid-th row (hv2_kernel's form) took 24.3 instead of 20.6 ms on the 18-site 9/9 basis in FP32 and
  // 64.0 instead of 55.7 ms in int64; with the rows handed out by a counter 22.4 and 59.1 ms.
  const int g = blockIdx.x;
  const int64_t u = a.order ? (int64_t)a.order[g] : g;
  if (threadIdx.x < 32)
    hv2_up_list(a.hop_up, a.maxhops_up, a.dim_up, u, ld, upoff, &npos_s, &nneg_s);
  __syncthreads();
  const int npos = npos_s, nneg = nneg_s;
  const uint32_t ub = a.up_bits[u];
  const E* xrow = x + u * ld;
  for (int s = 0; s < 2; ++s) {
    const int c0 = s ? a.cstart1 : a.cstart0, c1 = s ? a.cstart2 : a.cstart1;
    const int oth = s ? a.cstart0 : a.cstart1;  // start of the other slice
    const int lds = c1 - c0;
    // ---- stage the slice through its slot map (the previous slice's gathers are done);
    // slots lds .. lds + G - 1 are zero, one in each bank group
    __syncthreads();
    for (int i = threadIdx.x; i < lds + G; i += T)
      xs[i < lds ? (i & ~(G - 1)) | a.slot_lo[c0 + i] : i] = i < lds ? xrow[c0 + i] : E(0);
    __syncthreads();
    for (int d0 = c0 + threadIdx.x * V; d0 < c1; d0 += T * V) {
      E acc[V];
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = E(0);
      // ---- down part: in-slice hops from shared memory, +1 rows first
      const uchar4 kpn = a.kpn[d0 / (32 * V)];
      const uint16_t* tp = a.dtab + d0;
      for (int k = 0; k < kpn.x; ++k) {
        const Pack<uint16_t, V> e = *reinterpret_cast<const Pack<uint16_t, V>*>(tp + (size_t)k * ld);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] += xs[e.v[v]];
      }
      for (int k = kpn.x; k < kpn.x + kpn.y; ++k) {
        const Pack<uint16_t, V> e = *reinterpret_cast<const Pack<uint16_t, V>*>(tp + (size_t)k * ld);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] -= xs[e.v[v]];
      }
      // ---- cross-slice hops from the row in global memory
      const E* xo = xrow + oth;
      const uint16_t* xp = a.xtab + d0;
      for (int k = 0; k < kpn.z; ++k) {
        const Pack<uint16_t, V> e = *reinterpret_cast<const Pack<uint16_t, V>*>(xp + (size_t)k * ld);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] += xo[e.v[v]];
      }
      for (int k = kpn.z; k < kpn.z + kpn.w; ++k) {
        const Pack<uint16_t, V> e = *reinterpret_cast<const Pack<uint16_t, V>*>(xp + (size_t)k * ld);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] -= xo[e.v[v]];
      }
      // ---- up part: the slice's columns of the neighbour rows
      const E* xb = x + d0;
#pragma unroll 8
      for (int k = 0; k < npos; ++k) {
        const Pack<E, V> q = *reinterpret_cast<const Pack<E, V>*>(xb + upoff[k]);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] += q.v[v];
      }
#pragma unroll 4
      for (int k = 0; k < nneg; ++k) {
        const Pack<E, V> q = *reinterpret_cast<const Pack<E, V>*>(xb + upoff[npos + k]);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] -= q.v[v];
      }
      // ---- diagonal and the Lanczos epilogue (as hv2_kernel)
      const Pack<uint32_t, V> db = *reinterpret_cast<const Pack<uint32_t, V>*>(a.dn_bits + d0);
      E* yp = y + u * ld + d0;
      const Pack<E, V> P = ldcs_pack(reinterpret_cast<const Pack<E, V>*>(yp));
      const Pack<uint8_t, V> lo = *reinterpret_cast<const Pack<uint8_t, V>*>(a.slot_lo + d0);
      Pack<E, V> W;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const E xc = xs[((d0 + v - c0) & ~(G - 1)) | lo.v[v]];
        const int n = __popc(ub & db.v[v]);
        if constexpr (sizeof(E) == 4) {
          const float hx = fmaf(-a.t, (float)acc[v], a.U * (float)n * (float)xc);
          const float w = fmaf(sc, hx, -bsp * (float)P.v[v]);
          W.v[v] = (E)w;
          dotf.add(w, sc * (float)xc);
        } else {
          const long long xi = (long long)xc;
          const W128 p = add128(add128(smul128(ca, (long long)acc[v]), smul128(cb, xi * n)),
                                smul128(cc, (long long)P.v[v]));
          const long long w = round_shift128(p, ck);
          W.v[v] = (E)w;
          a192_add_prod(dota, w, xi);
        }
      }
      stcs_pack(reinterpret_cast<Pack<E, V>*>(yp), W);
    }
  }
  if constexpr (sizeof(E) == 4) {
    const double v = block_sum(dotf.get(), red);
    if (threadIdx.x == 0) reinterpret_cast<double*>(partial)[blockIdx.x] = v;
  } else {
    fx_hv_end(S, cur, dota.w0, dota.w1, dota.w2, reinterpret_cast<long long*>(partial), 0);
  }
}

}  // namespace ed
