// Learned Lanczos start vector: a small network over the occupation bits of a basis state
// (and U) predicts the ground-state amplitude; its predictions over the whole basis become
// f_1 of Algorithm 1 (Sec. 2.2). The paper has no learned component.
//
//   x = (up bits, down bits, bf16(U/8)) in R^(2L+1); h1 = tanh(W1^T x + b1);
//   h2 = tanh(W2^T bf16(h1) + b2);
//   (a, z) = W3^T h2 + b3; psi0 = sign(z) exp(a).       64 hidden units per layer.
// Weights: FP32 master copy (Adam, Kingma & Ba 2015), rounded to bfloat16 (nearest even)
// for every forward pass; FP32 accumulation. The U feature and the first layer's output
// enter the next product rounded to bfloat16 (the operands of the tensor-core products of
// the inference kernel); the backward pass treats these roundings as the identity.
// Inference evaluates tanh with the special-function unit's approximation (PTX
// tanh.approx.f32, maximum relative error about 2^-11: one instruction instead of the ~19 of
// an accurate tanhf, which made the inference issue-bound); training uses tanhf. The
// predicted vector only starts Algorithm 1, so an error of that size in the activations
// changes nothing the method relies on.
// Training: samples drawn uniformly from the basis with weight dim * psi^2; loss per sample
// (a - log|psi|)^2 + log(1 + exp(-sign(psi) z)); deterministic per-CTA gradient partials
// reduced in a fixed order.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "ed_internal.cuh"
#include "ed_tcgen05.cuh"

namespace ed {

constexpr int kH = 64;         // hidden units
constexpr int kTile = 64;      // samples per tile in the training kernel
constexpr int kMThreads = 256;

struct MlpDims {
  int L, nin;
  int oW1, ob1, oW2, ob2, oW3, ob3, P;
};

__host__ __device__ inline MlpDims mlp_dims(int L) {
  MlpDims d;
  d.L = L;
  d.nin = 2 * L + 1;
  d.oW1 = 0;
  d.ob1 = d.oW1 + d.nin * kH;
  d.oW2 = d.ob1 + kH;
  d.ob2 = d.oW2 + kH * kH;
  d.oW3 = d.ob2 + kH;
  d.ob3 = d.oW3 + kH * 2;
  d.P = d.ob3 + 2;
  return d;
}

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// tanh on the special-function unit (PTX tanh.approx.f32, sm_75 and later)
__device__ __forceinline__ float tanh_sfu(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Two FP32 additions / multiply-adds in one instruction (PTX f32x2, sm_100 and later); each half is
// rounded as by fadd / fmaf.
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
      "fma.rn.f32x2 x, x, y, z;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// ------------------------------------------------------------------ inference
// 5th-generation tensor cores: a CTA of 4 warps evaluates tiles of 128 basis states, one
// state per thread (TMEM lane). The features of the tile (bits as 0/1, bf16(U/8), zero
// padding to K1 = 16 ceil(nin/16)) and later bf16(h1) are written to shared memory in the
// K-major core-matrix layout; one thread issues tcgen05.mma (BF16 x BF16 -> FP32 in TMEM
// columns 0..63: D1 = X W1, then D2 = bf16(h1) W2 over it, once every thread has read D1)
// and commits to an mbarrier; every thread then reads its row of the accumulator with
// tcgen05.ld and applies
// bias (CUDA cores) and tanh (special-function unit); the 64 -> 2 output layer stays on the
// CUDA cores. 128 tanh per state on the special-function unit (16 per cycle and SM) are 0.31 ms for
// 11.8 M states; the other instructions have to fit beside them: features come from a table
// of four-bit groups (8 bytes of operand per load; a table of bytes took 4 KB of every CTA, and with
// it a resident CTA from 16 sites on: 16 sites 834 -> 810 us for 19 M states, 32 sites 1,279 -> 1,167
// for 25 M, 14 sites 505 -> 503 for 11.8 M), additions and the output layer go two at a time, states are
// carried from tile to tile without a division.
// Waits on the mbarrier are bounded (1 s of the global timer); on expiry the kernel sets
// *err, frees its TMEM and returns.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

constexpr int kTcRows = 128;      // states per tile = threads per CTA = TMEM lanes used
constexpr uint32_t kTcCols = 64;   // TMEM columns of D1, then of D2
// At most 8 CTAs per SM (8 x 64 = all 512 TMEM columns, so no allocation ever waits): with
// 1 KB reserved per CTA, 9 x (25 KB + 1 KB) exceeds the SM's 228 KB. The register bound
// (launch bounds) makes 5 resident; the grid is one wave of them.
constexpr int kTcSmemMin = 25600;
constexpr int kTcCtasPerSm = 5;

struct TcLayout {
  int K1;
  uint32_t a1, a2, b1, b2, par, lut, mbar, tslot, total;
};

__host__ __device__ inline TcLayout tc_layout(int nin) {
  auto up = [](uint32_t v, uint32_t a) { return (v + a - 1) / a * a; };
  TcLayout t;
  t.K1 = (nin + 15) / 16 * 16;
  t.a1 = 0;
  t.a2 = up(t.a1 + (uint32_t)kTcRows * t.K1 * 2, 1024);
  t.b1 = up(t.a2 + (uint32_t)kTcRows * kH * 2, 1024);
  t.b2 = up(t.b1 + (uint32_t)kH * t.K1 * 2, 1024);
  t.par = up(t.b2 + (uint32_t)kH * kH * 2, 1024);
  t.lut = up(t.par + (uint32_t)(4 * kH + 2) * 4, 16);
  t.mbar = t.lut + 16 * 8;
  t.tslot = t.mbar + 8;
  t.total = up(t.tslot + 8, 1024);
  return t;
}

template <typename T>
__global__ void __launch_bounds__(kTcRows, kTcCtasPerSm)
mlp_infer_tc_kernel(const float* __restrict__ params, int L, float U, const uint32_t* __restrict__ upb,
                    const uint32_t* __restrict__ dnb, int64_t dim_dn, int64_t dim, T* __restrict__ out,
                    int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  const MlpDims d = mlp_dims(L);
  const TcLayout ly = tc_layout(d.nin);
  const int K1 = ly.K1;
  unsigned char* A1 = tsm + ly.a1;
  unsigned char* A2 = tsm + ly.a2;
  unsigned char* B1 = tsm + ly.b1;
  unsigned char* B2 = tsm + ly.b2;
  float* sb1 = reinterpret_cast<float*>(tsm + ly.par);
  float* sb2 = sb1 + kH;
  float* sW3 = sb2 + kH;
  float* sb3 = sW3 + 2 * kH;
  uint2* lut = reinterpret_cast<uint2*>(tsm + ly.lut);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tsm + ly.tslot);
  const uint32_t mbar = smem_addr(tsm + ly.mbar);
  const int tid = threadIdx.x, warp = tid >> 5;

  // rounded weights: W1, W2 as K-major B operands (row n = output unit), the rest in FP32
  for (int i = tid; i < kH * K1; i += blockDim.x) {
    const int n = i / K1, k = i - n * K1;
    const float w = k < d.nin ? params[d.oW1 + k * kH + n] : 0.f;
    *reinterpret_cast<__nv_bfloat16*>(B1 + cm_offset(n, k, K1)) = __float2bfloat16_rn(w);
  }
  for (int i = tid; i < kH * kH; i += blockDim.x) {
    const int n = i / kH, k = i - n * kH;
    *reinterpret_cast<__nv_bfloat16*>(B2 + cm_offset(n, k, kH)) =
        __float2bfloat16_rn(params[d.oW2 + k * kH + n]);
  }
  for (int i = tid; i < kH; i += blockDim.x) {
    sb1[i] = bf16r(params[d.ob1 + i]);
    sb2[i] = bf16r(params[d.ob2 + i]);
    sW3[2 * i] = bf16r(params[d.oW3 + 2 * i]);
    sW3[2 * i + 1] = bf16r(params[d.oW3 + 2 * i + 1]);
  }
  if (tid < 2) sb3[tid] = bf16r(params[d.ob3 + tid]);
  // the bf16 features (0 or 1) of every four bits: 128 bytes, one to each bank
  if (tid < 16) {
    auto pair = [&](int k) { return ((tid >> k) & 1 ? 0x3F80u : 0u) | ((tid >> (k + 1)) & 1 ? 0x3F800000u : 0u); };
    lut[tid] = make_uint2(pair(0), pair(2));
  }
  if (tid == 0) mbar_init(mbar, 1);
  if (warp == 0) tc_alloc(smem_addr(tslot), kTcCols);
  fence_smem_to_async();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t lanes = (uint32_t)(warp * 32) << 16;  // this warp's TMEM lane quarter
  const uint32_t u8bits = pack_bf16(U * 0.125f, 0.f);  // bf16(U/8) in the low half
  const uint32_t idesc = tc_idesc_bf16_f32(kTcRows, kH);
  const uint32_t a1s = smem_addr(A1), a2s = smem_addr(A2), b1s = smem_addr(B1), b2s = smem_addr(B2);
  const uint32_t sbo1 = (uint32_t)(K1 >> 3) << 7, sbo2 = (uint32_t)(kH >> 3) << 7;
  constexpr unsigned long long kWaitNs = 1000000000ull;
  uint32_t phase = 0;
  bool ok = true;
  const int64_t ntiles = (dim + kTcRows - 1) / kTcRows;
  // this thread's state (up rank, down rank), carried from one tile of the CTA to the next
  const int64_t step = (int64_t)gridDim.x * kTcRows, su = step / dim_dn, sd = step - su * dim_dn;
  int64_t u = ((int64_t)blockIdx.x * kTcRows + tid) / dim_dn;
  int64_t dd = (int64_t)blockIdx.x * kTcRows + tid - u * dim_dn;
  for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, u += su, dd += sd) {
    if (dd >= dim_dn) {
      dd -= dim_dn;
      ++u;
    }
    const int64_t e = tile * kTcRows + tid;
    const bool valid = e < dim;
    uint32_t ub = 0, db = 0;
    if (valid) {
      ub = upb[u];
      db = dnb[dd];
    }
    // the bits of both species in feature order, eight features (16 bytes) from two table entries; the
    // U feature (2 L) comes after them, zeros to K1
    const unsigned long long bits = (unsigned long long)ub | ((unsigned long long)db << L);
    for (int j = 0; j < K1; j += 8) {
      const uint32_t f8 = j < 64 ? (uint32_t)(bits >> j) & 0xFFu : 0u;
      const uint2 lo = lut[f8 & 15u], hi = lut[f8 >> 4];
      uint4 w = make_uint4(lo.x, lo.y, hi.x, hi.y);
      if (j == (2 * L & ~7)) {
        const uint32_t v = u8bits << (16 * (2 * L & 1));
        const int q = (2 * L & 7) >> 1;
        if (q == 0) w.x |= v;
        else if (q == 1) w.y |= v;
        else if (q == 2) w.z |= v;
        else w.w |= v;
      }
      *reinterpret_cast<uint4*>(A1 + cm_offset(tid, j, K1)) = w;
    }
    // ---- layer 1 on the tensor cores
    fence_smem_to_async();
    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after_sync();
      for (int s = 0; s < K1 / 16; ++s)
        tc_mma_f16(tmem, tc_smem_desc(a1s + s * 256, 128, sbo1), tc_smem_desc(b1s + s * 256, 128, sbo1),
                   idesc, s > 0);
      tc_commit(mbar);
    }
    ok = __syncthreads_and(mbar_wait_bounded(mbar, phase, kWaitNs)) != 0;
    phase ^= 1u;
    if (!ok) break;
    tc_fence_after_sync();
    float h[kH];
    tc_ld32(tmem + lanes, h);
    tc_ld32(tmem + lanes + 32, h + 32);
#pragma unroll
    for (int j = 0; j < kH; j += 8) {
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
      {
        const float2 t = add2(make_float2(h[j + 2 * q], h[j + 2 * q + 1]), ld2(sb1 + j + 2 * q));
        w[q] = pack_bf16(tanh_sfu(t.x), tanh_sfu(t.y));
      }
      *reinterpret_cast<uint4*>(A2 + cm_offset(tid, j, kH)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    // ---- layer 2 on the tensor cores
    fence_smem_to_async();
    tc_fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after_sync();
      for (int s = 0; s < kH / 16; ++s)
        tc_mma_f16(tmem, tc_smem_desc(a2s + s * 256, 128, sbo2), tc_smem_desc(b2s + s * 256, 128, sbo2),
                   idesc, s > 0);
      tc_commit(mbar);
    }
    ok = __syncthreads_and(mbar_wait_bounded(mbar, phase, kWaitNs)) != 0;
    phase ^= 1u;
    if (!ok) break;
    tc_fence_after_sync();
    tc_ld32(tmem + lanes, h);
    tc_ld32(tmem + lanes + 32, h + 32);
    // ---- output layer on the CUDA cores
    float2 az = ld2(sb3);
#pragma unroll
    for (int n = 0; n < kH; n += 2) {
      const float2 x = add2(make_float2(h[n], h[n + 1]), ld2(sb2 + n));
      const float t0 = tanh_sfu(x.x), t1 = tanh_sfu(x.y);
      const float4 w = *reinterpret_cast<const float4*>(sW3 + 2 * n);
      az = fma2(make_float2(t0, t0), make_float2(w.x, w.y), az);
      az = fma2(make_float2(t1, t1), make_float2(w.z, w.w), az);
    }
    if (valid) {
      const float v = expf(az.x);
      out[e] = (T)(az.y >= 0.f ? v : -v);
    }
    tc_fence_before_sync();  // this tile's TMEM reads before the next tile's MMAs
  }
  if (!ok && tid == 0) atomicExch(err, 1);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tc_dealloc(tmem, kTcCols);
  }
}

// ------------------------------------------------------------------ loss and gradient
// A CTA takes tiles of kTile samples. Every product of a tile (X W1, bf16(h1) W2, G2 W2^T and the
// two weight gradients) is a 64-wide matrix product out of shared memory in FP32; each of the 256
// threads holds a 4 x 4 block of the result in registers, so that two or four 16-byte loads feed
// 16 or 64 multiply-adds (with one output per thread and two 4-byte loads per multiply-add the
// kernel took 176 us for 16,384 samples of 29 features; 300 M multiply-adds are 8 us at the FP32
// rate). Rows are kLdT floats apart: eight consecutive rows start in eight different bank groups.
// A thread keeps its blocks of the weight gradients over all tiles of its CTA; partial[cta][P] and
// lpart[cta] are then reduced in CTA order.
constexpr int kLdT = 68;  // row stride of the tiles: 64 features (65 of X) and the bank offset

struct GradLayout {
  int W1, W2, small, X, H1, H1B, H2, DO, total;  // in floats
};
__host__ __device__ inline GradLayout grad_layout(int nin) {
  GradLayout g;
  const int n4 = (nin + 3) / 4 * 4;
  g.W1 = 0;                       // [n4][64]
  g.W2 = g.W1 + n4 * kH;          // [64][kLdT]
  g.small = g.W2 + kH * kLdT;     // b1 | b2 | W3 (o, c) | b3
  g.X = g.small + 4 * kH + 4;     // [kTile][kLdT]
  g.H1 = g.X + kTile * kLdT;      // h1, then G1
  g.H1B = g.H1 + kTile * kLdT;    // bf16(h1)
  g.H2 = g.H1B + kTile * kLdT;    // h2, then G2
  g.DO = g.H2 + kTile * kLdT;     // [kTile][2]
  g.total = g.DO + 2 * kTile;
  return g;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float get4(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// acc[q][r] += sum_{k < K} A[(ty + 16 q)][k] B[k][4 tx + r] (K a multiple of 4; rows of A kLdT
// apart, rows of B ldb).
__device__ __forceinline__ void mm_forward(float (&acc)[4][4], const float* A, const float* B, int ldb, int K,
                                           int ty, int tx) {
  for (int k = 0; k < K; k += 4) {
    float4 a[4], b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = ld4(A + (ty + 16 * q) * kLdT + k);
#pragma unroll
    for (int i = 0; i < 4; ++i) b[i] = ld4(B + (k + i) * ldb + 4 * tx);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = fmaf(get4(a[q], i), get4(b[i], r), acc[q][r]);
  }
}

// sum[q][r] += sum_s A[s][4 ty + q] B[s][4 tx + r] over the tile's samples in order. The tile's sum is
// formed by itself: carried on through all tiles of a CTA, a chain of additions grows with the batch
// (55,000 of them at 2^24 samples instead of 64 and one per tile).
__device__ __forceinline__ void mm_outer(float (&sum)[4][4], const float* A, const float* B, int ty, int tx) {
  float acc[4][4] = {};
#pragma unroll 4
  for (int t = 0; t < kTile; ++t) {
    const float4 a = ld4(A + t * kLdT + 4 * ty), b = ld4(B + t * kLdT + 4 * tx);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[q][r] = fmaf(get4(a, q), get4(b, r), acc[q][r]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) sum[q][r] += acc[q][r];
}

__global__ void __launch_bounds__(kMThreads, 2)
mlp_grad_kernel(const float* __restrict__ params, int L, float U, const uint32_t* __restrict__ upb,
                const uint32_t* __restrict__ dnb, int64_t dim_dn, const int64_t* __restrict__ idx,
                const double* __restrict__ target, int64_t n, double wscale,
                float* __restrict__ partial, double* __restrict__ lpart) {
  extern __shared__ __align__(16) float gsm[];
  __shared__ uint32_t ubits[kTile], dbits[kTile];
  __shared__ double lred[kTile];
  const MlpDims d = mlp_dims(L);
  const GradLayout g = grad_layout(d.nin);
  const int n4 = (d.nin + 3) / 4 * 4;
  float* W1 = gsm + g.W1;
  float* W2 = gsm + g.W2;
  float* sb1 = gsm + g.small;
  float* sb2 = sb1 + kH;
  float* W3 = sb2 + kH;
  float* sb3 = W3 + 2 * kH;
  float* X = gsm + g.X;
  float* H1 = gsm + g.H1;
  float* H1B = gsm + g.H1B;
  float* H2 = gsm + g.H2;
  float* DO = gsm + g.DO;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // ---- rounded weights
  for (int i = tid; i < n4 * kH; i += kMThreads) W1[i] = i < d.nin * kH ? bf16r(params[d.oW1 + i]) : 0.f;
  for (int i = tid; i < kH * kH; i += kMThreads) W2[(i / kH) * kLdT + i % kH] = bf16r(params[d.oW2 + i]);
  for (int i = tid; i < kH; i += kMThreads) {
    sb1[i] = bf16r(params[d.ob1 + i]);
    sb2[i] = bf16r(params[d.ob2 + i]);
  }
  for (int i = tid; i < 2 * kH; i += kMThreads) W3[i] = bf16r(params[d.oW3 + i]);
  if (tid < 2) sb3[tid] = bf16r(params[d.ob3 + tid]);
  const float u8b = bf16r(U * 0.125f);
  float gW2[4][4] = {}, gW1[4][4] = {};
  float gW1last = 0.f;  // W1's row 64 (32 sites: the U feature), entry tid < 64
  float gX = 0.f;   // thread t: W3 entry t (t < 128), b1 (t < 192), b2 (t < 256)
  float gB3 = 0.f;  // threads 0 and 1: b3
  double lsum = 0.0;
  const int64_t ntiles = (n + kTile - 1) / kTile;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t s0 = tile * kTile;
    __syncthreads();
    if (tid < kTile) {
      uint32_t ub = 0, db = 0;
      if (s0 + tid < n) {
        const int64_t e = idx[s0 + tid];
        const int64_t u = e / dim_dn;
        ub = upb[u];
        db = dnb[e - u * dim_dn];
      }
      ubits[tid] = ub;
      dbits[tid] = db;
    }
    __syncthreads();
    for (int i = tid; i < kTile * n4; i += kMThreads) {
      const int t = i / n4, f = i - t * n4;
      float v = 0.f;
      if (s0 + t < n) {
        if (f < L) v = (float)((ubits[t] >> f) & 1u);
        else if (f < 2 * L) v = (float)((dbits[t] >> (f - L)) & 1u);
        else if (f == 2 * L) v = u8b;
      }
      X[t * kLdT + f] = v;
    }
    __syncthreads();
    // ---- forward
    {
      float acc[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = sb1[4 * tx + r];
      mm_forward(acc, X, W1, kH, n4, ty, tx);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float4 h, hb;
        h = make_float4(tanhf(acc[q][0]), tanhf(acc[q][1]), tanhf(acc[q][2]), tanhf(acc[q][3]));
        hb = make_float4(bf16r(h.x), bf16r(h.y), bf16r(h.z), bf16r(h.w));
        *reinterpret_cast<float4*>(H1 + (ty + 16 * q) * kLdT + 4 * tx) = h;
        *reinterpret_cast<float4*>(H1B + (ty + 16 * q) * kLdT + 4 * tx) = hb;
      }
    }
    __syncthreads();
    {
      float acc[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = sb2[4 * tx + r];
      mm_forward(acc, H1B, W2, kLdT, kH, ty, tx);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(H2 + (ty + 16 * q) * kLdT + 4 * tx) =
            make_float4(tanhf(acc[q][0]), tanhf(acc[q][1]), tanhf(acc[q][2]), tanhf(acc[q][3]));
    }
    __syncthreads();
    // ---- outputs, loss and d(loss)/d(a, z) per sample
    if (tid < kTile) {
      const int64_t k = s0 + tid;
      float da = 0.f, dz = 0.f;
      if (k < n) {
        float a = sb3[0], z = sb3[1];
        const float* h = H2 + tid * kLdT;
        // (unrolled whole, its 192 loads took the registers of the running gradients to local memory: 780
        // bytes of spills; 16,384 samples 68.6 -> 65.7 us, 2^20 1,474 -> 1,356)
#pragma unroll 16
        for (int o = 0; o < kH; ++o) {
          a = fmaf(h[o], W3[2 * o], a);
          z = fmaf(h[o], W3[2 * o + 1], z);
        }
        const double psi = target[k];
        if (psi != 0.0) {
          const double w = wscale * psi * psi;
          const double l = log(fabs(psi));
          const double sg = psi >= 0.0 ? 1.0 : -1.0;
          const double diff = (double)a - l;
          const double mz = -sg * (double)z;
          const double E = exp(-fabs(mz));  // softplus and its slope from one exponential
          lsum += w * (diff * diff + (mz > 0.0 ? mz : 0.0) + log1p(E));
          da = (float)(w * 2.0 * diff / (double)n);
          dz = (float)(w * (-sg) * (mz >= 0.0 ? 1.0 : E) / (1.0 + E) / (double)n);
        }
      }
      DO[2 * tid] = da;
      DO[2 * tid + 1] = dz;
    }
    __syncthreads();
    // ---- output layer's gradient (reads h2), then G2 over h2
    if (tid < 2 * kH) {  // W3 (o, c)
      const int o = tid >> 1, c = tid & 1;
      float acc = 0.f;
      for (int t = 0; t < kTile; ++t) acc = fmaf(H2[t * kLdT + o], DO[2 * t + c], acc);
      gX += acc;
    }
    if (tid < 2) {
      float acc = 0.f;
      for (int t = 0; t < kTile; ++t) acc += DO[2 * t + tid];
      gB3 += acc;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = ty + 16 * q;
      const float da = DO[2 * t], dz = DO[2 * t + 1];
      float4* p = reinterpret_cast<float4*>(H2 + t * kLdT + 4 * tx);
      const float4 h = *p, wa = ld4(W3 + 8 * tx), wb = ld4(W3 + 8 * tx + 4);
      *p = make_float4(fmaf(da, wa.x, dz * wa.y) * (1.f - h.x * h.x), fmaf(da, wa.z, dz * wa.w) * (1.f - h.y * h.y),
                       fmaf(da, wb.x, dz * wb.y) * (1.f - h.z * h.z), fmaf(da, wb.z, dz * wb.w) * (1.f - h.w * h.w));
    }
    __syncthreads();
    // ---- G1 = (G2 W2^T) (1 - h1^2), over h1: rows ty + 16 q, hidden units tx + 16 r
    {
      float acc[4][4] = {};
      for (int o = 0; o < kH; o += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = ld4(H2 + (ty + 16 * q) * kLdT + o);
#pragma unroll
        for (int r = 0; r < 4; ++r) b[r] = ld4(W2 + (tx + 16 * r) * kLdT + o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[q][r] = fmaf(get4(a[q], i), get4(b[r], i), acc[q][r]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float* p = H1 + (ty + 16 * q) * kLdT + tx + 16 * r;
          const float h = *p;
          *p = acc[q][r] * (1.f - h * h);
        }
    }
    __syncthreads();
    // ---- weight gradients
    mm_outer(gW2, H1B, H2, ty, tx);
    if (4 * ty < n4) mm_outer(gW1, X, H1, ty, tx);
    if (d.nin > kH && tid < kH) {
      float acc = 0.f;
      for (int t = 0; t < kTile; ++t) acc = fmaf(X[t * kLdT + kH], H1[t * kLdT + tid], acc);
      gW1last += acc;
    }
    if (tid >= 2 * kH) {  // b1, b2
      const float* G = tid < 3 * kH ? H1 + (tid - 2 * kH) : H2 + (tid - 3 * kH);
      float acc = 0.f;
      for (int t = 0; t < kTile; ++t) acc += G[t * kLdT];
      gX += acc;
    }
  }
  float* out = partial + (size_t)blockIdx.x * d.P;
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) out[d.oW2 + (4 * ty + q) * kH + 4 * tx + r] = gW2[q][r];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (4 * ty + q < d.nin)
#pragma unroll
      for (int r = 0; r < 4; ++r) out[d.oW1 + (4 * ty + q) * kH + 4 * tx + r] = gW1[q][r];
  if (d.nin > kH && tid < kH) out[d.oW1 + kH * kH + tid] = gW1last;
  if (tid < 2) out[d.ob3 + tid] = gB3;
  if (tid < 2 * kH) out[d.oW3 + tid] = gX;
  else if (tid < 3 * kH) out[d.ob1 + tid - 2 * kH] = gX;
  else out[d.ob2 + tid - 3 * kH] = gX;
  if (tid < kTile) lred[tid] = lsum;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int i = 0; i < kTile; ++i) t += lred[i];
    lpart[blockIdx.x] = t / (double)n;
  }
}

// Sum of the per-CTA partials in a fixed order, the mean loss, and optionally an Adam step on
// the master weights. A CTA takes 32 parameters, one warp per eighth of the partials (one thread
// per parameter and 152 loads one after the other took 27 us).
__global__ void __launch_bounds__(kMThreads)
mlp_reduce_kernel(const float* __restrict__ partial, int ncta, int P, const double* __restrict__ lpart,
                  float* __restrict__ grad, double* __restrict__ loss, float* __restrict__ params,
                  float* __restrict__ m, float* __restrict__ v, int step, float lr, int do_adam) {
  __shared__ float sum[kMThreads / 32][32];
  __shared__ double red[33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  float g = 0.f;
  if (i < P) {
#pragma unroll 8
    for (int c = w; c < ncta; c += kMThreads / 32) g += partial[(size_t)c * P + i];
  }
  sum[w][lane] = g;
  __syncthreads();
  if (w == 0 && i < P) {
    g = 0.f;
#pragma unroll
    for (int k = 0; k < kMThreads / 32; ++k) g += sum[k][lane];
    grad[i] = g;
    if (do_adam) {
      const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
      const float mi = b1 * m[i] + (1.f - b1) * g;
      const float vi = b2 * v[i] + (1.f - b2) * g * g;
      m[i] = mi;
      v[i] = vi;
      const float mh = mi / (1.f - powf(b1, (float)step));
      const float vh = vi / (1.f - powf(b2, (float)step));
      params[i] -= lr * mh / (sqrtf(vh) + eps);
    }
  }
  if (blockIdx.x == 0) {
    const double s = block_sum_array(lpart, ncta, red);
    if (threadIdx.x == 0) *loss = s;
  }
}

// Uniform sample of batch indices (SplitMix64 counters) and their target amplitudes.
__global__ void mlp_sample_kernel(uint64_t seed, int64_t dim, int64_t n, const double* __restrict__ psi,
                                  int64_t* __restrict__ idx, double* __restrict__ tgt) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = seed + ((uint64_t)k + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    const int64_t g = (int64_t)((unsigned __int128)z * (unsigned long long)dim >> 64);
    idx[k] = g;
    tgt[k] = psi[g];
  }
}

// Glorot-uniform initial weights from SplitMix64 counters; biases zero.
__global__ void mlp_init_kernel(int L, uint64_t seed, float* __restrict__ params) {
  const MlpDims d = mlp_dims(L);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.P; i += gridDim.x * blockDim.x) {
    int fan_in = 0, fan_out = 0;
    if (i < d.ob1) fan_in = d.nin, fan_out = kH;
    else if (i >= d.oW2 && i < d.ob2) fan_in = kH, fan_out = kH;
    else if (i >= d.oW3 && i < d.ob3) fan_in = kH, fan_out = 2;
    float v = 0.f;
    if (fan_in) {
      uint64_t z = seed + ((uint64_t)i + 1ull) * 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z = z ^ (z >> 31);
      const double u = 2.0 * ((double)(z >> 11) * 0x1.0p-53) - 1.0;
      v = (float)(u * sqrt(6.0 / (fan_in + fan_out)));
    }
    params[i] = v;
  }
}

}  // namespace ed

using namespace ed;

struct ed_mlp {
  int device = 0;
  cudaStream_t stream = nullptr;
  int L = 0;
  MlpDims d{};
  float* params = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  float* grad = nullptr;
  float* partial = nullptr;
  double* lpart = nullptr;
  double* loss = nullptr;
  int64_t* idx = nullptr;
  double* tgt = nullptr;
  int64_t cap = 0;  // batch capacity of idx / tgt
  int ncta = 0;
  int step = 0;
  int* err = nullptr;  // timeout flag of the inference kernel
};

namespace {
ed_status mlp_grad(ed_mlp* M, const ed_basis* b, double U, const int64_t* idx, const double* tgt,
                   int64_t n, double wscale, int adam, float lr) {
  cudaStream_t s = M->stream;
  const size_t sm = (size_t)grad_layout(M->d.nin).total * sizeof(float);
  ED_TRY_CUDA(allow_max_smem(mlp_grad_kernel));
  const int ncta = (int)std::min<int64_t>((n + kTile - 1) / kTile, M->ncta);
  mlp_grad_kernel<<<ncta, kMThreads, sm, s>>>(M->params, M->L, (float)U, b->user_up().bits,
                                                  b->user_dn().bits, b->user_dn().dim, idx, tgt, n,
                                                  wscale, M->partial, M->lpart);
  if (adam) ++M->step;
  mlp_reduce_kernel<<<(M->d.P + 31) / 32, kMThreads, 0, s>>>(
      M->partial, ncta, M->d.P, M->lpart, M->grad, M->loss, M->params, M->m,
      M->v, M->step, lr, adam);
  ED_TRY_CUDA(cudaGetLastError());
  return ED_OK;
}
}  // namespace

extern "C" void ed_mlp_destroy(ed_mlp* M) {
  if (!M) return;
  int prev = 0;
  cudaGetDevice(&prev);
  if (prev != M->device) cudaSetDevice(M->device);
  if (M->stream) cudaStreamSynchronize(M->stream);
  float* fs[] = {M->params, M->m, M->v, M->grad, M->partial};
  for (float* f : fs)
    if (f) cudaFree(f);
  if (M->lpart) cudaFree(M->lpart);
  if (M->loss) cudaFree(M->loss);
  if (M->idx) cudaFree(M->idx);
  if (M->tgt) cudaFree(M->tgt);
  if (M->err) cudaFree(M->err);
  if (prev != M->device) cudaSetDevice(prev);
  delete M;
}

extern "C" ed_status ed_mlp_create(int32_t n_sites, uint64_t seed, void* stream, ed_mlp** out) {
  clear_error();
  ED_CHECK_ARG(out != nullptr, "ed_mlp_create: out is NULL");
  *out = nullptr;
  ED_CHECK_ARG(n_sites >= 1 && n_sites <= kMaxSites, "ed_mlp_create: n_sites outside [1, 32]");
  ed_mlp* M = new ed_mlp();
  cudaGetDevice(&M->device);
  M->stream = (cudaStream_t)stream;
  M->L = n_sites;
  M->d = mlp_dims(n_sites);
  M->ncta = 2 * sm_count();  // CTAs of the gradient kernel: two per SM
  const size_t P = M->d.P;
  bool ok = cudaMalloc((void**)&M->params, P * 4) == cudaSuccess &&
            cudaMalloc((void**)&M->m, P * 4) == cudaSuccess &&
            cudaMalloc((void**)&M->v, P * 4) == cudaSuccess &&
            cudaMalloc((void**)&M->grad, P * 4) == cudaSuccess &&
            cudaMalloc((void**)&M->partial, (size_t)M->ncta * P * 4) == cudaSuccess &&
            cudaMalloc((void**)&M->lpart, (size_t)M->ncta * 8) == cudaSuccess &&
            cudaMalloc((void**)&M->loss, 8) == cudaSuccess &&
            cudaMalloc((void**)&M->err, sizeof(int)) == cudaSuccess;
  if (!ok) {
    ed_mlp_destroy(M);
    set_error("ed_mlp_create: out of device memory");
    return ED_ERR_OOM;
  }
  mlp_init_kernel<<<(int)((P + 255) / 256), 256, 0, M->stream>>>(n_sites, seed, M->params);
  cudaMemsetAsync(M->m, 0, P * 4, M->stream);
  cudaMemsetAsync(M->v, 0, P * 4, M->stream);
  if (cudaGetLastError() != cudaSuccess) {
    ed_mlp_destroy(M);
    set_error("ed_mlp_create: initialisation failed");
    return ED_ERR_CUDA;
  }
  *out = M;
  return ED_OK;
}

extern "C" ed_status ed_mlp_params(ed_mlp* M, float** params, int64_t* count) {
  clear_error();
  ED_CHECK_ARG(M != nullptr, "ed_mlp_params: NULL handle");
  if (params) *params = M->params;
  if (count) *count = M->d.P;
  return ED_OK;
}

extern "C" ed_status ed_mlp_loss_grad(ed_mlp* M, const ed_basis* b, double U, const int64_t* idx,
                                      const double* target, int64_t n, double weight_scale,
                                      double* loss, const float** grad) {
  clear_error();
  ED_CHECK_ARG(M && b && idx && target && n >= 1, "ed_mlp_loss_grad: bad arguments");
  ED_CHECK_ARG(b->n_sites == M->L, "ed_mlp_loss_grad: basis has %d sites, network %d", b->n_sites, M->L);
  ed_status r = mlp_grad(M, b, U, idx, target, n, weight_scale, 0, 0.f);
  if (r != ED_OK) return r;
  if (loss) {
    ED_TRY_CUDA(cudaMemcpyAsync(loss, M->loss, 8, cudaMemcpyDeviceToHost, M->stream));
    ED_TRY_CUDA(cudaStreamSynchronize(M->stream));
  }
  if (grad) *grad = M->grad;
  return ED_OK;
}

extern "C" ed_status ed_mlp_train_step(ed_mlp* M, const ed_basis* b, double U, const double* psi,
                                       int64_t batch, double lr, uint64_t seed, double* loss) {
  clear_error();
  ED_CHECK_ARG(M && b && psi && batch >= 1 && batch <= (1LL << 24), "ed_mlp_train_step: bad arguments");
  ED_CHECK_ARG(b->n_sites == M->L, "ed_mlp_train_step: basis has %d sites, network %d", b->n_sites, M->L);
  if (batch > M->cap) {
    if (M->idx) cudaFree(M->idx);
    if (M->tgt) cudaFree(M->tgt);
    M->idx = nullptr;
    M->tgt = nullptr;
    M->cap = 0;
    ED_TRY_CUDA(cudaMalloc((void**)&M->idx, batch * 8));
    ED_TRY_CUDA(cudaMalloc((void**)&M->tgt, batch * 8));
    M->cap = batch;
  }
  mlp_sample_kernel<<<sm_count() * 4, 256, 0, M->stream>>>(seed, b->dim, batch, psi, M->idx, M->tgt);
  ED_TRY_CUDA(cudaGetLastError());
  ed_status r = mlp_grad(M, b, U, M->idx, M->tgt, batch, (double)b->dim, 1, (float)lr);
  if (r != ED_OK) return r;
  if (loss) {
    ED_TRY_CUDA(cudaMemcpyAsync(loss, M->loss, 8, cudaMemcpyDeviceToHost, M->stream));
    ED_TRY_CUDA(cudaStreamSynchronize(M->stream));
  }
  return ED_OK;
}

extern "C" ed_status ed_mlp_infer(ed_mlp* M, const ed_basis* b, double U, ed_dtype dtype, void* out) {
  clear_error();
  ED_CHECK_ARG(M && b && out && aligned16(out), "ed_mlp_infer: bad arguments");
  ED_CHECK_ARG(b->n_sites == M->L, "ed_mlp_infer: basis has %d sites, network %d", b->n_sites, M->L);
  const TcLayout ly = tc_layout(M->d.nin);
  const int sm = (int)std::max<uint32_t>(ly.total, (uint32_t)kTcSmemMin);
  const int64_t ntiles = (b->dim + kTcRows - 1) / kTcRows;
  ED_TRY_CUDA(allow_max_smem(mlp_infer_tc_kernel<float>));
  ED_TRY_CUDA(allow_max_smem(mlp_infer_tc_kernel<double>));
  // one wave of resident CTAs: kTcCtasPerSm while the shared memory allows them, else fewer
  int dev = 0, sm_bytes = 0, reserved = 0;
  ED_TRY_CUDA(cudaGetDevice(&dev));
  ED_TRY_CUDA(cudaDeviceGetAttribute(&sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  ED_TRY_CUDA(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  const int per_sm = std::max(1, std::min(kTcCtasPerSm, sm_bytes / (sm + reserved)));
  const int grid = (int)std::min<int64_t>(ntiles, (int64_t)sm_count() * per_sm);
  ED_TRY_CUDA(cudaMemsetAsync(M->err, 0, sizeof(int), M->stream));
  if (dtype == ED_F32) {
    mlp_infer_tc_kernel<float><<<grid, kTcRows, sm, M->stream>>>(
        M->params, M->L, (float)U, b->user_up().bits, b->user_dn().bits, b->user_dn().dim, b->dim,
        (float*)out, M->err);
  } else {
    mlp_infer_tc_kernel<double><<<grid, kTcRows, sm, M->stream>>>(
        M->params, M->L, (float)U, b->user_up().bits, b->user_dn().bits, b->user_dn().dim, b->dim,
        (double*)out, M->err);
  }
  ED_TRY_CUDA(cudaGetLastError());
  int h = 0;
  ED_TRY_CUDA(cudaMemcpyAsync(&h, M->err, sizeof(int), cudaMemcpyDeviceToHost, M->stream));
  ED_TRY_CUDA(cudaStreamSynchronize(M->stream));
  if (h) {
    set_error("ed_mlp_infer: a tensor-core completion wait ran out");
    return ED_ERR_TIMEOUT;
  }
  return ED_OK;
}
