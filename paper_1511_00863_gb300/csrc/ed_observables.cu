// Double occupancy of a state vector: D_i = <psi| n_i,up n_i,dn |psi> / <psi|psi> (the
// on-site operator of the interaction term added to Sec. 1 Eq. 1) and D = sum_i D_i, which
// equals dE0/dU for a normalised non-degenerate ground state (Hellmann-Feynman).
//
// One pass over psi (FP64, basis order u * dim_dn + d). A warp takes one up state and a run of
// down states at a time, so the sites that can count are the occupied ones of that up state, the
// same for every lane: a lane adds psi^2 to one register per such site when its down state holds
// it. GB300 issues one warp-wide FP64 instruction per 16 cycles and SM, so their number is the
// time: a square, the norm and N_up site sums per element, against a test of all 32 sites of
// every element, which took 840 us on the half-filled 14-site ring (11.8 M states). The lane's
// sums go to shared memory per run; CTAs write partials that one CTA per sum adds in a fixed
// order. D is the sum of the D_i.
#include <cmath>

#include "ed_internal.cuh"

namespace ed {

constexpr int kObsThreads = 256;
constexpr int kObsSums = 33;   // norm^2, 32 sites
constexpr int kObsRun = 2048;  // down states per run at most
constexpr int kObsSites = 8;   // sites per pass over a run (more only above 8 up particles)

__global__ void __launch_bounds__(kObsThreads)
obs_partials_kernel(const double* __restrict__ psi, const uint32_t* __restrict__ up,
                    const uint32_t* __restrict__ dn, int64_t dim_up, int64_t dim_dn, int n_sites,
                    int run, double* __restrict__ part) {
  extern __shared__ double site_sum[];  // [n_sites][kObsThreads]
  __shared__ double red[33];
  for (int i = 0; i < n_sites; ++i) site_sum[i * kObsThreads + threadIdx.x] = 0.0;
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kObsThreads / 32);
  const int64_t runs = (dim_dn + run - 1) / run;
  double nrm = 0.0;
  for (int64_t it = blockIdx.x * (int64_t)(kObsThreads / 32) + (threadIdx.x >> 5); it < dim_up * runs;
       it += warps) {
    const int64_t u = it / runs, d0 = (it - u * runs) * run;
    const int64_t d1 = d0 + run < dim_dn ? d0 + run : dim_dn;
    const double* row = psi + u * dim_dn;
    uint32_t left = up[u];  // occupied sites not summed yet
    bool first = true;
    do {
      uint32_t bit[kObsSites];
      double acc[kObsSites];
#pragma unroll
      for (int k = 0; k < kObsSites; ++k) {
        bit[k] = left & (0u - left);
        left ^= bit[k];
        acc[k] = 0.0;
      }
      for (int64_t d = d0 + lane; d < d1; d += 32) {
        const double v = row[d];
        const uint32_t m = dn[d];
        const double p2 = v * v;
        if (first) nrm += p2;
#pragma unroll
        for (int k = 0; k < kObsSites; ++k)
          if (m & bit[k]) acc[k] += p2;
      }
#pragma unroll
      for (int k = 0; k < kObsSites; ++k)
        if (bit[k]) site_sum[(__ffs(bit[k]) - 1) * kObsThreads + threadIdx.x] += acc[k];
      first = false;
    } while (left);
  }
  const double nr = block_sum(nrm, red);
  if (threadIdx.x == 0) part[(int64_t)blockIdx.x * kObsSums] = nr;
  for (int i = 0; i < n_sites; ++i) {
    const double si = block_sum(site_sum[i * kObsThreads + threadIdx.x], red);
    if (threadIdx.x == 0) part[(int64_t)blockIdx.x * kObsSums + 1 + i] = si;
  }
}

// CTA k: sum k of the partials, in CTA order.
__global__ void __launch_bounds__(kObsThreads)
obs_final_kernel(const double* __restrict__ part, int nparts, double* __restrict__ out) {
  __shared__ double red[33];
  double v = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) v += part[(int64_t)i * kObsSums + blockIdx.x];
  v = block_sum(v, red);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

}  // namespace ed

using namespace ed;

extern "C" ed_status ed_double_occupancy(const ed_basis* b, const double* psi, void* stream,
                                         double* D_total, double* D_site) {
  clear_error();
  ED_CHECK_ARG(b && psi && D_total, "ed_double_occupancy: NULL argument");
  ED_CHECK_ARG(aligned16(psi), "ed_double_occupancy: psi must be 16-byte aligned");
  cudaStream_t s = (cudaStream_t)stream;
  const int nsums = 1 + b->n_sites;
  const int64_t cap = (int64_t)sm_count() * 3;  // 64 KB of shared memory per CTA at most
  // Few rows are cut finer, into runs for four warps of every SM: one row of 12,376 states in runs of
  // 2,048 kept six warps busy, 157 us instead of 54; 91 rows of 3,432 states 122 us, now 66. No finer
  // than two loads per lane, and more rows stay whole: 924 rows of 924 in runs of 256 took 76 us, not 64.
  const int64_t per_row = (4 * (int64_t)sm_count() + b->up.dim - 1) / b->up.dim;
  const int64_t fine = ((b->dn.dim + per_row - 1) / per_row + 31) / 32 * 32;
  const int run = (int)(per_row <= 1 || fine >= kObsRun ? kObsRun : fine < 64 ? 64 : fine);
  const int64_t runs = (b->dn.dim + run - 1) / run;
  int64_t g64 = (b->up.dim * runs + kObsThreads / 32 - 1) / (kObsThreads / 32);
  const int grid = (int)(g64 < 1 ? 1 : (g64 < cap ? g64 : cap));
  double* part = nullptr;
  ED_TRY_CUDA(cudaMallocAsync((void**)&part, ((size_t)grid * kObsSums + kObsSums) * sizeof(double), s));
  double* out = part + (size_t)grid * kObsSums;
  const size_t smem = (size_t)b->n_sites * kObsThreads * sizeof(double);
  cudaError_t e = smem > 32 * 1024 ? allow_max_smem(obs_partials_kernel) : cudaSuccess;
  if (e == cudaSuccess) {
    obs_partials_kernel<<<grid, kObsThreads, smem, s>>>(psi, b->up.bits, b->dn.bits, b->up.dim,
                                                        b->dn.dim, b->n_sites, run, part);
    obs_final_kernel<<<nsums, kObsThreads, 0, s>>>(part, grid, out);
    e = cudaGetLastError();
  }
  double h[kObsSums] = {0.0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, out, nsums * sizeof(double), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(part, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_error("ed_double_occupancy: %s", cudaGetErrorString(e));
    return ED_ERR_CUDA;
  }
  ED_CHECK_ARG(h[0] > 0.0, "ed_double_occupancy: psi is the zero vector");
  double tot = 0.0;
  for (int i = 0; i < b->n_sites; ++i) tot += h[1 + i];
  *D_total = std::isinf(h[0]) ? NAN : tot / h[0];
  if (D_site)
    for (int i = 0; i < b->n_sites; ++i) D_site[i] = h[1 + i] / h[0];
  return ED_OK;
}
