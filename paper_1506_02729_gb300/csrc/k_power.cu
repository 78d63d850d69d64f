// k_power.cu - the fixed-order FP64 reduction of the z-pass's per-block bin
//   sums (Sec. III.A of the paper) and the bounded-wait diagnostic.  Gridding
//   and the scalars are in k_assign.cu, the three FFT passes in k_xpass.cu,
//   k_ypass.cu and k_zpass.cu.
#include <cuda_runtime.h>
#include <stdint.h>

#include "fkp_internal.h"

namespace fkp {

// One block per (quantity, bin): fixed-order FP64 tree sum over the blocks.
// blockIdx.y picks the mock of a fused launch (partials at pstride / pcstride,
// bins and counts at ostride, in 8-byte words).
__global__ void __launch_bounds__(256) k_reduce_bins(const double* __restrict__ part, const int* __restrict__ partc,
                                                     int nblk, int nbins, double* __restrict__ out,
                                                     long long* __restrict__ outc, long long pstride,
                                                     long long pcstride, long long ostride) {
  part += (long long)blockIdx.y * pstride;
  partc += (long long)blockIdx.y * pcstride;
  out += (long long)blockIdx.y * ostride;
  outc += (long long)blockIdx.y * ostride;
  __shared__ double sh[32];
  const int row = blockIdx.x;  // 0 .. BQ_N*nbins (float rows) then nbins (count rows)
  double s = 0.0;
  if (row < BQ_N * nbins) {
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += part[(size_t)row * nblk + b];
    s = block_sum_f64(s, sh);
    if (threadIdx.x == 0) out[row] = s;
  } else {
    const int r = row - BQ_N * nbins;
    long long cs = 0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) cs += partc[(size_t)r * nblk + b];
    s = block_sum_f64((double)cs, sh);
    if (threadIdx.x == 0) outc[r] = (long long)s;
  }
}

// Diagnostic of the bounded wait: one block initialises an mbarrier that
// nothing ever arrives at and no copy targets, then waits on its first phase
// with the passes' bounded wait (mbar_wait_n) for `polls` polls.  flag gets
// 1 when the wait gave up (the expected outcome), 2 if it completed.
__global__ void k_wait_selftest(unsigned polls, int* __restrict__ flag) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && mbar_wait_n(&bar, 0u, flag, 1, polls)) atomicOr(flag, 2);
}

// ----------------------------------------------------------------------------
// host-side launch wrappers (called by the C ABI)
// ----------------------------------------------------------------------------

cudaError_t launch_wait_selftest(unsigned polls, int* flag, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(polls, flag);
  return cudaGetLastError();
}

cudaError_t launch_reduce_bins(const double* part, const int* partc, int nblk, int nbins, double* out, long long* outc,
                               cudaStream_t s, int nmock, long long pstride, long long pcstride, long long ostride) {
  k_reduce_bins<<<dim3((BQ_N + 1) * nbins, nmock), 256, 0, s>>>(part, partc, nblk, nbins, out, outc, pstride,
                                                                pcstride, ostride);
  return cudaGetLastError();
}

}  // namespace fkp
