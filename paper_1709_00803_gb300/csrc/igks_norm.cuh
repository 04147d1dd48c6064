// igks_norm.cuh -- the reduction of the residual norms from partial norms (maxima and sums of
// squares), shared by the iteration and by the entry point that allocates nothing: the same
// values in the same order.
#pragma once

namespace igks {

constexpr int NORM_CELLS = 64;       // cells of one partial norm
constexpr int NORM_THREADS = 256;

// rmax, r2: the maximum of pmax[0..n) (non-negative) and the sum of psum[0..n), in thread 0 of
// a block of NORM_THREADS
__device__ __forceinline__ void norm_reduce(const double* pmax, const double* psum, int n, double* rmax, double* r2) {
  __shared__ double sm[NORM_THREADS / 32], ss[NORM_THREADS / 32];
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x; k < n; k += NORM_THREADS) {
    a = fmax(a, pmax[k]);
    b += psum[k];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) { sm[threadIdx.x >> 5] = a; ss[threadIdx.x >> 5] = b; }
  __syncthreads();
  *rmax = 0.0;
  *r2 = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < NORM_THREADS / 32; w++) { *rmax = fmax(*rmax, sm[w]); *r2 += ss[w]; }
}

}  // namespace igks
