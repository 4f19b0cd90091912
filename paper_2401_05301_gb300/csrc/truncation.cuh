// Block reductions and rule T (the tolerances of Sec. II B) on a sorted spectrum, shared by the dense and
// the particle-number-blocked truncation kernels.
#pragma once

#include <cuda_runtime.h>

namespace ptebd {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}

// Sum over the block (blockDim.x a multiple of 32, <= 1024); every thread gets the result.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = (l < nw) ? sh[l] : 0.0;
    t = warp_sum(t);
    if (l == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

// chi' of the K descending values s (shared memory) with ||theta'||^2 = total: chi_w = smallest k with
// sum_{i>k} s_i^2 <= w_cut total, chi_eps = #{s_k^2 > eps_rel total}, chi' = max(1, min(chi_max, chi_w,
// chi_eps, K)); the tail beyond the K values is total - sum s^2.  Writes chi', the kept norm and the
// discarded weight; a non-finite spectrum sets the status and chi' = 1.  The whole block calls it (one
// thread summing and dividing took 0.3 ms for 1024 values); red: 33 doubles.
__device__ __forceinline__ int truncation_rule(const double* s, int K, double total, int chi_max, double w_cut,
                                               double eps_rel, double* red, int* chi_out, double* norm_out,
                                               double* w_out, int* status) {
  double sum = 0.0, eps_n = 0.0, bad_n = 0.0;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const double p = s[i] * s[i];
    if (!isfinite(s[i])) bad_n = 1.0;
    sum += p;
    if (p / total > eps_rel) eps_n += 1.0;
  }
  const double sumK = block_sum(sum, red);
  const int chi_eps = max(1, (int)block_sum(eps_n, red));
  const bool bad = block_sum(bad_n, red) > 0.0 || !(total > 0.0) || !isfinite(total);
  __shared__ int chi_sh;
  if (threadIdx.x == 0) {
    int chi_w = K;
    if (!bad) {
      const double thr = w_cut * total;
      double tail = fmax(0.0, total - sumK);
      for (int k = K; k >= 1; --k) {
        if (tail <= thr) chi_w = k; else break;
        tail += s[k - 1] * s[k - 1];
      }
    }
    chi_sh = bad ? 1 : max(1, min(min(chi_max, chi_w), min(chi_eps, K)));
  }
  __syncthreads();
  const int chi = chi_sh;
  double kept = 0.0, cut = 0.0;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const double p = s[i] * s[i];
    if (i < chi) kept += p;
    else cut += p;
  }
  kept = block_sum(kept, red);
  cut = block_sum(cut, red);
  if (threadIdx.x == 0) {
    *chi_out = chi;
    *norm_out = sqrt(kept);
    *w_out = bad ? 0.0 : (fmax(0.0, total - sumK) + cut) / total;
    if (bad) atomicExch(status, -7);  // TEBD_ERR_NONFINITE
  }
  __syncthreads();
  return chi;
}

}  // namespace ptebd
