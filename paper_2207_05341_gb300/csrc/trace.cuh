// Tr X of the computed X, and the likelihood's constant that goes with it (povm.cu, povm_fast.cu, povm_pauli.cu).
#pragma once

#include "impl.h"

namespace qst {

// One CTA of 256 threads: scal[0] = sum_i Re X_ii (a fixed-order FP64 sum), and the constant sum f / Tr X of
// dL/dq in both precisions (kConst64, kConst32), so that the likelihood passes divide once and not per thread.
template <class R> __device__ __forceinline__ void block_trace(const cx_t<R>* __restrict__ X, int d, double* scal) {
  __shared__ double red[8];
  // every diagonal load of a thread is issued before the first add (one memory latency, not d / 256)
  constexpr int kPer = 16;  // d <= 4096 = 16 x 256
  R v[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int i = threadIdx.x + k * 256;
    v[k] = i < d ? X[(long long)i * d + i].x : R(0);
  }
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (threadIdx.x + k * 256 < d) acc += (double)v[k];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    const double c = scal[1] / t;
    scal[0] = t;
    scal[kConst64] = c;
    *reinterpret_cast<float*>(scal + kConst32) = (float)c;
  }
}

template <class R> __device__ __forceinline__ R likelihood_const(const double* scal);
template <> __device__ __forceinline__ double likelihood_const<double>(const double* scal) { return scal[kConst64]; }
template <> __device__ __forceinline__ float likelihood_const<float>(const double* scal) {
  return *reinterpret_cast<const float*>(scal + kConst32);
}

}  // namespace qst
