// Reductions in a fixed order shared by the Dslash epilogues and the solvers' vector kernels: a thread's running
// sum, its sum over a warp and a block, and sums of per-block partial results.
#pragma once
#include <cuda_runtime.h>

namespace hisq {

// A thread's running sum of terms in the arithmetic precision, kept to FP64 accuracy without FP64 instructions
// where the terms are FP32: GB300's FP64 pipe takes a warp's operation in 16 cycles and is shared by the whole SM,
// so a conversion and an add per term, five more per warp and a division per thread cost a streaming kernel
// microseconds. FP32 terms go into an error-free pair (hi + lo, Knuth's two-sum: about 48 bits). The pair's range is
// FP32's, so a thread's own terms (one to some tens) have to add up to less than 3.4e38; sums over the warp and
// beyond are not bound by it.
template <typename T>
struct SumAcc;
template <>
struct SumAcc<double> {
  double v = 0.0;
  __device__ __forceinline__ void add(double t) { v += t; }
  // the sum over the warp, in every lane
  __device__ __forceinline__ double warp_total() const {
    double s = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
};
template <>
struct SumAcc<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float t) {
    const float s = __fadd_rn(hi, t), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(t, b)));
    hi = s;
  }
  __device__ __forceinline__ double warp_total() const {
    SumAcc<float> a = *this;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h = __shfl_xor_sync(0xffffffffu, a.hi, o), l = __shfl_xor_sync(0xffffffffu, a.lo, o);
      a.add(h);
      a.lo = __fadd_rn(a.lo, l);
    }
    // Beyond FP32's range (or with a non-finite term) the pair has lost the sum, though each lane's own may be
    // finite: once more in FP64. hi is the same in every lane, so the whole warp takes the branch.
    if (!isfinite(a.hi)) {
      double s = isfinite(hi) ? (double)hi + (double)lo : (double)hi;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      return s;
    }
    return (double)a.hi + (double)a.lo;
  }
};

// Sum of every thread's a over the block (blockDim.x a multiple of 32); every lane of warp 0 gets it. smem: 32
// doubles, free again after the caller's next __syncthreads.
template <typename T>
__device__ __forceinline__ double block_sum_acc(const SumAcc<T>& a, double* smem) {
  const double w = a.warp_total();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) smem[warp] = w;
  __syncthreads();
  double s = 0.0;
  if (warp == 0) {
    s = lane < (int)(blockDim.x >> 5) ? smem[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;
}

// Sums of several quantities over the block with one barrier: get(q) is this thread's running sum of quantity q < N;
// put(q, s) is called by one lane with each total. smem: N * 16 doubles (blocks of at most 512 threads).
template <int N, typename Get, typename Put>
__device__ __forceinline__ void block_sums_acc(double* smem, Get get, Put put) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const double w = get(q).warp_total();
    if (lane == 0) smem[q * 16 + warp] = w;
  }
  __syncthreads();
  for (int q = warp; q < N; q += nw) {  // a warp per quantity
    double s = lane < nw ? smem[q * 16 + lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) put(q, s);
  }
}

// Sum of partials[0..n) by the 32 lanes of one warp, in a fixed order: eight independent accumulators
// per lane keep eight L2 loads in flight, then a fixed shuffle tree; every lane gets the total.
__device__ __forceinline__ double warp_sum_partials(const double* partials, int n) {
  const int lane = threadIdx.x & 31;
  double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int i = lane; i < n; i += 8 * 32) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = i + k * 32 < n ? __ldcg(partials + i + k * 32) : 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] += v[k];
  }
  double t = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  return t;
}

}  // namespace hisq
