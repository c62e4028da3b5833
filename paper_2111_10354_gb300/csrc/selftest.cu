// Self-tests of device-side building blocks: the failure path of the bounded waits (an mbarrier completion wait of
// the tensor-core kernels and the grid-barrier wait of the fused CG update), exercised without a fault or a hang, and
// the fused CG update's sum over the grid.
#include <string.h>

#include <vector>

#include "internal.cuh"
#include "reduce_warp.cuh"
#include "solver_common.cuh"
#include "tc.cuh"

namespace hisq {

// One block waits on an mbarrier that nothing arrives at, with the same bounded wait the tensor-core
// kernels use for their completion barriers; when the wait gives up, the kernel records it and exits.
__global__ void k_selftest_wait(int* flag, uint32_t limit) {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t addr = tc::smem_addr(&bar);
  if (threadIdx.x == 0) tc::mbar_init(addr, 1);
  __syncthreads();
  const bool completed = tc::mbar_wait(addr, 0, limit);  // phase 0 of a fresh barrier never completes
  if (threadIdx.x == 0) *flag = completed ? 2 : 1;
}

// One block waits at the fused CG update's grid barrier for a generation that nobody advances (the word
// is zero and no block arrives), with the update's own bounded wait; when it gives up, the kernel records it.
__global__ void k_selftest_grid_wait(int* flag, const unsigned* word, long limit) {
  const bool passed = grid_wait64_warp(word, 0u, limit);
  if (threadIdx.x == 0) *flag = passed ? 2 : 1;
}

// The sum of n terms as the fused CG update forms |r|^2: a running sum per thread, the block's share, the grid
// barrier, and every block adding all shares itself. Repeated, with the shares scaled by 1, 2 or 4 in turn, so that a
// block which read an earlier repetition's share would get another total. totals[block]; status: bit 0 a wait ran out,
// bit 1 a repetition differed. Cooperative launch; shares: two sets of gridDim.x.
__global__ void __launch_bounds__(256) k_selftest_sum(const float* terms, size_t n, int repeats, double* shares,
                                                      unsigned* bar, double* totals, int* status) {
  __shared__ double red[32];
  __shared__ int s_ok;
  for (int k = 0; k < repeats; ++k) {
    SumAcc<float> v;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
      v.add(terms[i]);
    const double bs = block_sum_acc(v, red), scale = (double)(1 << k % 3);
    double* set = shares + (size_t)(k & 1) * gridDim.x;
    if (threadIdx.x == 0) set[blockIdx.x] = bs * scale;
    unsigned gen;
    bool last;
    grid_arrive_release(bar, &gen, &last);
    if (threadIdx.x < 32) {
      const bool ok = grid_wait64_warp(bar, gen);
      const double t = warp_sum_partials(set, gridDim.x) / scale;
      if (threadIdx.x == 0) {
        s_ok = ok ? 1 : 0;
        if (!ok) atomicOr(status, 1);
        if (k == 0) totals[blockIdx.x] = t;
        else if (__double_as_longlong(totals[blockIdx.x]) != __double_as_longlong(t)) atomicOr(status, 2);
      }
    }
    __syncthreads();
    if (!s_ok) return;
  }
}

}  // namespace hisq

using namespace hisq;

extern "C" int hisq_selftest_bounded_wait(hisq_ctx* ctx) {
  if (!ctx) return set_error(HISQ_EINVAL, "null context");
  // flags [0] mbarrier wait, [1] grid-barrier wait; then the grid barrier's 64-bit word (8-byte aligned)
  int* d_flag = (int*)workspace(ctx, "selftest_flag", 2 * sizeof(int) + sizeof(unsigned long long));
  if (!d_flag) return set_error(HISQ_ENOMEM, "self-test flag");
  const unsigned* word = reinterpret_cast<const unsigned*>(d_flag + 2);
  HISQ_CUDA(cudaMemsetAsync(d_flag, 0, 2 * sizeof(int) + sizeof(unsigned long long), ctx->stream));
  k_selftest_wait<<<1, 32, 0, ctx->stream>>>(d_flag, 1u << 16);
  k_selftest_grid_wait<<<1, 32, 0, ctx->stream>>>(d_flag + 1, word, 1L << 16);
  HISQ_CUDA(cudaGetLastError());
  note_launch(ctx, 2);
  int flag[2] = {0, 0};
  HISQ_CUDA(cudaMemcpyAsync(flag, d_flag, sizeof flag, cudaMemcpyDeviceToHost, ctx->stream));
  HISQ_CUDA(cudaStreamSynchronize(ctx->stream));
  if (flag[0] == 1 && flag[1] == 1)
    return set_error(HISQ_ETIMEOUT, "self-test: both bounded waits gave up as intended");
  if (flag[0] == 2 || flag[1] == 2) return set_error(HISQ_EINVAL, "self-test: a wait nothing could end completed");
  return set_error(HISQ_ECUDA, "self-test kernels did not run");
}

extern "C" int hisq_selftest_sum(hisq_ctx* ctx, const float* terms, long long n, int repeats, double* total) {
  if (!ctx || !terms || !total || n < 0 || repeats < 1) return set_error(HISQ_EINVAL, "bad argument");
  const int nblk = ctx->num_sms;
  // shares [2][nblk], totals [nblk], the barrier's 64-bit word, the status
  double* d = (double*)workspace(ctx, "selftest_sum", (3 * (size_t)nblk + 2) * sizeof(double));
  if (!d) return set_error(HISQ_ENOMEM, "self-test sum");
  double* totals = d + 2 * (size_t)nblk;
  unsigned* bar = reinterpret_cast<unsigned*>(d + 3 * (size_t)nblk);
  int* status = reinterpret_cast<int*>(d + 3 * (size_t)nblk + 1);
  HISQ_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(double), ctx->stream));
  size_t count = (size_t)n;
  double* shares = d;
  void* args[] = {&terms, &count, &repeats, &shares, &bar, &totals, &status};
  HISQ_CUDA(cudaLaunchCooperativeKernel((const void*)k_selftest_sum, dim3(nblk), dim3(256), args, 0, ctx->stream));
  note_launch(ctx);
  std::vector<double> t(nblk);
  int st = 0;
  HISQ_CUDA(cudaMemcpyAsync(t.data(), totals, nblk * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  HISQ_CUDA(cudaMemcpyAsync(&st, status, sizeof st, cudaMemcpyDeviceToHost, ctx->stream));
  HISQ_CUDA(cudaStreamSynchronize(ctx->stream));
  if (st & 1) return set_error(HISQ_ETIMEOUT, "self-test: a grid-barrier wait ran out");
  for (int i = 1; i < nblk; ++i)
    if (memcmp(&t[i], &t[0], sizeof(double)) != 0) st |= 2;
  if (st & 2) return set_error(HISQ_ECUDA, "self-test: the blocks' sums differ");
  *total = t[0];
  return HISQ_OK;
}
