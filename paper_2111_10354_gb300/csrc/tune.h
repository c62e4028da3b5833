// Launch autotuner: the first launch of a kernel under a given key (kernel, precisions,
// rhs group, epilogue; the context fixes the lattice) times each candidate form and block size
// with CUDA events on the context's stream and keeps the fastest. Only idempotent
// kernels are tuned this way (the Dslash family: out = f(in) with no read of out).
// Inside a stream capture nothing is timed: an untuned key falls back to 256 threads.
#pragma once
#include <stdio.h>

#include "internal.cuh"

namespace hisq {

// Grid cap for grid-stride kernels: two waves of a fully occupied GPU.
inline int max_grid_blocks(const hisq_ctx* ctx, int block) { return ctx->num_sms * (2048 / block) * 2; }
// Room per rhs in reduction-partials buffers (covers the smallest tuned block, 64).
inline size_t partial_stride(const hisq_ctx* ctx) { return (size_t)ctx->num_sms * 64; }

// Milliseconds of one run() (idempotent launches on the context's stream, warmed up by the caller), or below 0 on an
// error. Three runs; where those take less than 60 us in all, twenty, so that the events' own cost and the launch of
// the first one do not decide between small kernels.
template <typename Run>
float time_launches(hisq_ctx* ctx, cudaEvent_t e0, cudaEvent_t e1, Run&& run) {
  for (int reps = 3;; reps = 20) {
    float ms = 0;
    cudaEventRecord(e0, ctx->stream);
    for (int r = 0; r < reps; ++r) run();
    cudaEventRecord(e1, ctx->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return -1.f;
    cudaEventElapsedTime(&ms, e0, e1);
    ms /= (float)reps;
    if (reps == 20 || ms >= 0.02f) return ms;
  }
}

// Times every (kernel form, block size) pair once per key and caches the fastest as form * 10000 + block. func[nv]: the
// forms' kernels (for the block-size limit); run(form, block) launches one. With one form this is a plain block-size
// tuner. The forms are plain pointers because every launch lists them, also of a tuned key, and launches on small
// lattices are bound by the host (std::function objects in a std::vector: 2.9 us of its time a call at 8^4, now 2.7).
template <typename Run>
int tuned_variant(hisq_ctx* ctx, const char* key, const void* const* func, int nv, Run&& run, int* vi_out, int* block_out) {
  auto it = ctx->tune.find(key);
  if (it != ctx->tune.end() && it->second > 0) {
    *vi_out = it->second / 10000;
    *block_out = it->second % 10000;
    return HISQ_OK;
  }
  if (it != ctx->tune.end()) {
    // a choice loaded from a report (stored negated until checked) is kept only if it names an
    // existing form and a block size that form can launch; otherwise the key is tuned again
    const int vi = -it->second / 10000, b = -it->second % 10000;
    cudaFuncAttributes fa;
    if (vi < nv && b >= 32 && b % 32 == 0 &&
        cudaFuncGetAttributes(&fa, func[vi]) == cudaSuccess && b <= fa.maxThreadsPerBlock) {
      it->second = -it->second;
      *vi_out = vi;
      *block_out = b;
      return HISQ_OK;
    }
    cudaGetLastError();
    ctx->tune.erase(it);
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  HISQ_CUDA(cudaStreamIsCapturing(ctx->stream, &cap));
  if (!ctx->autotune || cap != cudaStreamCaptureStatusNone) {
    cudaFuncAttributes fa;
    HISQ_CUDA(cudaFuncGetAttributes(&fa, func[0]));
    const int b = fa.maxThreadsPerBlock >= 256 ? 256 : 128;
    *vi_out = 0;
    *block_out = b;
    if (cap == cudaStreamCaptureStatusNone) ctx->tune[key] = b;
    return HISQ_OK;
  }
  // powers of two and the sizes between them: on small lattices a block size that spreads the
  // blocks evenly over the SMs matters
  static const int cands[] = {64, 96, 128, 160, 192, 224, 256, 384, 512};
  cudaEvent_t e0, e1;
  HISQ_CUDA(cudaEventCreate(&e0));
  HISQ_CUDA(cudaEventCreate(&e1));
  float best = 1e30f;
  int best_v = 0, best_b = 128;
  for (int i = 0; i < nv; ++i) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, func[i]) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    for (int b : cands) {
      if (b > fa.maxThreadsPerBlock) continue;
      cudaError_t err = run(i, b);  // warm-up
      if (err != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      note_launch(ctx);
      const float ms = time_launches(ctx, e0, e1, [&] {
        run(i, b);
        note_launch(ctx);
      });
      if (ms < 0.f) break;
      if (ms < best) {
        best = ms;
        best_v = i;
        best_b = b;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  HISQ_CUDA(cudaGetLastError());
  ctx->tune[key] = best_v * 10000 + best_b;
  *vi_out = best_v;
  *block_out = best_b;
  return HISQ_OK;
}

// The fastest of n ways to make a call, each timed once per key (run(way) makes it and returns a status; its own launches
// are tuned by its first run); kept as way + 1. Not timed inside a capture or with the tuner off: the first way.
template <typename Run>
int tuned_way(hisq_ctx* ctx, const char* key, const int* ways, int n, Run&& run, int* way) {
  *way = ways[0];
  auto it = ctx->tune.find(key);
  if (it != ctx->tune.end()) {
    const int v = it->second < 0 ? -it->second : it->second;  // negative: loaded from a report, unchecked
    for (int i = 0; i < n; ++i)
      if (ways[i] + 1 == v) {
        it->second = v;
        *way = ways[i];
        return HISQ_OK;
      }
    ctx->tune.erase(it);
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  HISQ_CUDA(cudaStreamIsCapturing(ctx->stream, &cap));
  if (!ctx->autotune || cap != cudaStreamCaptureStatusNone) return HISQ_OK;
  cudaEvent_t e0, e1;
  HISQ_CUDA(cudaEventCreate(&e0));
  HISQ_CUDA(cudaEventCreate(&e1));
  float best = 1e30f;
  int rc = HISQ_OK;
  for (int i = 0; i < n && rc == HISQ_OK; ++i) {
    if ((rc = run(ways[i])) != HISQ_OK) break;
    const float ms = time_launches(ctx, e0, e1, [&] {
      const int r = run(ways[i]);
      if (r != HISQ_OK) rc = r;
    });
    if (ms >= 0.f && ms < best) {
      best = ms;
      *way = ways[i];
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != HISQ_OK) return rc;
  HISQ_CUDA(cudaGetLastError());
  ctx->tune[key] = *way + 1;
  return HISQ_OK;
}

}  // namespace hisq
