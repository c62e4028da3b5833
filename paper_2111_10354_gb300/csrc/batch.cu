// Batched mixed-precision CG over many independent lattices of uneven sizes.
//
// Every step of the solve is one launch for all lattices: a persistent grid walks the tiles (consecutive output
// sites of one lattice) of the lattices that still iterate, so small and large lattices share the GPU without one
// launch per lattice. Each block lists those lattices when it starts, from flags that no block of the launch changes
// (they are committed by the last block of the grid to finish), so all blocks walk the same tiles; with a table of
// all tiles, blocks spent a launch's last microseconds looking up tiles of finished lattices. Reductions are per
// lattice and deterministic: each block writes its part, and the last block of a lattice's to do so sums them
// in tile order. One CUDA graph, kept for the next solves, holds the reliable_period inner iterations of a
// cycle (FP32 links and spinors, FP32 correction e); the fold x += s e, the FP64 true residual and the reliable
// update follow it, and the host polls once per cycle.
// The Dslash tile (its block size) is chosen by the autotuner.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <chrono>
#include <type_traits>
#include <vector>

#include "dslash_impl.cuh"
#include "solver_common.cuh"
#include "trace.h"
#include "tune.h"

namespace hisq {

bool is_device_ptr(const void* p);
double dslash_bytes(const hisq_ctx* ctx, int lp, int sp, int nrhs);

constexpr int MAXB = 256;  // lattices per batch

struct BatchState {
  double rr[MAXB], rr_new[MAXB], pAp[MAXB], bb[MAXB], tol2[MAXB], scale[MAXB], rr_true[MAXB], a[MAXB];
  double alpha[MAXB], beta[MAXB];           // formed once per lattice (an FP64 division per thread costs microseconds)
  float af[MAXB], alphaf[MAXB], betaf[MAXB];  // a, alpha and beta rounded to FP32
  int done[MAXB];   // frozen for the rest of the cycle (inner tolerance met, or verified)
  int conv[MAXB];   // true FP64 residual verified below tolerance
  int iters[MAXB];  // inner iterations per lattice
  unsigned cnt[6][MAXB];  // per-lattice tile counters, one row per reduction kernel
  unsigned grid_cnt[6];   // per-kernel CTA counters (last CTA does global bookkeeping)
  int nlat, cycle_done, cycle_iter, cycle_limit, breakdown, nonfinite, all_conv, x_nonzero;
};

// First tile of every lattice in a numbering of all tiles of one size (where the tiles' partials go).
struct TileTable {
  int ntiles = 0;
  int* lat_tile0 = nullptr;  // [nlat + 1]
};

struct BatchArgs {
  const Geom* geoms;         // [nlat]
  const char* const* links;  // [nlat] link storage of one precision
  const size_t* blk_bytes;   // [nlat]
  const size_t* site_off;    // [nlat] offset of lattice l's vectors, in sites
  const int* lat_tile0;
  int tile;                  // sites per tile
  int nlat;
};

// ------------------------------------------------------------------ the lattices a launch works on
struct ActiveTiles {
  int n;               // lattices listed
  unsigned nb, q, rem;  // blocks that get tiles in the reducing launches; tiles / nb and tiles % nb
  int lat[MAXB];
  int tile0[MAXB + 1];  // first tile of each in the launch's numbering; [n]: all tiles
};

// Lists the lattices whose skip flag is 0 (every thread of the block calls it).
__device__ __forceinline__ void list_active(ActiveTiles& A, const BatchArgs& a, const int* skip) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int n = 0, tiles = 0;
    for (int l0 = 0; l0 < a.nlat; l0 += 32) {
      const int l = l0 + lane;
      // flag and tile count in flight together
      const int sk = l < a.nlat ? skip[l] : 1, t0 = a.lat_tile0[min(l, a.nlat)], t1 = a.lat_tile0[min(l + 1, a.nlat)];
      const bool on = sk == 0;
      const int cnt = on ? t1 - t0 : 0;
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
      }
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) {
        const int k = n + __popc(m & ((1u << lane) - 1));
        A.lat[k] = l;
        A.tile0[k] = tiles + incl - cnt;
      }
      n += __popc(m);
      tiles += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) {
      A.n = n;
      A.tile0[n] = tiles;
      A.nb = min((unsigned)tiles, gridDim.x);
      A.q = A.nb ? tiles / A.nb : 0;
      A.rem = tiles - A.q * A.nb;
    }
  }
  __syncthreads();
}

// The list number of tile t's lattice (binary search); *local: the tile's number within it.
__device__ __forceinline__ int tile_lattice(const ActiveTiles& A, int t, int* local) {
  int lo = 0, hi = A.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (A.tile0[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  *local = t - A.tile0[lo];
  return lo;
}

// ------------------------------------------------------------------ reduction helpers
// The reducing launches give every block one contiguous range of the launch's tiles, [tile_begin(b), tile_begin(b+1)),
// so that a block reduces once per lattice it meets (mostly one) instead of once per tile. With fewer tiles than
// blocks the first blocks get one each and the others none.
__device__ __forceinline__ int tile_begin(const ActiveTiles& A, unsigned b) {
  return b >= A.nb ? A.tile0[A.n] : (int)(b * A.q + min(b, A.rem));
}
__device__ __forceinline__ int tile_owner(const ActiveTiles& A, int t) {  // the block whose range holds tile t
  const unsigned big = A.rem * (A.q + 1);  // the first rem blocks have a tile more
  return (unsigned)t < big ? (int)((unsigned)t / (A.q + 1)) : (int)(A.rem + ((unsigned)t - big) / A.q);
}

// This block's part of lattice number k (of the list)'s sum -> the total by the CTA that is last to bring its part.
// Returns true in thread 0 of that CTA, with the total in *total.
template <typename T>
__device__ __forceinline__ bool lattice_reduce(const SumAcc<T>& v, const ActiveTiles& A, int k, const BatchArgs& a,
                                               double* partials, unsigned* cnt, double* red, double* total) {
  __shared__ bool last;
  const double s = block_sum_acc(v, red);
  const int l = A.lat[k], p0 = a.lat_tile0[l];
  int n = 0;
  if (threadIdx.x < 32) {  // the blocks that share this lattice
    const int b0 = tile_owner(A, A.tile0[k]);
    n = tile_owner(A, A.tile0[k + 1] - 1) - b0 + 1;
    if (threadIdx.x == 0) {
      partials[p0 + blockIdx.x - b0] = s;
      __threadfence();
      last = atomicAdd(&cnt[l], 1u) == (unsigned)n - 1;
    }
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return false;
  __threadfence();
  *total = warp_sum_partials(partials + p0, n);
  if (threadIdx.x == 0) cnt[l] = 0u;
  return threadIdx.x == 0;
}

// True in every thread of the last CTA of the grid to reach this point.
__device__ __forceinline__ bool grid_last(unsigned* c) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(c, 1u) == gridDim.x - 1;
    if (last) {
      __threadfence();
      *c = 0u;
    }
  }
  __syncthreads();
  return last;
}

// ------------------------------------------------------------------ batched Dslash
// out_l = D in_l (EPI_PLAIN) or out_l = a_l y_l - D in_l with pAp_l = Re<y_l, out_l> and alpha_l = rr_l / pAp_l
// (EPI_AXPY), for every lattice l whose skip[l] is 0. FP32 takes 80 registers (three blocks of 256 per SM): at 64, like
// the single-lattice form, the tile walk spills (16 lattices, all active: 174 and 196 us against 164 and 181 us). NARROW:
// 72 registers in blocks of 128, seven per SM. It spills more and is slower (those 16 lattices 53.0 ms a solve
// against 51.4, six 16^4 20.8 against 18.9), except where its 14% more threads take all sites at once and 80
// registers leave some for a second round (four 16^4: 13.8 against 15.6); FP32 is tuned over both.
template <typename LR, typename SR, int EPI, bool NARROW>
__global__ void __launch_bounds__(NARROW ? 128 : 256, NARROW ? 7 : sizeof(LR) == 4 ? 3 : 0)
    k_bdslash(const BatchArgs a, int p, void* out, const void* in,
                                                                         const void* y, const int* skip, BatchState* st,
                                                                         double* partials, int red_row) {
  using A = typename Real<LR>::acc;
  using SA = typename Real<SR>::acc;
  __shared__ double red[32];
  __shared__ ActiveTiles act;
  list_active(act, a, skip);
  constexpr bool RED = EPI == EPI_AXPY;
  const int t1 = RED ? tile_begin(act, blockIdx.x + 1) : act.tile0[act.n];
  SumAcc<SA> dot;
  for (int t = RED ? tile_begin(act, blockIdx.x) : (int)blockIdx.x; t < t1; t += RED ? 1 : (int)gridDim.x) {
    int local;
    const int kl = tile_lattice(act, t, &local), l = act.lat[kl];
    const Geom g = a.geoms[l];
    const int cb = local * a.tile + threadIdx.x;  // blockDim.x == a.tile
    const size_t base = a.site_off[l];
    if (cb < g.half) {
      cplx<A> acc[1][3];
      const char* in_l = (const char*)in + base * 6 * sizeof(SR);
      dslash_site<LR, SR, 1>(g, a.links[l], a.blk_bytes[l], p, cb, in_l, 0, acc);
      cplx<SA> o[3];
      if (EPI == EPI_PLAIN) {
#pragma unroll
        for (int i = 0; i < 3; ++i) o[i] = {SA(acc[0][i].re), SA(acc[0][i].im)};
      } else {
        cplx<SA> yv[3];
        VecIO<SR>::load(y, base + cb, yv);
        A al;
        if constexpr (std::is_same<A, float>::value) al = st->af[l];
        else al = st->a[l];
        SA tt = SA(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          o[i].re = SA(fma(al, A(yv[i].re), -acc[0][i].re));
          o[i].im = SA(fma(al, A(yv[i].im), -acc[0][i].im));
          tt += yv[i].re * o[i].re + yv[i].im * o[i].im;
        }
        dot.add(tt);
      }
      VecIO<SR>::store(out, base + cb, o);
    }
    if (RED && (t + 1 == t1 || t + 1 == act.tile0[kl + 1])) {  // the block's last tile of this lattice
      double tot;
      if (lattice_reduce(dot, act, kl, a, partials, st->cnt[red_row], red, &tot)) {
        st->pAp[l] = tot;
        const double alpha = tot > 0.0 && isfinite(tot) ? st->rr[l] / tot : 0.0;
        st->alpha[l] = alpha;
        st->alphaf[l] = (float)alpha;
      }
      dot = SumAcc<SA>();
    }
  }
}

// ------------------------------------------------------------------ batched BLAS-1
// Tiles of BLAS_TILE sites, whose 16-byte words (two complex FP32 entries, one FP64) a block of BLAS_BLOCK takes one
// (two) per thread, all loads before the first store. Larger tiles leave SMs idle in small batches.
constexpr int BLAS_TILE = 128, BLAS_BLOCK = BLAS_TILE * 3 / 2;
template <typename S>
struct Word;
template <>
struct Word<float> {
  using V = float4;
  static constexpr int PER_TILE = BLAS_TILE * 3 / 2, J = PER_TILE / BLAS_BLOCK;
  __device__ __forceinline__ static V axpy(float a, V x, V y) {  // a x + y
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
  }
  __device__ __forceinline__ static float norm2(V x) { return (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w); }
};
template <>
struct Word<double> {
  using V = double2;
  static constexpr int PER_TILE = BLAS_TILE * 3, J = PER_TILE / BLAS_BLOCK;
  __device__ __forceinline__ static V axpy(double a, V x, V y) { return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y)); }
  __device__ __forceinline__ static double norm2(V x) { return x.x * x.x + x.y * x.y; }
};

// e_l += alpha_l p_l; r_l -= alpha_l Ap_l; rr_new_l = |r_l|^2, beta_l = rr_new_l / rr_l. S = double: e is the FP64
// solution itself (true units, scale_l); S = float: inner units, k_bfold scales.
template <typename S>
__global__ void __launch_bounds__(BLAS_BLOCK) k_bupdate(const BatchArgs a, S* e, S* r, const S* p, const S* Ap, BatchState* st,
                                                 double* partials) {
  if (st->cycle_done) return;
  using W = Word<S>;
  using V = typename W::V;
  constexpr bool F = std::is_same<S, float>::value;
  __shared__ double red[32];
  __shared__ ActiveTiles act;
  list_active(act, a, st->done);
  const int t1 = tile_begin(act, blockIdx.x + 1);
  SumAcc<S> v;
  for (int t = tile_begin(act, blockIdx.x); t < t1; ++t) {
    int local;
    const int kl = tile_lattice(act, t, &local), l = act.lat[kl];
    const int nw = a.geoms[l].half * (W::PER_TILE / (BLAS_TILE / 2)) / 2;  // words of the lattice
    const size_t off = a.site_off[l] * (W::PER_TILE / (BLAS_TILE / 2)) / 2;
    const int w0 = local * W::PER_TILE + threadIdx.x;
    S al, ax;
    if constexpr (F) {
      al = ax = st->alphaf[l];
    } else {
      al = st->alpha[l];
      ax = al * st->scale[l];
    }
    V rv[W::J], av[W::J], pv[W::J], xv[W::J];
#pragma unroll
    for (int j = 0; j < W::J; ++j) {
      const int w = w0 + j * BLAS_BLOCK;
      if (w < nw) {
        rv[j] = reinterpret_cast<const V*>(r)[off + w];
        av[j] = reinterpret_cast<const V*>(Ap)[off + w];
        pv[j] = reinterpret_cast<const V*>(p)[off + w];
        xv[j] = reinterpret_cast<const V*>(e)[off + w];
      }
    }
#pragma unroll
    for (int j = 0; j < W::J; ++j) {
      const int w = w0 + j * BLAS_BLOCK;
      if (w < nw) {
        rv[j] = W::axpy(-al, av[j], rv[j]);
        reinterpret_cast<V*>(r)[off + w] = rv[j];
        reinterpret_cast<V*>(e)[off + w] = W::axpy(ax, pv[j], xv[j]);
        v.add(W::norm2(rv[j]));
      }
    }
    if (t + 1 != t1 && t + 1 != act.tile0[kl + 1]) continue;
    double tot;
    if (lattice_reduce(v, act, kl, a, partials, st->cnt[1], red, &tot)) {
      st->rr_new[l] = tot;
      const double beta = tot / st->rr[l];
      st->beta[l] = beta;
      st->betaf[l] = (float)beta;
      const double pap = st->pAp[l];
      if (!(pap > 0.0 && isfinite(pap))) st->breakdown = 1;
      if (!isfinite(tot)) st->nonfinite = 1;
    }
    v = SumAcc<S>();
  }
}

// p_l = r_l + beta_l p_l; last CTA of the grid: per lattice commit rr, count the iteration, inner convergence; end
// of cycle when every lattice is frozen or the cycle is full.
template <typename S>
__global__ void __launch_bounds__(BLAS_BLOCK) k_bpupdate(const BatchArgs a, const S* r, S* p, BatchState* st) {
  if (st->cycle_done) return;
  using W = Word<S>;
  using V = typename W::V;
  __shared__ ActiveTiles act;
  list_active(act, a, st->done);
  for (int t = blockIdx.x; t < act.tile0[act.n]; t += gridDim.x) {
    int local;
    const int l = act.lat[tile_lattice(act, t, &local)];
    const int nw = a.geoms[l].half * (W::PER_TILE / (BLAS_TILE / 2)) / 2;
    const size_t off = a.site_off[l] * (W::PER_TILE / (BLAS_TILE / 2)) / 2;
    const int w0 = local * W::PER_TILE + threadIdx.x;
    S beta;
    if constexpr (std::is_same<S, float>::value) beta = st->betaf[l];
    else beta = st->beta[l];
    V rv[W::J], pv[W::J];
#pragma unroll
    for (int j = 0; j < W::J; ++j) {
      const int w = w0 + j * BLAS_BLOCK;
      if (w < nw) {
        rv[j] = reinterpret_cast<const V*>(r)[off + w];
        pv[j] = reinterpret_cast<const V*>(p)[off + w];
      }
    }
#pragma unroll
    for (int j = 0; j < W::J; ++j) {
      const int w = w0 + j * BLAS_BLOCK;
      if (w < nw) reinterpret_cast<V*>(p)[off + w] = W::axpy(beta, pv[j], rv[j]);
    }
  }
  if (!grid_last(&st->grid_cnt[2])) return;
  bool all = true;
  for (int l = threadIdx.x; l < st->nlat; l += blockDim.x) {
    if (!st->done[l]) {
      const double rr = st->rr_new[l], s = st->scale[l];
      st->rr[l] = rr;
      st->iters[l] += 1;
      if (rr * s * s <= st->tol2[l]) st->done[l] = 1;
      else all = false;
    }
  }
  all = __syncthreads_and(all);
  if (threadIdx.x == 0) {
    st->cycle_iter += 1;
    if (all || st->cycle_iter >= st->cycle_limit || st->breakdown || st->nonfinite) st->cycle_done = 1;
  }
}

// x_l += scale_l e_l; e_l = 0 (all lattices not yet verified).
__global__ void __launch_bounds__(BLAS_BLOCK) k_bfold(const BatchArgs a, double2* x, float* e, BatchState* st) {
  __shared__ ActiveTiles act;
  list_active(act, a, st->conv);
  for (int t = blockIdx.x; t < act.tile0[act.n]; t += gridDim.x) {
    int local;
    const int l = act.lat[tile_lattice(act, t, &local)];
    const int n = a.geoms[l].half * 3;
    const size_t off = a.site_off[l] * 3;
    const double s = st->scale[l];
    for (int i = local * BLAS_TILE * 3 + threadIdx.x; i < n && i < (local + 1) * BLAS_TILE * 3; i += BLAS_BLOCK) {
      float2* ep = reinterpret_cast<float2*>(e) + off + i;
      const float2 ev = *ep;
      double2 xv = x[off + i];
      xv.x += s * (double)ev.x;
      xv.y += s * (double)ev.y;
      x[off + i] = xv;
      *ep = make_float2(0.f, 0.f);
    }
  }
}

// Sets st->x_nonzero if any of the n entries of the initial guess is not zero.
__global__ void k_bnonzero(const double2* __restrict__ x, size_t n, BatchState* st) {
  bool nz = false;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double2 v = x[i];
    nz = nz || v.x != 0.0 || v.y != 0.0;
  }
  if (nz) st->x_nonzero = 1;
}

// r_hi = b - Ax (FP64; Ax null: a zero guess, r_hi = b); rr_true and (init) bb per lattice.
__global__ void __launch_bounds__(BLAS_BLOCK) k_bresidual(const BatchArgs a, const double2* b, const double2* Ax, double2* rh,
                                                   BatchState* st, double* partials, size_t pstride, int init) {
  __shared__ double red[32];
  __shared__ ActiveTiles act;
  list_active(act, a, st->conv);
  const int t1 = tile_begin(act, blockIdx.x + 1);
  SumAcc<double> v0, v1;
  for (int t = tile_begin(act, blockIdx.x); t < t1; ++t) {
    int local;
    const int kl = tile_lattice(act, t, &local), l = act.lat[kl];
    const int n = a.geoms[l].half * 3;
    const size_t off = a.site_off[l] * 3;
    for (int i = local * BLAS_TILE * 3 + threadIdx.x; i < n && i < (local + 1) * BLAS_TILE * 3; i += BLAS_BLOCK) {
      const double2 bv = b[off + i], av = Ax ? Ax[off + i] : make_double2(0.0, 0.0);
      const double2 rv = make_double2(bv.x - av.x, bv.y - av.y);
      rh[off + i] = rv;
      v0.add(rv.x * rv.x + rv.y * rv.y);
      if (init) v1.add(bv.x * bv.x + bv.y * bv.y);
    }
    if (t + 1 != t1 && t + 1 != act.tile0[kl + 1]) continue;
    double tot;
    if (lattice_reduce(v0, act, kl, a, partials, st->cnt[3], red, &tot)) {
      st->rr_true[l] = tot;
      if (!isfinite(tot)) st->nonfinite = 1;
    }
    __syncthreads();
    if (init && lattice_reduce(v1, act, kl, a, partials + pstride, st->cnt[4], red, &tot)) st->bb[l] = tot;
    __syncthreads();
    v0 = v1 = SumAcc<double>();
  }
}

// Reliable update per lattice not yet verified: r_lo = r_hi / s, p = r_lo, rr = rr_true / s^2; verified lattices
// are frozen for good. Last CTA: the per-lattice bookkeeping; new cycle, or all verified.
template <typename S>
__global__ void __launch_bounds__(BLAS_BLOCK) k_breliable(const BatchArgs a, const double2* rh, S* r, S* p, BatchState* st) {
  __shared__ ActiveTiles act;
  __shared__ double s_inv;
  list_active(act, a, st->conv);
  for (int t = blockIdx.x; t < act.tile0[act.n]; t += gridDim.x) {
    int local;
    const int l = act.lat[tile_lattice(act, t, &local)];
    const int n = a.geoms[l].half * 3;
    const size_t off = a.site_off[l] * 3;
    __syncthreads();
    if (threadIdx.x == 0) {
      const double s = sqrt(st->rr_true[l] / (double)n);
      s_inv = !(st->rr_true[l] <= st->tol2[l]) && s > 0.0 ? 1.0 / s : 0.0;
    }
    __syncthreads();
    const double inv = s_inv;
    if (inv == 0.0) continue;  // verified now: frozen (uniform over the block)
    for (int i = local * BLAS_TILE * 3 + threadIdx.x; i < n && i < (local + 1) * BLAS_TILE * 3; i += BLAS_BLOCK) {
      const double2 w = rh[off + i];
      const S re = S(w.x * inv), im = S(w.y * inv);
      r[2 * (off + i)] = re;
      r[2 * (off + i) + 1] = im;
      p[2 * (off + i)] = re;
      p[2 * (off + i) + 1] = im;
    }
  }
  if (!grid_last(&st->grid_cnt[5])) return;
  bool all = true;
  for (int l = threadIdx.x; l < st->nlat; l += blockDim.x) {
    if (st->conv[l]) continue;
    const bool c = st->rr_true[l] <= st->tol2[l];
    const double s = sqrt(st->rr_true[l] / (3.0 * a.geoms[l].half));
    st->conv[l] = c;
    st->done[l] = c;
    if (!c && s > 0.0) {
      st->scale[l] = s;
      st->rr[l] = st->rr_true[l] / (s * s);
    }
    all = all && c;
  }
  all = __syncthreads_and(all);
  if (threadIdx.x == 0) {
    st->all_conv = all;
    st->cycle_done = all ? 1 : 0;
    st->cycle_iter = 0;
  }
}

}  // namespace hisq

// ------------------------------------------------------------------ batch object
struct hisq_batch {
  int nlat = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<hisq_ctx*> lat;     // one context per lattice (its links, packing, tuning)
  std::vector<size_t> site_off;   // prefix sums of half
  size_t total_half = 0;
  int num_sms = 0;
  hisq::Geom* d_geoms = nullptr;
  size_t* d_site_off = nullptr;
  const char** d_links[4] = {nullptr, nullptr, nullptr, nullptr};
  size_t* d_blk[4] = {nullptr, nullptr, nullptr, nullptr};
  std::map<int, hisq::TileTable> tiles;  // by tile size
  std::map<std::string, int> tune;
  hisq_ctx* tune_ctx = nullptr;  // borrowed for the tuner's bookkeeping (lattice 0)
  std::map<std::string, DevBuf> ws;
  void* pinned = nullptr;
  long long launches = 0;
  // instantiated iteration graphs, keyed by what their kernels capture
  std::map<std::string, std::pair<cudaGraphExec_t, long long>> graphs;
};

namespace hisq {

static void release_batch_graphs(hisq_batch* B) {
  for (auto& kv : B->graphs) cudaGraphExecDestroy(kv.second.first);
  B->graphs.clear();
}

static void* bws(hisq_batch* B, const char* name, size_t bytes) {
  DevBuf& b = B->ws[name];
  if (b.ptr && b.bytes >= bytes) return b.ptr;
  if (b.ptr) {
    cudaStreamSynchronize(B->stream);
    cudaFree(b.ptr);
    b.ptr = nullptr;
  }
  if (cudaMalloc(&b.ptr, bytes) != cudaSuccess) {
    cudaGetLastError();
    b.ptr = nullptr;
    b.bytes = 0;
    return nullptr;
  }
  b.bytes = bytes;
  return b.ptr;
}

static int tile_table(hisq_batch* B, int tile, TileTable** out) {
  auto it = B->tiles.find(tile);
  if (it != B->tiles.end()) {
    *out = &it->second;
    return HISQ_OK;
  }
  std::vector<int> l0 = {0};
  for (int l = 0; l < B->nlat; ++l) l0.push_back(l0.back() + (B->lat[l]->g.half + tile - 1) / tile);
  TileTable T;
  T.ntiles = l0.back();
  HISQ_CUDA(cudaMalloc(&T.lat_tile0, l0.size() * sizeof(int)));
  HISQ_CUDA(cudaMemcpy(T.lat_tile0, l0.data(), l0.size() * sizeof(int), cudaMemcpyHostToDevice));
  B->tiles[tile] = T;
  *out = &B->tiles[tile];
  return HISQ_OK;
}

static BatchArgs batch_args(hisq_batch* B, int prec, int tile, const TileTable& T) {
  BatchArgs a;
  a.geoms = B->d_geoms;
  a.links = B->d_links[prec];
  a.blk_bytes = B->d_blk[prec];
  a.site_off = B->d_site_off;
  a.lat_tile0 = T.lat_tile0;
  a.tile = tile;
  a.nlat = B->nlat;
  return a;
}

static int persistent_grid(hisq_batch* B, const void* func, int block) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, func, block, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  return B->num_sms * per_sm;
}

struct BatchBufs {
  double2 *x, *b, *rh, *Ax, *t64;
  void *r, *p, *Ap, *t, *e;
  BatchState* st;
  double* partials;
  size_t pstride;  // doubles per row of partials
};

// Launch the batched Dslash in link/spinor type LR/SR with the tuned tile size.
template <typename LR, typename SR, int EPI>
static int bdslash(hisq_batch* B, int p, void* out, const void* in, const void* y, const int* skip, BatchState* st,
                   double* partials, int red_row) {
  constexpr int FORMS = sizeof(LR) == 4 ? 2 : 1;
  decltype(&k_bdslash<LR, SR, EPI, false>) kerns[2] = {k_bdslash<LR, SR, EPI, false>, nullptr};
  if constexpr (FORMS == 2) kerns[1] = k_bdslash<LR, SR, EPI, true>;
  int form = 0;
  char key[64];
  snprintf(key, sizeof key, "bdslash/l%d/s%d/e%d", Real<LR>::prec, Real<SR>::prec, EPI);
  int block = 0;
  auto it = B->tune.find(key);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  HISQ_CUDA(cudaStreamIsCapturing(B->stream, &cap));
  if (it != B->tune.end()) {
    form = it->second / 10000;
    block = it->second % 10000;
  } else if (cap != cudaStreamCaptureStatusNone) {
    block = 128;
  } else {
    // Autotune the form and the tile size: each whole number of warps from 64 sites to 256, by the time with all
    // lattices active (three parts) and with the largest alone (one part; the launch is idempotent). How the tiles
    // fall on the SMs decides, which no few sizes suit for every batch, and the tile that is best for all lattices may
    // be the worst for the few of a solve's last cycles: FP64, 14^2x18x22 + 10x12x26x30 + 18^4, 256 is best with all
    // active and gave 115.7 ms a solve, 96 108.1; four 16^4 57.5 with 224 and 60-63 with any other.
    std::vector<int> act(2 * B->nlat, 1);
    int largest = 0;
    for (int l = 1; l < B->nlat; ++l)
      if (B->lat[l]->g.half > B->lat[largest]->g.half) largest = l;
    for (int l = 0; l < B->nlat; ++l) act[l] = 0;
    act[B->nlat + largest] = 0;
    int* d_act = (int*)bws(B, "tile_act", act.size() * sizeof(int));
    if (!d_act) return set_error(HISQ_ENOMEM, "batch workspace");
    HISQ_CUDA(cudaMemcpyAsync(d_act, act.data(), act.size() * sizeof(int), cudaMemcpyHostToDevice, B->stream));
    HISQ_CUDA(cudaStreamSynchronize(B->stream));
    cudaEvent_t e0, e1;
    HISQ_CUDA(cudaEventCreate(&e0));
    HISQ_CUDA(cudaEventCreate(&e1));
    float best = 1e30f;
    for (int k = 0; k < FORMS * 7; ++k) {
      const int f = k / 7, c = 64 + 32 * (k % 7);
      if (f == 1 && c != 128) continue;  // the one size that fills an SM's 896 threads
      auto kern = kerns[f];
      TileTable* T;
      int rc = tile_table(B, c, &T);
      if (rc != HISQ_OK) return rc;
      const BatchArgs a = batch_args(B, Real<LR>::prec, c, *T);
      const int grid = persistent_grid(B, (const void*)kern, c);
      auto run = [&](const int* sk) { kern<<<grid, c, 0, B->stream>>>(a, p, out, in, y, sk, st, partials, red_row); };
      if (k % 7 == 0 || f == 1) {  // warm-up of a kernel
        run(d_act + B->nlat);
        B->launches += 1;
      }
      // milliseconds of a launch: one; where it takes less than 0.4 ms two more, less than 0.1 four
      auto timed = [&](const int* sk, float* ms, bool once) -> cudaError_t {
        for (int reps = 1;; reps = *ms < 0.1f ? 4 : 2) {
          cudaEventRecord(e0, B->stream);
          for (int r = 0; r < reps; ++r) run(sk);
          cudaEventRecord(e1, B->stream);
          B->launches += reps;
          const cudaError_t e = cudaEventSynchronize(e1);
          if (e != cudaSuccess) return e;
          cudaEventElapsedTime(ms, e0, e1);
          *ms /= (float)reps;
          if (once || reps > 1 || *ms >= 0.4f) return cudaSuccess;
        }
      };
      float ms = 0, alone = 0;
      HISQ_CUDA(timed(d_act, &ms, false));
      HISQ_CUDA(timed(d_act + B->nlat, &alone, ms >= 0.4f));
      ms = 3.f * ms + alone;
      if (ms < best) {
        best = ms;
        form = f;
        block = c;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    B->tune[key] = form * 10000 + block;
  }
  auto kern = kerns[form];
  TileTable* T;
  int rc = tile_table(B, block, &T);
  if (rc != HISQ_OK) return rc;
  const BatchArgs a = batch_args(B, Real<LR>::prec, block, *T);
  kern<<<persistent_grid(B, (const void*)kern, block), block, 0, B->stream>>>(a, p, out, in, y, skip, st, partials,
                                                                            red_row);
  HISQ_CUDA(cudaGetLastError());
  if (cap == cudaStreamCaptureStatusNone) B->launches += 1;
  return HISQ_OK;
}

// Arguments of the BLAS kernels and their grid: one wave of resident blocks, or a block per tile if those are fewer.
static int blas_args(hisq_batch* B, const void* func, BatchArgs* a, int* grid) {
  TileTable* T;
  int rc = tile_table(B, BLAS_TILE, &T);
  if (rc != HISQ_OK) return rc;
  *a = batch_args(B, HISQ_F64, BLAS_TILE, *T);
  *grid = persistent_grid(B, func, BLAS_BLOCK);
  if (*grid > T->ntiles) *grid = T->ntiles;
  return HISQ_OK;
}

// r_hi = b - A_64 x for every lattice not yet verified (zero: x is zero and A x need not be formed).
static int b_true_residual(hisq_batch* B, const BatchBufs& U, int init, bool zero = false) {
  int rc;
  if (!zero) {
    rc = bdslash<double, double, EPI_PLAIN>(B, 1, U.t64, U.x, nullptr, U.st->conv, U.st, U.partials, 0);
    if (rc != HISQ_OK) return rc;
    // the FP64 A uses a_l from the state and writes pAp and alpha, which the inner loop recomputes anyway
    rc = bdslash<double, double, EPI_AXPY>(B, 0, U.Ax, U.t64, U.x, U.st->conv, U.st, U.partials, 0);
    if (rc != HISQ_OK) return rc;
  }
  BatchArgs a;
  int grid;
  if ((rc = blas_args(B, (const void*)k_bresidual, &a, &grid)) != HISQ_OK) return rc;
  k_bresidual<<<grid, BLAS_BLOCK, 0, B->stream>>>(a, U.b, zero ? nullptr : U.Ax, U.rh, U.st, U.partials, U.pstride, init);
  HISQ_CUDA(cudaGetLastError());
  B->launches += 1;
  return HISQ_OK;
}

template <typename S>
static int b_reliable(hisq_batch* B, const BatchBufs& U) {
  BatchArgs a;
  int grid;
  int rc = blas_args(B, (const void*)k_breliable<S>, &a, &grid);
  if (rc != HISQ_OK) return rc;
  k_breliable<S><<<grid, BLAS_BLOCK, 0, B->stream>>>(a, U.rh, (S*)U.r, (S*)U.p, U.st);
  HISQ_CUDA(cudaGetLastError());
  B->launches += 1;
  return HISQ_OK;
}

template <typename S>
static int b_iteration(hisq_batch* B, const BatchBufs& U, int lp) {
  int rc;
  if (lp == HISQ_F64) {
    rc = bdslash<double, double, EPI_PLAIN>(B, 1, U.t, U.p, nullptr, U.st->done, U.st, U.partials, 0);
    if (rc == HISQ_OK)
      rc = bdslash<double, double, EPI_AXPY>(B, 0, U.Ap, U.t, U.p, U.st->done, U.st, U.partials, 0);
  } else {
    rc = bdslash<float, float, EPI_PLAIN>(B, 1, U.t, U.p, nullptr, U.st->done, U.st, U.partials, 0);
    if (rc == HISQ_OK) rc = bdslash<float, float, EPI_AXPY>(B, 0, U.Ap, U.t, U.p, U.st->done, U.st, U.partials, 0);
  }
  if (rc != HISQ_OK) return rc;
  BatchArgs a;
  int grid;
  if ((rc = blas_args(B, (const void*)k_bupdate<S>, &a, &grid)) != HISQ_OK) return rc;
  k_bupdate<S><<<grid, BLAS_BLOCK, 0, B->stream>>>(a, (S*)U.e, (S*)U.r, (const S*)U.p, (const S*)U.Ap, U.st,
                                            U.partials + 2 * U.pstride);
  if ((rc = blas_args(B, (const void*)k_bpupdate<S>, &a, &grid)) != HISQ_OK) return rc;
  k_bpupdate<S><<<grid, BLAS_BLOCK, 0, B->stream>>>(a, (const S*)U.r, (S*)U.p, U.st);
  HISQ_CUDA(cudaGetLastError());
  return HISQ_OK;
}

template <typename S>
static int run_batch(hisq_batch* B, double2* x, const double2* b, const double* mass, double tol, int maxiter,
                     const hisq_solver_opts& o, hisq_solver_stats* stats, int* iters_out, double* res_out) {
  auto t0 = std::chrono::steady_clock::now();
  const int lp = o.inner_prec;
  const bool mixed = lp != HISQ_F64;
  const size_t n = B->total_half * 3;
  BatchBufs U;
  U.x = x;
  U.b = const_cast<double2*>(b);
  U.rh = (double2*)bws(B, "rh", n * sizeof(double2));
  U.Ax = (double2*)bws(B, "Ax", n * sizeof(double2));
  U.t64 = (double2*)bws(B, "t64", n * sizeof(double2));
  U.r = bws(B, "r", n * 2 * sizeof(S));
  U.p = bws(B, "p", n * 2 * sizeof(S));
  U.Ap = bws(B, "Ap", n * 2 * sizeof(S));
  U.t = bws(B, "t", n * 2 * sizeof(S));
  U.e = mixed ? bws(B, "e", n * 2 * sizeof(float)) : (void*)x;
  U.st = (BatchState*)bws(B, "state", sizeof(BatchState));
  // partials: 4 rows of one double per tile of the smallest tile size (64)
  size_t max_tiles = 0;
  for (int l = 0; l < B->nlat; ++l) max_tiles += (B->lat[l]->g.half + 63) / 64;
  U.partials = (double*)bws(B, "partials", 4 * max_tiles * sizeof(double));
  U.pstride = max_tiles;
  if (!U.rh || !U.Ax || !U.t64 || !U.r || !U.p || !U.Ap || !U.t || !U.e || !U.st || !U.partials)
    return set_error(HISQ_ENOMEM, "batch workspace");
  BatchState* h = (BatchState*)B->pinned;
  memset(h, 0, sizeof(BatchState));
  h->nlat = B->nlat;
  h->cycle_limit = mixed ? o.reliable_period : o.poll_every;
  for (int l = 0; l < B->nlat; ++l) {
    h->scale[l] = 1.0;
    h->a[l] = 4.0 * mass[l] * mass[l];
    h->af[l] = (float)h->a[l];
  }
  HISQ_CUDA(cudaMemcpyAsync(U.st, h, sizeof(BatchState), cudaMemcpyHostToDevice, B->stream));
  if (mixed) HISQ_CUDA(cudaMemsetAsync(U.e, 0, n * 2 * sizeof(float), B->stream));
  // a zero initial guess (the usual start) needs no A x: its residual is b
  k_bnonzero<<<B->num_sms * 8, 256, 0, B->stream>>>(x, n, U.st);
  HISQ_CUDA(cudaGetLastError());
  B->launches += 1;
  HISQ_CUDA(cudaMemcpyAsync(&h->x_nonzero, &U.st->x_nonzero, sizeof(int), cudaMemcpyDeviceToHost, B->stream));
  HISQ_CUDA(cudaStreamSynchronize(B->stream));
  int rc = b_true_residual(B, U, 1, h->x_nonzero == 0);
  if (rc != HISQ_OK) return rc;
  HISQ_CUDA(cudaMemcpyAsync(h, U.st, sizeof(BatchState), cudaMemcpyDeviceToHost, B->stream));
  HISQ_CUDA(cudaStreamSynchronize(B->stream));
  for (int l = 0; l < B->nlat; ++l) {
    if (!isfinite(h->bb[l]) || !isfinite(h->rr_true[l]))
      return set_error(HISQ_ENONFINITE, "non-finite source or guess in lattice %d", l);
    h->tol2[l] = tol * tol * h->bb[l];
  }
  HISQ_CUDA(cudaMemcpyAsync(U.st->tol2, h->tol2, sizeof(h->tol2), cudaMemcpyHostToDevice, B->stream));
  if ((rc = b_reliable<S>(B, U)) != HISQ_OK) return rc;
  // pre-tune the inner batched Dslash launches outside the capture: they are idempotent (the
  // pAp they write is recomputed by the first iteration before anything reads it)
  if (lp == HISQ_F64) {
    rc = bdslash<double, double, EPI_PLAIN>(B, 1, U.t, U.p, nullptr, U.st->done, U.st, U.partials, 0);
    if (rc == HISQ_OK) rc = bdslash<double, double, EPI_AXPY>(B, 0, U.Ap, U.t, U.p, U.st->done, U.st, U.partials, 0);
  } else {
    rc = bdslash<float, float, EPI_PLAIN>(B, 1, U.t, U.p, nullptr, U.st->done, U.st, U.partials, 0);
    if (rc == HISQ_OK) rc = bdslash<float, float, EPI_AXPY>(B, 0, U.Ap, U.t, U.p, U.st->done, U.st, U.partials, 0);
  }
  if (rc != HISQ_OK) return rc;

  // one graph = the inner iterations of one reliable cycle, kept in the batch for the next solves: it touches the
  // batch's own buffers only, except that FP64 solves accumulate in the caller's x (which is then in the key); x
  // and b enter in the launches after it
  const int cycle = h->cycle_limit;
  std::string key = "b/" + std::to_string(lp) + "/" + std::to_string(cycle);
  char buf[64];
  for (const void* ptr : {(const void*)U.r, (const void*)U.p, (const void*)U.Ap, (const void*)U.t, (const void*)U.e,
                          (const void*)U.st, (const void*)U.partials}) {
    snprintf(buf, sizeof buf, "/%p", ptr);
    key += buf;
  }
  cudaGraphExec_t exec = nullptr;
  long long nodes = 0;
  auto cached = B->graphs.find(key);
  if (cached != B->graphs.end()) {
    exec = cached->second.first;
    nodes = cached->second.second;
  } else {
    cudaGraph_t graph;
    HISQ_CUDA(cudaStreamBeginCapture(B->stream, cudaStreamCaptureModeThreadLocal));
    int crc = HISQ_OK;
    for (int i = 0; i < cycle && crc == HISQ_OK; ++i) crc = b_iteration<S>(B, U, lp);
    cudaError_t ce = cudaStreamEndCapture(B->stream, &graph);
    if (crc != HISQ_OK) return crc;
    HISQ_CUDA(ce);
    size_t gn = 0;
    cudaGraphGetNodes(graph, nullptr, &gn);
    nodes = (long long)gn;
    ce = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    HISQ_CUDA(ce);
    if (B->graphs.size() >= 8) release_batch_graphs(B);  // bound the cache
    B->graphs[key] = {exec, nodes};
  }
  auto reliable_update = [&]() -> int {
    int r2;
    if (mixed) {
      BatchArgs a;
      int grid;
      if ((r2 = blas_args(B, (const void*)k_bfold, &a, &grid)) != HISQ_OK) return r2;
      k_bfold<<<grid, BLAS_BLOCK, 0, B->stream>>>(a, U.x, (float*)U.e, U.st);
      HISQ_CUDA(cudaGetLastError());
      B->launches += 1;
    }
    if ((r2 = b_true_residual(B, U, 0)) != HISQ_OK) return r2;
    return b_reliable<S>(B, U);
  };

  int status = HISQ_OK;
  int cycles = 0;
  HISQ_CUDA(cudaMemcpyAsync(h, U.st, sizeof(BatchState), cudaMemcpyDeviceToHost, B->stream));
  HISQ_CUDA(cudaStreamSynchronize(B->stream));
  while (!h->all_conv) {
    int maxit = 0;
    for (int l = 0; l < B->nlat; ++l) maxit = h->iters[l] > maxit ? h->iters[l] : maxit;
    if (maxit >= maxiter) {
      status = HISQ_ENOCONV;
      break;
    }
    HISQ_CUDA(cudaGraphLaunch(exec, B->stream));
    B->launches += nodes;
    if ((rc = reliable_update()) != HISQ_OK) return rc;
    ++cycles;
    HISQ_CUDA(cudaMemcpyAsync(h, U.st, sizeof(BatchState), cudaMemcpyDeviceToHost, B->stream));
    HISQ_CUDA(cudaStreamSynchronize(B->stream));
    if (h->nonfinite) {
      status = set_error(HISQ_ENONFINITE, "non-finite residual in the batch");
      break;
    }
    if (h->breakdown) {
      status = set_error(HISQ_EBREAKDOWN, "<p, A p> <= 0 in the batch");
      break;
    }
  }
  double worst = 0.0;
  int total_it = 0;
  for (int l = 0; l < B->nlat; ++l) {
    const double rel = h->bb[l] > 0 ? sqrt(h->rr_true[l] / h->bb[l]) : sqrt(h->rr_true[l]);
    worst = rel > worst ? rel : worst;
    total_it = h->iters[l] > total_it ? h->iters[l] : total_it;
    if (iters_out) iters_out[l] = h->iters[l];
    if (res_out) res_out[l] = rel;
  }
  if (stats) {
    stats->iters = total_it;
    stats->reliable_updates = cycles;
    stats->converged = h->all_conv && status == HISQ_OK;
    stats->true_rel_residual = worst;
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    double bytes = 0;
    for (int l = 0; l < B->nlat; ++l)
      bytes += 2.0 * h->iters[l] * dslash_bytes(B->lat[l], lp, mixed ? HISQ_F32 : HISQ_F64, 1);
    stats->dslash_bytes = bytes;
  }
  if (status == HISQ_ENOCONV) return set_error(HISQ_ENOCONV, "batch: no convergence in %d iterations", maxiter);
  return status;
}

}  // namespace hisq

using namespace hisq;

extern "C" {

int hisq_batch_create(hisq_batch** out, int nlat, const int* dims, unsigned prec_mask, void* stream) {
  if (!out || !dims || nlat < 1 || nlat > MAXB) return set_error(HISQ_EINVAL, "need 1..%d lattices", MAXB);
  *out = nullptr;
  hisq_batch* B = new (std::nothrow) hisq_batch();
  if (!B) return set_error(HISQ_ENOMEM, "host allocation");
  B->nlat = nlat;
  int rc = HISQ_OK;
  if (stream) {
    B->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreate(&B->stream) != cudaSuccess) {
      delete B;
      return set_error(HISQ_ECUDA, "cudaStreamCreate");
    }
    B->own_stream = true;
  }
  prec_mask |= HISQ_PREC_BIT(HISQ_F64) | HISQ_PREC_BIT(HISQ_F32);
  for (int l = 0; l < nlat && rc == HISQ_OK; ++l) {
    hisq_ctx* c = nullptr;
    rc = hisq_create(&c, dims + 4 * l, prec_mask, B->stream);
    if (rc == HISQ_OK) B->lat.push_back(c);
  }
  if (rc == HISQ_OK) {
    B->num_sms = B->lat[0]->num_sms;
    size_t off = 0;
    std::vector<Geom> geoms;
    for (auto* c : B->lat) {
      B->site_off.push_back(off);
      off += c->g.half;
      geoms.push_back(c->g);
    }
    B->total_half = off;
    cudaError_t e = cudaMalloc(&B->d_geoms, nlat * sizeof(Geom));
    if (e == cudaSuccess) e = cudaMemcpy(B->d_geoms, geoms.data(), nlat * sizeof(Geom), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&B->d_site_off, nlat * sizeof(size_t));
    if (e == cudaSuccess)
      e = cudaMemcpy(B->d_site_off, B->site_off.data(), nlat * sizeof(size_t), cudaMemcpyHostToDevice);
    for (int p = 0; p < 4 && e == cudaSuccess; ++p) {
      if (!B->lat[0]->links[p]) continue;
      std::vector<const char*> ptrs;
      std::vector<size_t> blk;
      for (auto* c : B->lat) {
        ptrs.push_back(c->links[p]);
        blk.push_back(link_block_bytes(p, c->g.half));
      }
      e = cudaMalloc(&B->d_links[p], nlat * sizeof(char*));
      if (e == cudaSuccess) e = cudaMemcpy(B->d_links[p], ptrs.data(), nlat * sizeof(char*), cudaMemcpyHostToDevice);
      if (e == cudaSuccess) e = cudaMalloc(&B->d_blk[p], nlat * sizeof(size_t));
      if (e == cudaSuccess) e = cudaMemcpy(B->d_blk[p], blk.data(), nlat * sizeof(size_t), cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) e = cudaMallocHost(&B->pinned, sizeof(BatchState) + 4096);
    if (e != cudaSuccess) rc = cuda_error(e, "batch tables");
  }
  if (rc != HISQ_OK) {
    hisq_batch_destroy(B);
    return rc;
  }
  *out = B;
  return HISQ_OK;
}

int hisq_batch_destroy(hisq_batch* B) {
  if (!B) return HISQ_OK;
  if (B->stream) cudaStreamSynchronize(B->stream);
  release_batch_graphs(B);
  for (auto* c : B->lat) hisq_destroy(c);
  cudaFree(B->d_geoms);
  cudaFree(B->d_site_off);
  for (int p = 0; p < 4; ++p) {
    cudaFree(B->d_links[p]);
    cudaFree(B->d_blk[p]);
  }
  for (auto& kv : B->tiles) cudaFree(kv.second.lat_tile0);
  for (auto& kv : B->ws) cudaFree(kv.second.ptr);
  if (B->pinned) cudaFreeHost(B->pinned);
  if (B->own_stream) cudaStreamDestroy(B->stream);
  delete B;
  return HISQ_OK;
}

int hisq_batch_load_links(hisq_batch* B, int lattice, const double* fat, const double* lng, unsigned flags) {
  if (!B || lattice < 0 || lattice >= B->nlat) return set_error(HISQ_EINVAL, "bad batch or lattice index");
  return hisq_load_links(B->lat[lattice], fat, lng, flags);
}

long long hisq_batch_vector_offset(const hisq_batch* B, int lattice) {
  if (!B || lattice < 0 || lattice > B->nlat) return -1;
  return lattice == B->nlat ? (long long)B->total_half * 3 : (long long)B->site_off[lattice] * 3;
}

int hisq_selftest_batch_form(hisq_batch* B, int form, int tile) {
  if (!B) return set_error(HISQ_EINVAL, "null batch");
  if ((form != 0 && form != 1) || tile < 64 || tile > 256 || tile % 32 || (form == 1 && tile != 128))
    return set_error(HISQ_EINVAL, "no form %d with tiles of %d sites", form, tile);
  release_batch_graphs(B);
  for (int e : {EPI_PLAIN, EPI_AXPY}) {
    B->tune["bdslash/l1/s1/e" + std::to_string(e)] = form * 10000 + tile;
    B->tune["bdslash/l0/s0/e" + std::to_string(e)] = tile;
  }
  return HISQ_OK;
}

long long hisq_batch_launch_count(const hisq_batch* B) { return B ? B->launches : 0; }

int hisq_batch_cg(hisq_batch* B, double* x, const double* b, const double* mass, double rel_tol, int maxiter,
                  const hisq_solver_opts* opts, hisq_solver_stats* stats, int* iters, double* true_res) {
  TraceRange trace("hisq_batch_cg");
  if (!B || !x || !b || !mass) return set_error(HISQ_EINVAL, "null argument");
  for (int l = 0; l < B->nlat; ++l) {
    if (!B->lat[l]->links_ready) return set_error(HISQ_ENOLINKS, "lattice %d has no links", l);
    if (!(mass[l] > 0)) return set_error(HISQ_EINVAL, "mass of lattice %d must be > 0", l);
  }
  if (!(rel_tol > 0) || maxiter < 0) return set_error(HISQ_EINVAL, "need rel_tol > 0 and maxiter >= 0");
  hisq_solver_opts o;
  hisq_solver_opts_default(&o);
  if (opts) o = *opts;
  if (o.inner_prec != HISQ_F64 && o.inner_prec != HISQ_F32)
    return set_error(HISQ_EINVAL, "batched CG supports FP64 or FP32 inner precision");
  if (o.reliable_period < 1 || o.poll_every < 1) return set_error(HISQ_EINVAL, "periods must be >= 1");
  if ((uintptr_t)x % 16 || (uintptr_t)b % 16) return set_error(HISQ_EINVAL, "vectors must be 16-byte aligned");
  if (stats) memset(stats, 0, sizeof *stats);
  const size_t vb = B->total_half * 3 * sizeof(double2);
  const bool xh = !is_device_ptr(x), bh = !is_device_ptr(b);
  double2* dx = xh ? (double2*)bws(B, "user_x", vb) : (double2*)x;
  const double2* db = bh ? (const double2*)bws(B, "user_b", vb) : (const double2*)b;
  if (!dx || !db) return set_error(HISQ_ENOMEM, "staging");
  if (xh) HISQ_CUDA(cudaMemcpyAsync(dx, x, vb, cudaMemcpyHostToDevice, B->stream));
  if (bh) HISQ_CUDA(cudaMemcpyAsync((void*)db, b, vb, cudaMemcpyHostToDevice, B->stream));
  const long long l0 = B->launches;
  int rc = o.inner_prec == HISQ_F64 ? run_batch<double>(B, dx, db, mass, rel_tol, maxiter, o, stats, iters, true_res)
                                    : run_batch<float>(B, dx, db, mass, rel_tol, maxiter, o, stats, iters, true_res);
  if (stats) stats->kernel_launches = B->launches - l0;
  if (xh) {
    cudaError_t e = cudaMemcpyAsync(x, dx, vb, cudaMemcpyDeviceToHost, B->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(B->stream);
    if (e != cudaSuccess && rc == HISQ_OK) rc = cuda_error(e, "copy-out");
  }
  return rc;
}

}  // extern "C"
