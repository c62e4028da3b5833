// Dslash form for few sites: the 16 hops of a site are shared by HS neighbouring threads, each of which
// applies its hops' links to NR vectors; gridDim.y groups of NR vectors go in one launch.
//
// What bounds the one-thread-per-site forms on a small lattice is neither bandwidth nor arithmetic but the
// number of threads: 16^4 has 32,768 sites per parity, 6.7 warps per SM, and each thread walks 16 hops whose
// loads it waits for. HS = 8 gives every thread one forward and one backward hop and eight times the warps
// (16^4 FP32, one vector: 12.5 -> 8.0 us a launch, back to back). In FP64, whose pipe takes a warp's operation in 16
// cycles, it also spreads 8^4's 2,048 sites over all SMs (one vector: 21.0 -> 5.2 us); there the vectors go to
// gridDim.y with NR = 1, since the links of a small lattice are in L2 and arithmetic is what FP64 pays for.
#pragma once
#include "dslash_impl.cuh"

namespace hisq {

// neighbour_cb and the site's coordinate along a run-time direction, without indexing the coordinates (which
// would put them in local memory).
__device__ __forceinline__ int coord_of(const int c[4], int mu) {
  return mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
}
__device__ __forceinline__ int neighbour_cb_dyn(const Geom& g, int cmu, int idx, int mu, int k) {
  const int L = g.L[mu], st = g.stride[mu], cm = cmu + k;
  int n = idx + k * st;
  if (cm >= L) n -= L * st;
  if (cm < 0) n += L * st;
  return n >> 1;
}

template <typename T>
__device__ __forceinline__ T shfl_xor_real(T v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
__device__ __forceinline__ df64 shfl_xor_real(df64 v, int o) {
  return df64(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}

// One real of a vector in its storage type (index in reals), as the arithmetic type and back.
__device__ __forceinline__ double real_load(const double* v, size_t i) { return v[i]; }
__device__ __forceinline__ float real_load(const float* v, size_t i) { return v[i]; }
__device__ __forceinline__ float real_load(const __half* v, size_t i) { return __half2float(v[i]); }
__device__ __forceinline__ float real_load(const __nv_bfloat16* v, size_t i) { return __bfloat162float(v[i]); }
__device__ __forceinline__ void real_store(double* v, size_t i, double x) { v[i] = x; }
__device__ __forceinline__ void real_store(float* v, size_t i, float x) { v[i] = x; }
__device__ __forceinline__ void real_store(__half* v, size_t i, float x) { v[i] = __float2half_rn(x); }
__device__ __forceinline__ void real_store(__nv_bfloat16* v, size_t i, float x) { v[i] = __float2bfloat16_rn(x); }

constexpr int SPLIT_MAX_BLOCK = 256;

// Registers: one vector's sums and one link, held to 64 (four blocks of 256 per SM) for one or two vectors in
// FP32 and 16-bit storage as in the other forms; groups, FP64 and double-float links need more.
template <typename LR, typename SR, int NR, int EPI, int HS>
__global__ void __launch_bounds__(SPLIT_MAX_BLOCK, sizeof(LR) < 8 && NR <= 2 ? 4 : 2)
    dslash_split_kernel(const DslashKArgs k) {
  using A = typename Real<LR>::acc;
  using SA = typename Real<SR>::acc;
  using EA = typename std::conditional<std::is_same<A, df64>::value, double, A>::type;  // arithmetic of the axpy
  static_assert(HS == 2 || HS == 4 || HS == 8, "hop shares per site");
  constexpr int G = HS / 2;
  griddep_wait();  // a programmatic dependent launch (pdl.cuh): nothing is touched before this
  griddep_launch_dependents();
  if (k.skip && *k.skip) return;  // uniform over the grid
  const Geom& g = k.g;
  const int p = k.out_parity;
  const int j = threadIdx.x % HS, part = j / G, l = j % G;
  const int spb = (int)blockDim.x / HS;  // sites per block
  const int r0 = blockIdx.y * NR;
  const char* in = (const char*)k.in + (size_t)r0 * k.rhs_stride * 6 * sizeof(SR);
  SumAcc<SA> dot[NR];

  // all lanes of a warp stay in the loop together (the shares are combined by full-warp shuffles)
  for (int w0 = blockIdx.x * spb; w0 < g.half; w0 += gridDim.x * spb) {
    const int cb = w0 + (int)threadIdx.x / HS;
    const bool live = cb < g.half;
    cplx<A> acc[NR][3];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int a = 0; a < 3; ++a) acc[r][a] = {A(0), A(0)};
    if (live) {
      int c[4];
      site_coords(g, p, cb, c);
      const int idx = lex_index(g, c);
#pragma unroll
      for (int i = 0; i < 8 / HS; ++i) {
        const int q = j * (8 / HS) + i, mu = q >> 1, kind = q & 1, hop = 1 + 2 * kind;
        const int cmu = coord_of(c, mu);
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
          const int nb = neighbour_cb_dyn(g, cmu, idx, mu, dir ? -hop : hop);
          const char* blk = k.links + (size_t)((dir ? 1 - p : p) * 8 + kind * 4 + mu) * k.blk_bytes;
          cplx<A> U[9];
          LinkIO<LR>::load(blk, g.half, dir ? nb : cb, U);
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            cplx<SA> vs[3];
            VecIO<SR>::load(in, (size_t)r * k.rhs_stride + nb, vs);
            const cplx<A> v[3] = {{A(vs[0].re), A(vs[0].im)}, {A(vs[1].re), A(vs[1].im)}, {A(vs[2].re), A(vs[2].im)}};
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
              for (int b = 0; b < 3; ++b) {
                if (dir) cmac_conj_sub(acc[r][a], U[3 * b + a], v[b]);
                else cmac(acc[r][a], U[3 * a + b], v[b]);
              }
          }
        }
      }
    }
    // Combine the shares: the upper half of the lanes keeps the imaginary parts, the lower half the real parts;
    // then sums over the G lanes of each half, of which lane l finishes the colours l, l + G, ..
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      A v[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const A other = shfl_xor_real(part ? acc[r][a].re : acc[r][a].im, G);
        v[a] = (part ? acc[r][a].im : acc[r][a].re) + other;
      }
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = v[a] + shfl_xor_real(v[a], o);
      SA t = SA(0);
      if (live) {
        const size_t base = ((size_t)(r0 + r) * k.rhs_stride + cb) * 6 + part;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          if (a % G != l) continue;
          SA o;
          if (EPI == EPI_PLAIN) {
            o = SA(v[a]);
          } else {
            const SA yv = real_load((const SR*)k.y, base + 2 * a);
            o = SA(fma(axpy_coef<EA>(k, r0 + r), EA(yv), -EA(v[a])));
            t += yv * o;
          }
          real_store((SR*)k.out, base + 2 * a, o);
        }
      }
      if (EPI == EPI_AXPY) dot[r].add(t);
    }
  }

  if (EPI == EPI_AXPY) {
    if (k.partials == nullptr) return;  // uniform over the grid
    __shared__ double red[NR > 2 ? NR * 16 : 32];
    block_sums_acc<NR>(
        red, [&](int r) { return dot[r]; },
        [&](int r, double s) { k.partials[(size_t)(r0 + r) * gridDim.x + blockIdx.x] = s; });
    if (last_block_done(k.counter)) {
      const int lane = threadIdx.x & 31, nw = blockDim.x >> 5, nr = NR * gridDim.y;
      if (nr == 1) {
        const double s = sum_partials_dyn(k.partials, gridDim.x, red);
        if (threadIdx.x == 0) k.dot_out[0] = s;
      } else {
        for (int R = threadIdx.x >> 5; R < nr; R += nw) {
          const double s = warp_sum_partials(k.partials + (size_t)R * gridDim.x, gridDim.x);
          if (lane == 0) k.dot_out[R] = s;
        }
      }
    }
  }
}

}  // namespace hisq
