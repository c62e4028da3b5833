// Gauge-equivariant parallel-transport convolution (PTC) network on the GPU: the preconditioner apply
// z = N(r), the training loss and both layers' weight gradients, Adam, and the flexible CG that uses it.
//
// Layer: psi'_a(x) = sum_b sum_h W[a,b,h] (T_h psi_b)(x), 9 hops h = 0, +x..+t, -x..-t, with
//   T_+mu psi(x) = F_mu(x) psi(x+mu),  T_-mu psi(x) = F_mu(x-mu)^dag psi(x-mu)
// through the folded FP32 fat links of the context (the same links the Dslash uses).
// Network: layer 1 (1 -> C channels, full lattice), layer 2 (C -> 1, even sites); its input is an
// even-site vector embedded with zeros on odd sites.
//
// The network is linear in its input and in each layer's weights, and both the apply and the training use
// that: the two layers compose into one map whose mixing of the hops is an 8 x 8 matrix, and the loss
// depends on the fields only through an 8 x 8 matrix of inner products (k_ptc_grad). Transports, mixing and
// inner products are FP32 arithmetic on the CUDA cores with the weights rounded to BF16, sums across blocks
// FP64. Master weights and Adam moments are FP32.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <string>
#include <vector>

#include "internal.cuh"
#include "pdl.cuh"
#include "reduce_warp.cuh"
#include "trace.h"

namespace hisq {

bool is_device_ptr(const void* p);
double dslash_bytes(const hisq_ctx* ctx, int lp, int sp, int nrhs);

constexpr int NHOP = 9;

struct PtcGeom {
  Geom g;
  const char* fat32;  // FP32 link storage (16 blocks), fat = kind 0
  size_t blk_bytes;
};

// ------------------------------------------------------------------ preconditioner apply and forward pass
// The network is linear, so its two layers compose into one operator. With the input r on even sites
// (zeros on odd sites) and the output read on even sites x:
//   N(r)(x) = c0 r(x) + sum_{h != 0} T_h phi_h (x),   phi_h(y) = sum_{h' != 0} C[h][h'] (T_h' r)(y)
// on the odd sites y = x + h, with c0 = sum_a W2[a][0] W1[a][0] and C[h][h'] = sum_a W2[a][h] W1[a][h']
// (hops h, h' in +x..+t, -x..-t; at an even site only the identity hop of layer 1 sees r, at an odd
// site only its eight neighbour hops). The 8-channel activation is thereby replaced by the eight
// mixed transports phi_h of each odd site, written once and read once (an activation of half the
// lattice that layer 2 needs at x + h only), and each stencil pass reads every fat link once. The
// weights enter rounded to BF16.
__device__ __forceinline__ cplx<float> bf16c(float2 w) {
  return {__bfloat162float(__float2bfloat16_rn(w.x)), __bfloat162float(__float2bfloat16_rn(w.y))};
}

// mix[0] = c0, mix[1 + 8 (h-1) + (h'-1)] = C[h][h'], from W1 [C][1][9] and W2 [1][C][9].
__global__ void k_ptc_mixing(const float2* __restrict__ w1, const float2* __restrict__ w2, int C, float2* mix) {
  const int t = threadIdx.x;
  if (t > 64) return;
  const int h = t == 0 ? 0 : 1 + (t - 1) / 8, hp = t == 0 ? 0 : 1 + (t - 1) % 8;
  cplx<float> s = {0.f, 0.f};
  for (int a = 0; a < C; ++a) cmac(s, bf16c(w2[a * NHOP + h]), bf16c(w1[a * NHOP + hp]));
  mix[t] = make_float2(s.re, s.im);
}

// The hop h = 1..8 from a site with coordinates c (lexicographic idx, parity par): neighbour cb, and
// the link block and cb of the transport's link (F_mu(x) forward, F_mu(x - mu) backward).
__device__ __forceinline__ int ptc_hop(const PtcGeom& G, const int c[4], int idx, int par, int h, const char** blk,
                                       int* lcb) {
  const Geom& g = G.g;
  const int mu = (h - 1) & 3;
  const bool fwd = h <= 4;
  const int nb = neighbour_cb(g, c, idx, mu, fwd ? 1 : -1);
  *blk = G.fat32 + (size_t)((fwd ? par : 1 - par) * 8 + mu) * G.blk_bytes;
  *lcb = fwd ? (idx >> 1) : nb;
  return nb;
}

// Pass 1, odd sites y: phi_h(y) = sum_h' C[h][h'] (T_h' r)(y), stored as 8 planes [h-1][cb][3] of FP16
// pairs (relative rounding 2^-11, below the network's BF16 weights' 2^-8). Blocks of 128 held to 72
// registers (7 per SM): at 80 registers 32^3x8's 131,072 odd sites needed 1.12 waves of resident
// threads, and the second wave's few blocks ran alone (ncu: 41% of DRAM peak).
__global__ void __launch_bounds__(128, 7) k_ptc_apply_odd(const PtcGeom G, const float2* __restrict__ r,
                                                       __half2* __restrict__ phi, const float2* __restrict__ mix,
                                                       const int* skip) {
  griddep_wait();  // a programmatic dependent launch (pdl.cuh): nothing is touched before this
  griddep_launch_dependents();
  if (skip && *skip) return;
  const Geom& g = G.g;
  for (int cb = blockIdx.x * blockDim.x + threadIdx.x; cb < g.half; cb += gridDim.x * blockDim.x) {
    int c[4];
    site_coords(g, 1, cb, c);
    const int idx = lex_index(g, c);
    cplx<float> acc[8][3];
#pragma unroll
    for (int h = 0; h < 8; ++h)
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[h][k] = {0.f, 0.f};
#pragma unroll 1
    for (int hp = 1; hp <= 8; ++hp) {
      const char* blk;
      int lcb;
      const int nb = ptc_hop(G, c, idx, 1, hp, &blk, &lcb);
      cplx<float> U[9], v[3], s[3];
      LinkIO<float>::load(blk, g.half, lcb, U);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 w = __ldg(r + (size_t)nb * 3 + k);
        v[k] = {w.x, w.y};
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        s[i] = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if (hp <= 4) cmac(s[i], U[3 * i + j], v[j]);
          else cmac_conj(s[i], U[3 * j + i], v[j]);
        }
      }
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const float2 m = __ldg(mix + 1 + 8 * h + (hp - 1));
        const cplx<float> cm = {m.x, m.y};
#pragma unroll
        for (int k = 0; k < 3; ++k) cmac(acc[h][k], cm, s[k]);
      }
    }
#pragma unroll
    for (int h = 0; h < 8; ++h)
#pragma unroll
      for (int k = 0; k < 3; ++k) phi[((size_t)h * g.half + cb) * 3 + k] = __floats2half2_rn(acc[h][k].re, acc[h][k].im);
  }
}

struct FcgState {
  double pq;             // <p, A p> (real: A Hermitian positive)
  double pr[2];          // <p, r>
  double qz[2];          // <q, z>
  double rr, rr_true, bb, tol2, scale;
  int done, iter, cycle_iter, cycle_limit, conv, nonfinite, breakdown, pad;
};

// Sums of a complex quantity over the grid to FP64 accuracy: per-block partials, added in a fixed order by the last
// block to finish; true in thread 0 of that block, with the totals in out. smem: 32 doubles.
__device__ __forceinline__ bool grid_sum2(const SumAcc<float>& re, const SumAcc<float>& im, double* partials,
                                          unsigned* counter, double* smem, double (&out)[2]) {
  const double sr = block_sum_acc(re, smem);
  __syncthreads();
  const double si = block_sum_acc(im, smem);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = sr;
    partials[gridDim.x + blockIdx.x] = si;
  }
  if (!last_block_done(counter)) return false;
  if (threadIdx.x < 64) {
    const double t = warp_sum_partials(partials + (threadIdx.x < 32 ? 0 : gridDim.x), gridDim.x);
    if ((threadIdx.x & 31) == 0) smem[threadIdx.x >> 5] = t;
  }
  __syncthreads();
  out[0] = smem[0];
  out[1] = smem[1];
  return threadIdx.x == 0;
}

// Pass 2, even sites x: z(x) = c0 r(x) + sum_h T_h phi_h (x). DOT: also st->qz = <q, z>, which saves the flexible
// CG a launch and a read of z (12.5 us at 32^3x8).
template <bool DOT>
__global__ void __launch_bounds__(256) k_ptc_apply_even(const PtcGeom G, const float2* __restrict__ r,
                                                        const __half2* __restrict__ phi, float2* __restrict__ z,
                                                        const float2* __restrict__ mix, const int* skip,
                                                        const float2* __restrict__ q, FcgState* st, double* partials,
                                                        unsigned* counter) {
  griddep_wait();  // a programmatic dependent launch (pdl.cuh): nothing is touched before this
  griddep_launch_dependents();
  if (skip && *skip) return;
  const Geom& g = G.g;
  const float2 m0 = __ldg(mix);
  const cplx<float> c0 = {m0.x, m0.y};
  SumAcc<float> vr, vi;
  for (int cb = blockIdx.x * blockDim.x + threadIdx.x; cb < g.half; cb += gridDim.x * blockDim.x) {
    int c[4];
    site_coords(g, 0, cb, c);
    const int idx = lex_index(g, c);
    cplx<float> acc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 w = __ldg(r + (size_t)cb * 3 + k);
      acc[k] = {0.f, 0.f};
      cmac(acc[k], c0, cplx<float>{w.x, w.y});
    }
#pragma unroll 4
    for (int h = 1; h <= 8; ++h) {
      const char* blk;
      int lcb;
      const int nb = ptc_hop(G, c, idx, 0, h, &blk, &lcb);
      cplx<float> U[9], v[3];
      LinkIO<float>::load(blk, g.half, lcb, U);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 w = __half22float2(__ldg(phi + ((size_t)(h - 1) * g.half + nb) * 3 + k));
        v[k] = {w.x, w.y};
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if (h <= 4) cmac(acc[i], U[3 * i + j], v[j]);
          else cmac_conj(acc[i], U[3 * j + i], v[j]);
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) z[(size_t)cb * 3 + k] = make_float2(acc[k].re, acc[k].im);
    if (DOT) {
      float tr = 0.f, ti = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 w = __ldg(q + (size_t)cb * 3 + k);
        tr += w.x * acc[k].re + w.y * acc[k].im;
        ti += w.x * acc[k].im - w.y * acc[k].re;
      }
      vr.add(tr);
      vi.add(ti);
    }
  }
  if (DOT) {
    __shared__ double red[32];
    double t[2];
    if (grid_sum2(vr, vi, partials, counter, red, t)) {
      st->qz[0] = t[0];
      st->qz[1] = t[1];
    }
  }
}

// ------------------------------------------------------------------ training: loss and gradients
// With d = N(b) - x on even sites, the loss of a pair is |d|^2 / |x|^2 and its derivatives are (sums over
// odd sites y and colours; hops h, h' in +x..-t, adj h the opposite hop)
//   dL/dconj W1[a][h'] = sum_h  conj(W2[a][h])  M[h'][adj h] / |x|^2,  M[h'][k] = sum conj((T_h' b)(y)) (T_k d)(y)
//   dL/dconj W2[a][h]  = sum_h' conj(W1[a][h']) M[h'][adj h] / |x|^2
//   and for the identity hops conj(W2[a][0]) m0 / |x|^2 and conj(W1[a][0]) m0 / |x|^2, m0 = sum_x conj(b(x)) d(x):
// layer 1's activation at an odd site is sum_h' W1[a][h'] T_h' b, the loss's derivative with respect to it is
// sum_h conj(W2[a][h]) T_(adj h) d, and T_h^dag = T_(adj h). So a pair costs three stencil passes over the
// fat links (two forward, one for M) and keeps no per-channel field. Groups of up to NV = 4 pairs share
// every link read. 16 pairs at 32^3x8: 32.3 ms with the layers one after the other on the tensor cores (72
// transported planes per pair written and gathered, a host read-back per pair, BF16 operands: gradients
// 1.6e-5 from FP64), 0.76 ms in this form (2.8e-8). A group's three passes take 61, 55 and 58 us under ncu with
// the caches flushed, against about 30 us each for their bytes: they issue on 58, 38 and 64% of the cycles
// (multiply-adds and shared-memory words of the mixing and of the inner products) at 16 warps per SM.
//
// All three passes walk tiles of 32 sites with one warp per hop: a warp loads its hop's link once for the
// group's vectors, and every load of a site (8 links, 8 NV vectors) is in flight at once, where a thread per
// site took the hops in turn and waited for each (with NV threads per site the same passes took 70, 56 and
// 56 us for 4 pairs at 32^3x8).
constexpr int PT_PART = 4;     // per-block partials of a pair: |d|^2, |x|^2, Re m0, Im m0
constexpr int PT_CHUNK = 16;   // pairs whose partials are kept at once
constexpr int PT_SITES = 32;   // sites of a tile
constexpr int PT_ROW = 34;     // float2 per (colour, hop) row of a tile: rows 4 apart lie 16 banks apart
constexpr int PT_FIELD = 3 * 8 * PT_ROW;  // one transported vector's tile [colour][hop][site]

// The link of hop h = 1..8 at site cb of parity par, and the neighbour it transports from.
__device__ __forceinline__ int ptc_tile_link(const PtcGeom& G, int par, int cb, int h, cplx<float> (&U)[9]) {
  int c[4];
  site_coords(G.g, par, cb, c);
  const char* blk;
  int lcb;
  const int nb = ptc_hop(G, c, lex_index(G.g, c), par, h, &blk, &lcb);
  LinkIO<float>::load(blk, G.g.half, lcb, U);
  return nb;
}

// v transported through U (dagger for the hops -mu), into one site's column of a tile field.
__device__ __forceinline__ void ptc_tile_put(float2* field, const cplx<float> (&U)[9], const cplx<float> (&v)[3],
                                             int warp, int lane) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cplx<float> s = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (warp < 4) cmac(s, U[3 * i + j], v[j]);
      else cmac_conj(s, U[3 * j + i], v[j]);
    }
    field[(i * 8 + warp) * PT_ROW + lane] = make_float2(s.re, s.im);
  }
}

// Pass 1 of training, odd sites: phi_h = sum_h' C[h][h'] T_h' b for NV vectors, FP32 planes
// [vector][h][colour][cb] (no FP16 here: training takes inputs of any scale whose squares and products, summed over a
// block's sites in FP32, are FP32 numbers: 1e-18 to 1e16 up to 144^3x36). The next tile's link and vectors are loaded
// while this tile is mixed.
template <int NV>
__global__ void __launch_bounds__(256, 2) k_ptc_train_odd(const PtcGeom G, const float2* __restrict__ b,
                                                          float2* __restrict__ phi, const float2* __restrict__ mix) {
  __shared__ float2 tile[NV * PT_FIELD];
  __shared__ float4 smix[32];  // C[h][h'], two entries each
  griddep_wait();
  griddep_launch_dependents();
  const Geom& g = G.g;
  const size_t half = g.half;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 32) {
    const float2 m0 = __ldg(mix + 1 + 2 * threadIdx.x), m1 = __ldg(mix + 2 + 2 * threadIdx.x);
    smix[threadIdx.x] = make_float4(m0.x, m0.y, m1.x, m1.y);
  }
  const int ntiles = (g.half + PT_SITES - 1) / PT_SITES;
  cplx<float> U[9], v[NV][3];
  auto load = [&](int cb) {
    if (cb >= g.half) return;
    const int nb = ptc_tile_link(G, 1, cb, warp + 1, U);
#pragma unroll
    for (int f = 0; f < NV; ++f)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 w = __ldg(b + ((size_t)f * half + nb) * 3 + k);
        v[f][k] = {w.x, w.y};
      }
  };
  load(blockIdx.x * PT_SITES + lane);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int cb = t * PT_SITES + lane;
    if (cb < g.half) {
#pragma unroll
      for (int f = 0; f < NV; ++f) ptc_tile_put(tile + f * PT_FIELD, U, v[f], warp, lane);
    }
    load(cb + gridDim.x * PT_SITES);
    __syncthreads();
    for (int q = warp; q < NV * 6; q += 8) {  // (vector, colour, four of the eight phi)
      const int f = q / 6, col = (q % 6) >> 1, h0 = (q & 1) * 4;
      cplx<float> s[8];
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const float2 w = tile[f * PT_FIELD + (col * 8 + h) * PT_ROW + lane];
        s[h] = {w.x, w.y};
      }
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        cplx<float> a = {0.f, 0.f};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float4 m = smix[(h0 + o) * 4 + h];
          cmac(a, cplx<float>{m.x, m.y}, s[2 * h]);
          cmac(a, cplx<float>{m.z, m.w}, s[2 * h + 1]);
        }
        if (cb < g.half) phi[((size_t)((f * 8 + h0 + o) * 3 + col)) * half + cb] = make_float2(a.re, a.im);
      }
    }
    __syncthreads();
  }
}

// Pass 2 of training, even sites: d = N(b) - x for NV vectors, planes [vector][colour][cb], and this block's
// sums of |d|^2, |x|^2 and conj(b) d: FP32 terms, summed over a thread's sites (14 at 32^3x8, growing with the lattice)
// and its warp to FP64 accuracy (SumAcc; plain FP32 sums were off by 6e-7 at 32^3x24), FP64 over the block.
template <int NV>
__global__ void __launch_bounds__(256, 2) k_ptc_train_even(const PtcGeom G, const float2* __restrict__ b,
                                                           const float2* __restrict__ phi, const float2* __restrict__ x,
                                                           float2* __restrict__ d, const float2* __restrict__ mix,
                                                           double* __restrict__ part) {
  __shared__ float2 tile[NV * PT_FIELD];
  __shared__ double red[NV * 3][PT_PART];
  griddep_wait();
  griddep_launch_dependents();
  const Geom& g = G.g;
  const size_t half = g.half;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float2 m0 = __ldg(mix);
  constexpr int ITEMS = (NV * 3 + 7) / 8;  // (vector, colour) pairs per warp
  SumAcc<float> s[ITEMS][PT_PART];
  const int ntiles = (g.half + PT_SITES - 1) / PT_SITES;
  cplx<float> U[9], v[NV][3];
  auto load = [&](int cb) {
    if (cb >= g.half) return;
    const int nb = ptc_tile_link(G, 0, cb, warp + 1, U);
#pragma unroll
    for (int f = 0; f < NV; ++f)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 w = __ldg(phi + (size_t)((f * 8 + warp) * 3 + k) * half + nb);
        v[f][k] = {w.x, w.y};
      }
  };
  load(blockIdx.x * PT_SITES + lane);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int cb = t * PT_SITES + lane;
    if (cb < g.half) {
#pragma unroll
      for (int f = 0; f < NV; ++f) ptc_tile_put(tile + f * PT_FIELD, U, v[f], warp, lane);
    }
    load(cb + gridDim.x * PT_SITES);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int q = warp + 8 * j, f = q / 3, col = q % 3;
      if (q < NV * 3 && cb < g.half) {
        const size_t i = ((size_t)f * half + cb) * 3 + col;
        const float2 bv = __ldg(b + i), xv = __ldg(x + i);
        cplx<float> z = {0.f, 0.f};
        cmac(z, cplx<float>{m0.x, m0.y}, cplx<float>{bv.x, bv.y});
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          const float2 w = tile[f * PT_FIELD + (col * 8 + h) * PT_ROW + lane];
          z.re += w.x;
          z.im += w.y;
        }
        const float dx = z.re - xv.x, dy = z.im - xv.y;
        d[((size_t)f * 3 + col) * half + cb] = make_float2(dx, dy);
        s[j][0].add(dx * dx + dy * dy);
        s[j][1].add(xv.x * xv.x + xv.y * xv.y);
        s[j][2].add(bv.x * dx + bv.y * dy);
        s[j][3].add(bv.x * dy - bv.y * dx);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < ITEMS; ++j)
#pragma unroll
    for (int p = 0; p < PT_PART; ++p) {
      const double w = s[j][p].warp_total();
      if (lane == 0 && warp + 8 * j < NV * 3) red[warp + 8 * j][p] = w;
    }
  __syncthreads();
  if (threadIdx.x < NV * PT_PART) {
    const int f = threadIdx.x / PT_PART, p = threadIdx.x % PT_PART;
    part[((size_t)f * gridDim.x + blockIdx.x) * PT_PART + p] = (red[3 * f][p] + red[3 * f + 1][p]) + red[3 * f + 2][p];
  }
}

// This block's part of M for NV pairs: part[pair][block][h' * 8 + k] (FP32 sums over the block's tiles, as in the
// accumulators of a matrix instruction; FP64 over the blocks). After
// the transports of b and d at a tile's odd sites each thread adds its share of the sites to a 4 x 4 corner of
// the 8 x 8 inner products, which stay in registers over the tiles of a persistent grid.
template <int NV>
__global__ void __launch_bounds__(256, 2) k_ptc_grad(const PtcGeom G, const float2* __restrict__ b,
                                                     const float2* __restrict__ d, float2* __restrict__ part) {
  extern __shared__ float2 tile[];  // [pair][b or d][PT_FIELD]
  griddep_wait();
  griddep_launch_dependents();
  const Geom& g = G.g;
  const size_t half = g.half;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // products: WPV warps per pair, each with 8 groups of sites (lane & 7) of 4 corners (lane >> 3)
  constexpr int WPV = 8 / NV;
  const int pv = warp / WPV, pw = warp % WPV, sub = lane & 7, h0 = ((lane >> 3) & 1) * 4, k0 = (lane >> 4) * 4;
  cplx<float> acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = {0.f, 0.f};
  const int ntiles = (g.half + PT_SITES - 1) / PT_SITES;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int cb = t * PT_SITES + lane;
    if (cb < g.half) {
      cplx<float> U[9], v[2 * NV][3];
      const int nb = ptc_tile_link(G, 1, cb, warp + 1, U);
#pragma unroll
      for (int f = 0; f < NV; ++f)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float2 w = __ldg(b + ((size_t)f * half + nb) * 3 + k), e = __ldg(d + ((size_t)f * 3 + k) * half + nb);
          v[2 * f][k] = {w.x, w.y};
          v[2 * f + 1][k] = {e.x, e.y};
        }
#pragma unroll
      for (int f = 0; f < 2 * NV; ++f) ptc_tile_put(tile + f * PT_FIELD, U, v[f], warp, lane);
    } else {
      for (int f = 0; f < 2 * NV; ++f)
        for (int i = 0; i < 3; ++i) tile[f * PT_FIELD + (i * 8 + warp) * PT_ROW + lane] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    const float2* u = tile + (size_t)(2 * pv) * PT_FIELD + h0 * PT_ROW;
    const float2* s = tile + (size_t)(2 * pv + 1) * PT_FIELD + k0 * PT_ROW;
#pragma unroll 1
    for (int q = pw; q < 3 * (PT_SITES / 8); q += WPV) {  // (colour, group of 8 sites)
      const int o = (q / (PT_SITES / 8)) * 8 * PT_ROW + (q % (PT_SITES / 8)) * 8 + sub;
      cplx<float> uv[4], sv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 a = u[o + i * PT_ROW], e = s[o + i * PT_ROW];
        uv[i] = {a.x, a.y};
        sv[i] = {e.x, e.y};
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) cmac_conj(acc[i][j], uv[i], sv[j]);
    }
    __syncthreads();
  }
  // over the 8 site groups of a warp, then over the warps of a pair
  float2* red = tile;  // [warp][64]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float re = acc[i][j].re, im = acc[i][j].im;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (sub == 0) red[warp * 64 + (h0 + i) * 8 + k0 + j] = make_float2(re, im);
    }
  __syncthreads();
  for (int i = threadIdx.x; i < NV * 64; i += blockDim.x) {
    const int v = i / 64, e = i % 64;
    float re = 0.f, im = 0.f;
    for (int w = 0; w < WPV; ++w) {
      re += red[(v * WPV + w) * 64 + e].x;
      im += red[(v * WPV + w) * 64 + e].y;
    }
    part[((size_t)v * gridDim.x + blockIdx.x) * 64 + e] = make_float2(re, im);
  }
}

// The pairs' sums (FP64, in a fixed order). Block (pair, y) takes every PT_SPLIT-th block's part of M:
// tot[pair][y][0..63]; block (pair, 0) also m0 in [64], and |d|^2 and |x|^2 in [65]. Several blocks per pair
// because the conversions and adds are FP64 (one block per pair: 35 us).
constexpr int PT_SPLIT = 8;
constexpr int PT_TOT = 66;
__global__ void __launch_bounds__(256) k_ptc_train_sum(const double* __restrict__ epart, int nblk_e,
                                                       const float2* __restrict__ gpart, int nblk_g,
                                                       double2* __restrict__ tot) {
  griddep_wait();
  griddep_launch_dependents();
  const int pr = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ double es[8][PT_PART];
  __shared__ double2 gs[4][64];
  double2* o = tot + ((size_t)pr * PT_SPLIT + blockIdx.y) * PT_TOT;
  if (blockIdx.y == 0) {
    const double2* e = reinterpret_cast<const double2*>(epart + (size_t)pr * nblk_e * PT_PART);
    double s[PT_PART] = {0, 0, 0, 0};
    for (int i = threadIdx.x; i < nblk_e; i += blockDim.x) {
      const double2 a = e[2 * i], c = e[2 * i + 1];
      s[0] += a.x;
      s[1] += a.y;
      s[2] += c.x;
      s[3] += c.y;
    }
#pragma unroll
    for (int q = 0; q < PT_PART; ++q) {
#pragma unroll
      for (int k = 16; k > 0; k >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], k);
      if (lane == 0) es[warp][q] = s[q];
    }
  }
  {
    const int e = threadIdx.x & 63, part = threadIdx.x >> 6;
    const float2* gp = gpart + (size_t)pr * nblk_g * 64;
    double2 s = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int i = blockIdx.y + PT_SPLIT * part; i < nblk_g; i += 4 * PT_SPLIT) {
      const float2 w = gp[(size_t)i * 64 + e];
      s.x += (double)w.x;
      s.y += (double)w.y;
    }
    gs[part][e] = s;
  }
  __syncthreads();
  const int e = threadIdx.x;
  if (e < 64)
    o[e] = make_double2((gs[0][e].x + gs[1][e].x) + (gs[2][e].x + gs[3][e].x),
                        (gs[0][e].y + gs[1][e].y) + (gs[2][e].y + gs[3][e].y));
  if (blockIdx.y == 0 && (e == 64 || e == 65)) {
    const int q = e == 64 ? 2 : 0;  // (Re m0, Im m0), (|d|^2, |x|^2)
    double2 s = make_double2(0.0, 0.0);
    for (int w = 0; w < 8; ++w) {
      s.x += es[w][q];
      s.y += es[w][q + 1];
    }
    o[e] = s;
  }
}

// Adds the chunk's n pairs, weighted by 1 / (|x|^2 npairs), to acc[PT_TOT] (M, m0, the loss) and, after the last
// chunk, forms the gradients of both layers (C = 8 channels) from M and m0 and the loss (loss[0]).
__global__ void __launch_bounds__(544) k_ptc_train_final(const double2* __restrict__ tot, int n, int npairs,
                                                         double2* acc, int first, int last,
                                                         const float2* __restrict__ w1, const float2* __restrict__ w2,
                                                         int C, float2* __restrict__ g1, float2* __restrict__ g2,
                                                         float* __restrict__ loss) {
  griddep_wait();
  griddep_launch_dependents();
  constexpr int GROUPS = 8;  // groups of threads that each take every 8th pair: one after the other is 36 us
  __shared__ double2 m[PT_TOT], ms[GROUPS][PT_TOT];
  const int grp = threadIdx.x / PT_TOT, e = threadIdx.x % PT_TOT;
  if (grp < GROUPS) {
    double2 s = make_double2(0.0, 0.0);
    for (int i = grp; i < n; i += GROUPS) {
      const double2* t = tot + (size_t)i * PT_SPLIT * PT_TOT;
      const double2 sq = t[65];  // (|d|^2, |x|^2)
      double2 w = t[e];
      if (e < 64) {
#pragma unroll
        for (int y = 1; y < PT_SPLIT; ++y) {
          w.x += t[y * PT_TOT + e].x;
          w.y += t[y * PT_TOT + e].y;
        }
      }
      const double inv = 1.0 / (sq.y * npairs);
      s.x += w.x * inv;
      s.y += w.y * inv;
    }
    ms[grp][e] = s;
  }
  __syncthreads();
  if (threadIdx.x < PT_TOT) {
    double2 s = first ? make_double2(0.0, 0.0) : acc[e];
    for (int k = 0; k < GROUPS; ++k) {
      s.x += ms[k][e].x;
      s.y += ms[k][e].y;
    }
    acc[e] = s;
    m[e] = s;
  }
  __syncthreads();
  if (!last) return;
  if (threadIdx.x == 0) *loss = (float)m[65].x;
  for (int i = threadIdx.x; i < 2 * C * NHOP; i += blockDim.x) {
    const bool second = i >= C * NHOP;
    const int a = (i % (C * NHOP)) / NHOP, h = i % NHOP;
    const float2* w = (second ? w1 : w2) + a * NHOP;  // the other layer's weights of channel a
    double re = 0.0, im = 0.0;
    auto add = [&](cplx<float> c, double2 v) {  // += conj(c) v
      re += (double)c.re * v.x + (double)c.im * v.y;
      im += (double)c.re * v.y - (double)c.im * v.x;
    };
    if (h == 0) {
      add(bf16c(w[0]), m[64]);
    } else {
      for (int q = 0; q < 8; ++q) {
        // W1[h]: M[h][adj q] of W2's hop q; W2[h]: M[q][adj h] of W1's hop q
        const int row = second ? q : h - 1, col = ((second ? h - 1 : q) + 4) & 7;
        add(bf16c(w[1 + q]), m[row * 8 + col]);
      }
    }
    (second ? g2 : g1)[i % (C * NHOP)] = make_float2((float)re, (float)im);
  }
}

// ------------------------------------------------------------------ small kernels
__device__ __forceinline__ int adj_hop(int h) { return h == 0 ? 0 : (h <= 4 ? h + 4 : h - 4); }

// Tied network: W2[0][a][h] = conj(W1[a][0][adj(h)]).
__global__ void k_tie(const float2* __restrict__ w1, float2* __restrict__ w2, int C) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C * NHOP) return;
  const int a = i / NHOP, h = i % NHOP;
  const float2 w = w1[a * NHOP + adj_hop(h)];
  w2[i] = make_float2(w.x, -w.y);
}

// Tied gradient: G1[a][0][h] += conj(G2[0][a][adj(h)]).
__global__ void k_tie_grad(float2* __restrict__ g1, const float2* __restrict__ g2, int C) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C * NHOP) return;
  const int a = i / NHOP, h = i % NHOP;
  const float2 g = g2[a * NHOP + adj_hop(h)];
  g1[i].x += g.x;
  g1[i].y -= g.y;
}

// Adam on FP32 master weights with the real gradient 2*(Re G, Im G) of the Wirtinger gradient G.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v, const float* __restrict__ G,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gr = 2.f * G[i];
  m[i] = b1 * m[i] + (1.f - b1) * gr;
  v[i] = b2 * v[i] + (1.f - b2) * gr * gr;
  w[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
}

// ------------------------------------------------------------------ flexible CG
// The updates take one 16-byte word (two complex entries) of every vector per thread; one thread per block forms the
// complex quotients (see SumAcc on what FP64 costs). With a division by every thread and FP64 sums per site they
// took 15.1 and 17.7 us a launch at 32^3x8 (ncu, caches flushed), in this form 11.8-14.0 and 13.2-15.5 us (three captures).

// alpha = <p, r> / <p, q>; e += alpha p; r -= alpha q; rr = |r|^2; inner convergence, cycle count. nw: words.
__global__ void __launch_bounds__(256) k_fcg_update(float4* __restrict__ e, float4* __restrict__ r,
                                                    const float4* __restrict__ p, const float4* __restrict__ q, size_t nw,
                                                    FcgState* st, double* partials, unsigned* counter) {
  if (st->done) return;
  __shared__ double red[32];
  __shared__ float s_ar, s_ai;
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    const double pq = st->pq;
    const bool ok = pq > 0.0 && isfinite(pq);
    s_ar = ok ? (float)(st->pr[0] / pq) : 0.f;
    s_ai = ok ? (float)(st->pr[1] / pq) : 0.f;
    s_ok = ok;
  }
  __syncthreads();
  const float ar = s_ar, ai = s_ai;
  SumAcc<float> v;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nw; i += (size_t)gridDim.x * blockDim.x) {
    const float4 pv = p[i], qv = q[i];
    float4 rv = r[i], ev = e[i];
    ev.x += ar * pv.x - ai * pv.y;
    ev.y += ar * pv.y + ai * pv.x;
    ev.z += ar * pv.z - ai * pv.w;
    ev.w += ar * pv.w + ai * pv.z;
    rv.x -= ar * qv.x - ai * qv.y;
    rv.y -= ar * qv.y + ai * qv.x;
    rv.z -= ar * qv.z - ai * qv.w;
    rv.w -= ar * qv.w + ai * qv.z;
    e[i] = ev;
    r[i] = rv;
    v.add((rv.x * rv.x + rv.y * rv.y) + (rv.z * rv.z + rv.w * rv.w));
  }
  const double s = block_sum_acc(v, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
  if (!last_block_done(counter) || threadIdx.x >= 32) return;
  const double tot = warp_sum_partials(partials, gridDim.x);
  if (threadIdx.x != 0) return;
  st->rr = tot;
  if (!s_ok) st->breakdown = 1;
  if (!isfinite(tot)) st->nonfinite = 1;
  st->iter += 1;
  st->cycle_iter += 1;
  if (tot * st->scale * st->scale <= st->tol2 || st->cycle_iter >= st->cycle_limit || !s_ok || !isfinite(tot))
    st->done = 1;
}

// p = z + beta p with beta = -<q, z> / <p, q> (restart: beta = 0); pr = <p, r>. nw: words.
__global__ void __launch_bounds__(256) k_fcg_pupdate(float4* __restrict__ p, const float4* __restrict__ z,
                                                     const float4* __restrict__ r, size_t nw, FcgState* st, int restart,
                                                     double* partials, unsigned* counter) {
  if (st->done) return;
  __shared__ double red[32];
  __shared__ float s_br, s_bi;
  if (threadIdx.x == 0) {
    s_br = restart ? 0.f : (float)(-st->qz[0] / st->pq);
    s_bi = restart ? 0.f : (float)(-st->qz[1] / st->pq);
  }
  __syncthreads();
  const float br = s_br, bi = s_bi;
  SumAcc<float> vr, vi;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nw; i += (size_t)gridDim.x * blockDim.x) {
    // a restart never reads p (it may hold stale data)
    const float4 pv = restart ? make_float4(0.f, 0.f, 0.f, 0.f) : p[i], zv = z[i], rv = r[i];
    float4 o;
    o.x = zv.x + br * pv.x - bi * pv.y;
    o.y = zv.y + br * pv.y + bi * pv.x;
    o.z = zv.z + br * pv.z - bi * pv.w;
    o.w = zv.w + br * pv.w + bi * pv.z;
    p[i] = o;
    vr.add((o.x * rv.x + o.y * rv.y) + (o.z * rv.z + o.w * rv.w));  // Re conj(p) r
    vi.add((o.x * rv.y - o.y * rv.x) + (o.z * rv.w - o.w * rv.z));  // Im conj(p) r
  }
  double t[2];
  if (grid_sum2(vr, vi, partials, counter, red, t)) {
    st->pr[0] = t[0];
    st->pr[1] = t[1];
  }
}

// Reliable update, part 1: x += scale e, e = 0 (FP64 x).
__global__ void k_fcg_fold(double2* __restrict__ x, float2* __restrict__ e, size_t n, const FcgState* st) {
  const double s = st->scale;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float2 ev = e[i];
    double2 xv = x[i];
    xv.x += s * (double)ev.x;
    xv.y += s * (double)ev.y;
    x[i] = xv;
    e[i] = make_float2(0.f, 0.f);
  }
}

// r_hi = b - A x (FP64): rr_true (and bb with init).
__global__ void k_fcg_residual(const double2* __restrict__ b, const double2* __restrict__ Ax, double2* __restrict__ rh,
                               size_t n, FcgState* st, int init, double* partials, unsigned* counter) {
  double v0 = 0.0, v1 = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double2 bv = b[i], av = Ax[i];
    const double2 rv = make_double2(bv.x - av.x, bv.y - av.y);
    rh[i] = rv;
    v0 += rv.x * rv.x + rv.y * rv.y;
    v1 += bv.x * bv.x + bv.y * bv.y;
  }
  __shared__ double red[32];
  const double s0 = block_sum_dyn(v0, red), s1 = block_sum_dyn(v1, red);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = s0;
    partials[2 * blockIdx.x + 1] = s1;
  }
  if (!last_block_done(counter)) return;
  double a = 0.0, c = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
    a += __ldcg(partials + 2 * k);
    c += __ldcg(partials + 2 * k + 1);
  }
  a = block_sum_dyn(a, red);
  c = block_sum_dyn(c, red);
  if (threadIdx.x == 0) {
    st->rr_true = a;
    if (init) st->bb = c;
    if (!isfinite(a)) st->nonfinite = 1;
  }
}

// Reliable update, part 2: converged? else r = r_hi / s, rr = |r|^2, new cycle (done = 0).
__global__ void k_fcg_reliable(const double2* __restrict__ rh, float2* __restrict__ r, size_t n, FcgState* st,
                               unsigned* counter) {
  const bool conv = st->rr_true <= st->tol2;
  const double s = sqrt(st->rr_true / (double)n);
  if (!conv && s > 0.0) {
    const double inv = 1.0 / s;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
      const double2 w = rh[i];
      r[i] = make_float2((float)(w.x * inv), (float)(w.y * inv));
    }
  }
  if (last_block_done(counter) && threadIdx.x == 0) {
    st->conv = conv;
    st->done = conv ? 1 : 0;
    st->cycle_iter = 0;
    if (!conv && s > 0.0) {
      st->scale = s;
      st->rr = st->rr_true / (s * s);
    }
  }
}

}  // namespace hisq

// ------------------------------------------------------------------ flexible CG driver
namespace hisq {

static int fcg_true_residual(hisq_ctx* c, double2* x, const double2* b, double2* rh, double2* Ax, double2* t64,
                             FcgState* st, double a, int init, double* partials) {
  DslashCall c1;
  c1.out_parity = 1;
  c1.out = t64;
  c1.in = x;
  c1.nrhs = 1;
  c1.rhs_stride = c->g.half;
  int rc = dslash_launch(c, HISQ_F64, HISQ_F64, c1);
  if (rc != HISQ_OK) return rc;
  DslashCall c2 = c1;
  c2.out_parity = 0;
  c2.out = Ax;
  c2.in = t64;
  c2.y = x;
  c2.a = a;
  c2.epi = EPI_AXPY;
  if ((rc = dslash_launch(c, HISQ_F64, HISQ_F64, c2)) != HISQ_OK) return rc;
  const size_t n = (size_t)c->g.half * 3;
  k_fcg_residual<<<c->num_sms * 4, 256, 0, c->stream>>>(b, Ax, rh, n, st, init, partials, c->d_counters + 20);
  HISQ_CUDA(cudaGetLastError());
  note_launch(c);
  return HISQ_OK;
}

}  // namespace hisq

// ------------------------------------------------------------------ object + C ABI
struct hisq_ptc {
  hisq_ctx* ctx = nullptr;
  int C = 8;
  float2 *w1 = nullptr, *w2 = nullptr;  // FP32 master [C][1][9], [1][C][9]
  float *m1 = nullptr, *v1 = nullptr, *m2 = nullptr, *v2 = nullptr;
  float2 *g1 = nullptr, *g2 = nullptr;  // gradients
  int adam_t = 0;
  int tied = 0;  // layer 2 = adjoint of layer 1 (N = B^dag B)
  float2* mix = nullptr;  // the composed network's mixing coefficients (65 complex), for the apply
};

namespace hisq {

static PtcGeom ptc_geom(const hisq_ctx* c) {
  PtcGeom G;
  G.g = c->g;
  G.fat32 = c->links[HISQ_F32];
  G.blk_bytes = link_block_bytes(HISQ_F32, c->g.half);
  return G;
}

// z = N(r) for nvec even-site FP32 vectors (device), using workspaces of the context: the composed
// linear operator (mixing coefficients formed whenever the weights change, then one stencil pass over
// odd and one over even sites); phi needs 8 * V/2 * 3 half2 of workspace.
// With st: also st->qz = <q, z> (one vector).
static int network_apply(hisq_ptc* P, float2* z, const float2* r, int nvec, __half2* phi, const int* skip = nullptr,
                         const float2* q = nullptr, FcgState* st = nullptr, double* partials = nullptr) {
  hisq_ctx* c = P->ctx;
  const size_t nh = (size_t)c->g.half * 3;
  const PtcGeom G = ptc_geom(c);
  // one site per thread (the grid-stride loops then run once); the block scheduler balances the waves
  const int grid_odd = (c->g.half + 127) / 128;
  int grid_even = (c->g.half + 255) / 256;
  if (st && grid_even > c->num_sms * 64) grid_even = c->num_sms * 64;  // the dot's partials: two per block
  for (int v = 0; v < nvec; ++v) {
    const float2* rv = r + v * nh;
    float2* zv = z + v * nh;
    const float2* mix = P->mix;
    HISQ_CUDA(launch_dependent(c, k_ptc_apply_odd, grid_odd, 128, G, rv, phi, mix, skip));
    HISQ_CUDA(launch_dependent(c, st ? k_ptc_apply_even<true> : k_ptc_apply_even<false>, grid_even, 256, G, rv,
                               (const __half2*)phi, zv, mix, skip, q, st, partials, c->d_counters + 25));
    note_launch(c, 2);
  }
  return HISQ_OK;
}

// Forward pass and gradient sums of NV pairs: d in dv, the blocks' partial sums in epart and gpart.
template <int NV>
static int train_group(hisq_ptc* P, const float2* b, const float2* x, float2* phi, float2* dv, double* epart,
                       float2* gpart, int nblk) {
  hisq_ctx* c = P->ctx;
  const PtcGeom G = ptc_geom(c);
  const size_t smem = (size_t)NV * 2 * PT_FIELD * sizeof(float2);
  const float2* mix = P->mix;
  HISQ_CUDA(launch_dependent(c, k_ptc_train_odd<NV>, nblk, 256, G, b, phi, mix));
  HISQ_CUDA(launch_dependent(c, k_ptc_train_even<NV>, nblk, 256, G, b, (const float2*)phi, x, dv, mix, epart));
  HISQ_CUDA(cudaFuncSetAttribute(k_ptc_grad<NV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  HISQ_CUDA(launch_dependent_smem(c, k_ptc_grad<NV>, nblk, 256, smem, G, b, (const float2*)dv, gpart));
  note_launch(c, 3);
  return HISQ_OK;
}

}  // namespace hisq

using namespace hisq;

extern "C" {

int hisq_ptc_create(hisq_ptc** out, hisq_ctx* ctx, int channels) {
  if (!out || !ctx) return set_error(HISQ_EINVAL, "null argument");
  if (channels != 8) return set_error(HISQ_EINVAL, "the PTC network has 8 hidden channels");
  if (!ctx->links[HISQ_F32]) return set_error(HISQ_EINVAL, "the PTC network needs FP32 links resident");
  hisq_ptc* P = new (std::nothrow) hisq_ptc();
  if (!P) return set_error(HISQ_ENOMEM, "host allocation");
  P->ctx = ctx;
  P->C = channels;
  const size_t nw = (size_t)channels * NHOP;
  cudaError_t e = cudaMalloc(&P->w1, nw * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&P->w2, nw * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&P->g1, nw * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&P->g2, nw * sizeof(float2));
  if (e == cudaSuccess) e = cudaMalloc(&P->m1, 4 * nw * 2 * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(P->m1, 0, 4 * nw * 2 * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&P->mix, 65 * sizeof(float2));
  if (e != cudaSuccess) {
    hisq_ptc_destroy(P);
    return cuda_error(e, "ptc buffers");
  }
  P->v1 = P->m1 + nw * 2;
  P->m2 = P->v1 + nw * 2;
  P->v2 = P->m2 + nw * 2;
  *out = P;
  return HISQ_OK;
}

int hisq_ptc_destroy(hisq_ptc* P) {
  if (!P) return HISQ_OK;
  // the bound context may already be gone: touch only the network's own buffers (cudaFree
  // waits for the device work that may still use them)
  cudaFree(P->w1);
  cudaFree(P->w2);
  cudaFree(P->g1);
  cudaFree(P->g2);
  cudaFree(P->m1);
  cudaFree(P->mix);
  delete P;
  return HISQ_OK;
}

int hisq_ptc_set_weights(hisq_ptc* P, const float* w1, const float* w2) {
  if (!P || !w1 || !w2) return set_error(HISQ_EINVAL, "null argument");
  const size_t nb = (size_t)P->C * NHOP * sizeof(float2);
  HISQ_CUDA(cudaMemcpyAsync(P->w1, w1, nb, cudaMemcpyDefault, P->ctx->stream));
  HISQ_CUDA(cudaMemcpyAsync(P->w2, w2, nb, cudaMemcpyDefault, P->ctx->stream));
  HISQ_CUDA(cudaMemsetAsync(P->m1, 0, 4 * nb, P->ctx->stream));
  P->adam_t = 0;
  if (P->tied) k_tie<<<1, 128, 0, P->ctx->stream>>>(P->w1, P->w2, P->C);
  k_ptc_mixing<<<1, 96, 0, P->ctx->stream>>>(P->w1, P->w2, P->C, P->mix);
  HISQ_CUDA(cudaGetLastError());
  HISQ_CUDA(cudaStreamSynchronize(P->ctx->stream));
  return HISQ_OK;
}

int hisq_ptc_set_tied(hisq_ptc* P, int tied) {
  if (!P) return set_error(HISQ_EINVAL, "null network");
  P->tied = tied ? 1 : 0;
  if (P->tied) {
    k_tie<<<1, 128, 0, P->ctx->stream>>>(P->w1, P->w2, P->C);
    k_ptc_mixing<<<1, 96, 0, P->ctx->stream>>>(P->w1, P->w2, P->C, P->mix);
    HISQ_CUDA(cudaGetLastError());
    HISQ_CUDA(cudaStreamSynchronize(P->ctx->stream));
  }
  return HISQ_OK;
}

int hisq_ptc_bind(hisq_ptc* P, hisq_ctx* c) {
  if (!P || !c) return set_error(HISQ_EINVAL, "null argument");
  for (int m = 0; m < 4; ++m)
    if (c->g.L[m] != P->ctx->g.L[m]) return set_error(HISQ_EINVAL, "lattice shape differs");
  if (!c->links[HISQ_F32]) return set_error(HISQ_EINVAL, "the PTC network needs FP32 links resident");
  if (c->stream != P->ctx->stream) cudaStreamSynchronize(P->ctx->stream);
  P->ctx = c;
  return HISQ_OK;
}

int hisq_ptc_get_weights(hisq_ptc* P, float* w1, float* w2) {
  if (!P || !w1 || !w2) return set_error(HISQ_EINVAL, "null argument");
  const size_t nb = (size_t)P->C * NHOP * sizeof(float2);
  HISQ_CUDA(cudaMemcpyAsync(w1, P->w1, nb, cudaMemcpyDefault, P->ctx->stream));
  HISQ_CUDA(cudaMemcpyAsync(w2, P->w2, nb, cudaMemcpyDefault, P->ctx->stream));
  HISQ_CUDA(cudaStreamSynchronize(P->ctx->stream));
  return HISQ_OK;
}

int hisq_ptc_apply(hisq_ptc* P, float* z, const float* r, int nvec) {
  if (!P || !z || !r || nvec < 1) return set_error(HISQ_EINVAL, "bad argument");
  if (!P->ctx->links_ready) return set_error(HISQ_ENOLINKS, "links not loaded");
  if (!is_device_ptr(z) || !is_device_ptr(r)) return set_error(HISQ_EINVAL, "device vectors only");
  hisq_ctx* c = P->ctx;
  __half2* phi = (__half2*)workspace(c, "ptc_phi", (size_t)8 * c->g.half * 3 * sizeof(__half2));
  if (!phi) return set_error(HISQ_ENOMEM, "ptc workspace");
  // asynchronous on the stream, like hisq_dslash
  return network_apply(P, (float2*)z, (const float2*)r, nvec, phi);
}

// Loss (mean over pairs of |N(b)-x|^2/|x|^2) and Wirtinger gradients of both layers for npairs
// even-site FP32 (b, x) pairs; with lr > 0 an Adam step follows. g1, g2, loss: optional host outputs.
int hisq_ptc_train_step(hisq_ptc* P, const float* b, const float* x, int npairs, float lr, float* loss_out,
                        float* g1_out, float* g2_out) {
  TraceRange trace("hisq_ptc_train_step");
  if (!P || !b || !x || npairs < 1) return set_error(HISQ_EINVAL, "bad argument");
  if (!P->ctx->links_ready) return set_error(HISQ_ENOLINKS, "links not loaded");
  if (!is_device_ptr(b) || !is_device_ptr(x)) return set_error(HISQ_EINVAL, "device vectors only");
  hisq_ctx* c = P->ctx;
  const int C = P->C;
  const size_t nh = (size_t)c->g.half * 3, nw = (size_t)C * NHOP;
  const int nv_max = npairs >= 4 ? 4 : npairs >= 2 ? 2 : 1, chunk = npairs < PT_CHUNK ? npairs : PT_CHUNK;
  // persistent grids of two resident blocks per SM
  const int ntiles = (c->g.half + PT_SITES - 1) / PT_SITES;
  const int nblk = ntiles < 2 * c->num_sms ? ntiles : 2 * c->num_sms;
  float2* phi = (float2*)workspace(c, "ptc_phi32", nv_max * 8 * nh * sizeof(float2));
  float2* dv = (float2*)workspace(c, "ptc_d", nv_max * nh * sizeof(float2));
  double* epart = (double*)workspace(c, "ptc_epart", (size_t)chunk * nblk * PT_PART * sizeof(double));
  float2* gpart = (float2*)workspace(c, "ptc_gpart", (size_t)chunk * nblk * 64 * sizeof(float2));
  double2* tot = (double2*)workspace(c, "ptc_tot", (PT_CHUNK * PT_SPLIT + 1) * PT_TOT * sizeof(double2));
  float2* gw = (float2*)workspace(c, "ptc_gw", (2 * nw + 1) * sizeof(float2));
  if (!phi || !dv || !epart || !gpart || !tot || !gw) return set_error(HISQ_ENOMEM, "workspace");
  float2 *acc1 = gw, *acc2 = gw + nw;
  float* dloss = (float*)(gw + 2 * nw);
  double2* msum = tot + PT_CHUNK * PT_SPLIT * PT_TOT;
  int rc = HISQ_OK;
  for (int q0 = 0; q0 < npairs; q0 += chunk) {
    const int n = npairs - q0 < chunk ? npairs - q0 : chunk;
    for (int q = 0; q < n;) {
      const int nv = n - q >= 4 ? 4 : n - q >= 2 ? 2 : 1;
      const float2 *bq = (const float2*)b + (q0 + q) * nh, *xq = (const float2*)x + (q0 + q) * nh;
      double* ep = epart + (size_t)q * nblk * PT_PART;
      float2* gp = gpart + (size_t)q * nblk * 64;
      rc = nv == 4 ? train_group<4>(P, bq, xq, phi, dv, ep, gp, nblk)
           : nv == 2 ? train_group<2>(P, bq, xq, phi, dv, ep, gp, nblk)
                     : train_group<1>(P, bq, xq, phi, dv, ep, gp, nblk);
      if (rc != HISQ_OK) return rc;
      q += nv;
    }
    HISQ_CUDA(launch_dependent(c, k_ptc_train_sum, dim3(n, PT_SPLIT), 256, (const double*)epart, nblk,
                               (const float2*)gpart, nblk, tot));
    HISQ_CUDA(launch_dependent(c, k_ptc_train_final, 1, 544, (const double2*)tot, n, npairs, msum, (int)(q0 == 0),
                               (int)(q0 + n == npairs), (const float2*)P->w1, (const float2*)P->w2, C, acc1, acc2, dloss));
    note_launch(c, 2);
  }
  if (P->tied) {
    k_tie_grad<<<1, 128, 0, c->stream>>>(acc1, acc2, C);
    HISQ_CUDA(cudaGetLastError());
    note_launch(c);
  }
  if (loss_out || g1_out || g2_out) {  // one read-back for all three
    std::vector<float2> hg(2 * nw + 1);
    HISQ_CUDA(cudaMemcpyAsync(hg.data(), gw, hg.size() * sizeof(float2), cudaMemcpyDeviceToHost, c->stream));
    HISQ_CUDA(cudaStreamSynchronize(c->stream));
    if (loss_out) *loss_out = hg[2 * nw].x;
    if (g1_out) memcpy(g1_out, hg.data(), nw * sizeof(float2));
    if (g2_out) memcpy(g2_out, hg.data() + nw, nw * sizeof(float2));
  }
  if (lr > 0.f) {
    P->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)P->adam_t), c2 = 1.f - powf(b2, (float)P->adam_t);
    const int n = 2 * C * NHOP;
    k_adam<<<1, 256, 0, c->stream>>>((float*)P->w1, P->m1, P->v1, (const float*)acc1, n, lr, b1, b2, 1e-8f, c1, c2);
    if (P->tied)
      k_tie<<<1, 128, 0, c->stream>>>(P->w1, P->w2, C);
    else
      k_adam<<<1, 256, 0, c->stream>>>((float*)P->w2, P->m2, P->v2, (const float*)acc2, n, lr, b1, b2, 1e-8f, c1, c2);
    k_ptc_mixing<<<1, 96, 0, c->stream>>>(P->w1, P->w2, C, P->mix);
    HISQ_CUDA(cudaGetLastError());
    note_launch(c, 3);
    HISQ_CUDA(cudaStreamSynchronize(c->stream));
  }
  return HISQ_OK;
}


int hisq_fcg(hisq_ctx* c, hisq_ptc* P, double* x_user, const double* b_user, double mass, double rel_tol,
             int maxiter, const hisq_solver_opts* opts, hisq_solver_stats* stats) {
  TraceRange trace("hisq_fcg");
  if (!c || !P || !x_user || !b_user) return set_error(HISQ_EINVAL, "null argument");
  if (P->ctx != c) return set_error(HISQ_EINVAL, "the network belongs to another context");
  if (!c->links_ready) return set_error(HISQ_ENOLINKS, "links not loaded");
  if (!(mass > 0) || !(rel_tol > 0) || maxiter < 0) return set_error(HISQ_EINVAL, "need mass > 0, rel_tol > 0");
  if ((uintptr_t)x_user % 16 || (uintptr_t)b_user % 16) return set_error(HISQ_EINVAL, "vectors must be 16-byte aligned");
  hisq_solver_opts o;
  hisq_solver_opts_default(&o);
  if (opts) o = *opts;
  if (o.reliable_period < 1) return set_error(HISQ_EINVAL, "reliable_period must be >= 1");
  if (stats) memset(stats, 0, sizeof *stats);
  auto t_start = std::chrono::steady_clock::now();
  const long long l0 = c->launches;
  const int half = c->g.half;
  const size_t n = (size_t)half * 3;
  const bool xh = !is_device_ptr(x_user), bh = !is_device_ptr(b_user);
  double2* x = xh ? (double2*)workspace(c, "user_x", n * sizeof(double2)) : (double2*)x_user;
  double2* b = bh ? (double2*)workspace(c, "user_b", n * sizeof(double2)) : (double2*)b_user;
  double2* rh = (double2*)workspace(c, "fcg_rh", n * sizeof(double2));
  double2* Ax = (double2*)workspace(c, "fcg_Ax", n * sizeof(double2));
  double2* t64 = (double2*)workspace(c, "fcg_t64", n * sizeof(double2));
  float2* r = (float2*)workspace(c, "fcg_r", n * sizeof(float2));
  float2* p = (float2*)workspace(c, "fcg_p", n * sizeof(float2));
  float2* q = (float2*)workspace(c, "fcg_q", n * sizeof(float2));
  float2* t = (float2*)workspace(c, "fcg_t", n * sizeof(float2));
  float2* z = (float2*)workspace(c, "fcg_z", n * sizeof(float2));
  float2* e = (float2*)workspace(c, "fcg_e", n * sizeof(float2));
  __half2* phi = (__half2*)workspace(c, "ptc_phi", (size_t)8 * c->g.half * 3 * sizeof(__half2));
  FcgState* st = (FcgState*)workspace(c, "fcg_state", sizeof(FcgState));
  double* partials = (double*)workspace(c, "fcg_partials", 4 * (size_t)c->num_sms * 64 * sizeof(double));
  if (!x || !b || !rh || !Ax || !t64 || !r || !p || !q || !t || !z || !e || !phi || !st || !partials)
    return set_error(HISQ_ENOMEM, "fcg workspace");
  if (xh) HISQ_CUDA(cudaMemcpyAsync(x, x_user, n * sizeof(double2), cudaMemcpyHostToDevice, c->stream));
  if (bh) HISQ_CUDA(cudaMemcpyAsync(b, b_user, n * sizeof(double2), cudaMemcpyHostToDevice, c->stream));
  HISQ_CUDA(cudaMemsetAsync(e, 0, n * sizeof(float2), c->stream));
  FcgState* h = (FcgState*)c->pinned;
  memset(h, 0, sizeof(FcgState));
  h->scale = 1.0;
  h->cycle_limit = o.reliable_period;
  HISQ_CUDA(cudaMemcpyAsync(st, h, sizeof(FcgState), cudaMemcpyHostToDevice, c->stream));
  const double a = 4.0 * mass * mass;
  double* red = partials + 2 * (size_t)c->num_sms * 64;
  int rc = fcg_true_residual(c, x, b, rh, Ax, t64, st, a, 1, red);
  if (rc != HISQ_OK) return rc;
  HISQ_CUDA(cudaMemcpyAsync(h, st, sizeof(FcgState), cudaMemcpyDeviceToHost, c->stream));
  HISQ_CUDA(cudaStreamSynchronize(c->stream));
  if (!isfinite(h->bb) || !isfinite(h->rr_true)) return set_error(HISQ_ENONFINITE, "non-finite source or guess");
  h->tol2 = rel_tol * rel_tol * h->bb;
  HISQ_CUDA(cudaMemcpyAsync(&st->tol2, &h->tol2, sizeof(double), cudaMemcpyHostToDevice, c->stream));
  const int gb = c->num_sms * 4;
  // the updates: a 16-byte word (two complex entries) per thread, at most one wave of six blocks per SM
  const size_t nw = n / 2;
  const int gu = (int)std::min<size_t>((nw + 255) / 256, (size_t)c->num_sms * 6);
  auto restart = [&]() -> int {
    k_fcg_reliable<<<gb, 256, 0, c->stream>>>(rh, r, n, st, c->d_counters + 21);
    HISQ_CUDA(cudaGetLastError());
    int r2 = network_apply(P, z, r, 1, phi, &st->done);
    if (r2 != HISQ_OK) return r2;
    k_fcg_pupdate<<<gu, 256, 0, c->stream>>>((float4*)p, (const float4*)z, (const float4*)r, nw, st, 1, red,
                                             c->d_counters + 22);
    HISQ_CUDA(cudaGetLastError());
    note_launch(c, 2);
    return HISQ_OK;
  };
  if ((rc = restart()) != HISQ_OK) return rc;
  // pre-tune the inner Dslash launches (idempotent) outside the capture
  DslashCall c1;
  c1.out_parity = 1;
  c1.out = t;
  c1.in = p;
  c1.nrhs = 1;
  c1.rhs_stride = half;
  DslashCall c2 = c1;
  c2.out_parity = 0;
  c2.out = q;
  c2.in = t;
  c2.y = p;
  c2.a = a;
  c2.epi = EPI_AXPY;
  c2.partials = partials;
  c2.dot_out = &st->pq;
  c2.counter = c->d_counters + 23;
  if ((rc = dslash_launch(c, HISQ_F32, HISQ_F32, c1)) != HISQ_OK) return rc;
  if ((rc = dslash_launch(c, HISQ_F32, HISQ_F32, c2)) != HISQ_OK) return rc;
  c1.skip = &st->done;
  c2.skip = &st->done;
  auto iteration = [&]() -> int {
    int r2 = dslash_launch(c, HISQ_F32, HISQ_F32, c1);
    if (r2 == HISQ_OK) r2 = dslash_launch(c, HISQ_F32, HISQ_F32, c2);
    if (r2 != HISQ_OK) return r2;
    k_fcg_update<<<gu, 256, 0, c->stream>>>((float4*)e, (float4*)r, (const float4*)p, (const float4*)q, nw, st, red,
                                            c->d_counters + 24);
    HISQ_CUDA(cudaGetLastError());
    if ((r2 = network_apply(P, z, r, 1, phi, &st->done, q, st, red)) != HISQ_OK) return r2;
    k_fcg_pupdate<<<gu, 256, 0, c->stream>>>((float4*)p, (const float4*)z, (const float4*)r, nw, st, 0, red,
                                             c->d_counters + 22);
    HISQ_CUDA(cudaGetLastError());
    note_launch(c, 2);
    return HISQ_OK;
  };
  // one graph = the iterations of one reliable cycle, kept in the context for the next solves: it touches the
  // context's workspaces, links and the network's mixing coefficients only (the caller's x and b enter in the
  // launches after it)
  std::string key = "fcg/" + std::to_string(o.reliable_period);
  char buf[64];
  for (const void* ptr : {(const void*)r, (const void*)p, (const void*)q, (const void*)t, (const void*)z, (const void*)e,
                          (const void*)phi, (const void*)st, (const void*)partials, (const void*)P->mix}) {
    snprintf(buf, sizeof buf, "/%p", ptr);
    key += buf;
  }
  snprintf(buf, sizeof buf, "/%a", a);
  key += buf;
  cudaGraphExec_t exec = nullptr;
  long long nodes = 0;
  auto cached = c->graphs.find(key);
  if (cached != c->graphs.end()) {
    exec = cached->second.first;
    nodes = cached->second.second;
  } else {
    cudaGraph_t graph;
    HISQ_CUDA(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
    c->capturing = true;
    int crc = HISQ_OK;
    for (int i = 0; i < o.reliable_period && crc == HISQ_OK; ++i) crc = iteration();
    c->capturing = false;
    cudaError_t ce = cudaStreamEndCapture(c->stream, &graph);
    if (crc != HISQ_OK) return crc;
    HISQ_CUDA(ce);
    size_t gn = 0;
    cudaGraphGetNodes(graph, nullptr, &gn);
    nodes = (long long)gn;
    ce = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    HISQ_CUDA(ce);
    if (c->graphs.size() >= 32) release_graphs(c);  // bound the cache
    c->graphs[key] = {exec, nodes};
  }
  int status = HISQ_OK;
  int reliable = 0;
  HISQ_CUDA(cudaMemcpyAsync(h, st, sizeof(FcgState), cudaMemcpyDeviceToHost, c->stream));
  HISQ_CUDA(cudaStreamSynchronize(c->stream));
  while (!h->conv) {
    if (h->iter >= maxiter) {
      status = HISQ_ENOCONV;
      break;
    }
    HISQ_CUDA(cudaGraphLaunch(exec, c->stream));
    c->launches += nodes;
    // the reliable update: fold the correction into x, true residual in FP64, restart
    k_fcg_fold<<<gb, 256, 0, c->stream>>>(x, e, n, st);
    HISQ_CUDA(cudaGetLastError());
    note_launch(c);
    if ((rc = fcg_true_residual(c, x, b, rh, Ax, t64, st, a, 0, red)) != HISQ_OK) return rc;
    if ((rc = restart()) != HISQ_OK) return rc;
    ++reliable;
    HISQ_CUDA(cudaMemcpyAsync(h, st, sizeof(FcgState), cudaMemcpyDeviceToHost, c->stream));
    HISQ_CUDA(cudaStreamSynchronize(c->stream));
    if (h->nonfinite) {
      status = set_error(HISQ_ENONFINITE, "non-finite residual at iteration %d", h->iter);
      break;
    }
    if (h->breakdown) {
      status = set_error(HISQ_EBREAKDOWN, "<p, A p> <= 0 at iteration %d", h->iter);
      break;
    }
  }
  const double rel = h->bb > 0 ? sqrt(h->rr_true / h->bb) : sqrt(h->rr_true);
  if (stats) {
    stats->iters = h->iter;
    stats->reliable_updates = reliable;
    stats->converged = h->conv && status == HISQ_OK;
    stats->true_rel_residual = rel;
    stats->shift_residual[0] = rel;
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count();
    stats->dslash_calls = 2LL * h->iter + 2LL * (reliable + 1);
    stats->dslash_bytes = 2.0 * h->iter * dslash_bytes(c, HISQ_F32, HISQ_F32, 1) +
                          2.0 * (reliable + 1) * dslash_bytes(c, HISQ_F64, HISQ_F64, 1);
    stats->kernel_launches = c->launches - l0;
  }
  if (xh) {
    HISQ_CUDA(cudaMemcpyAsync(x_user, x, n * sizeof(double2), cudaMemcpyDeviceToHost, c->stream));
    HISQ_CUDA(cudaStreamSynchronize(c->stream));
  }
  if (status == HISQ_ENOCONV) return set_error(HISQ_ENOCONV, "fcg: no convergence in %d iterations (true residual %.3e)", h->iter, rel);
  return status;
}

}  // extern "C"
