// Host-side launcher of the Dslash kernel for one (link, spinor) precision pair: splits
// nrhs into groups that share each link read and picks the launch form and block size
// with the autotuner.
#pragma once
#include "dslash_split.cuh"
#include "sizing.h"
#include "tune.h"

namespace hisq {

// Tile height (z-planes) of the tiled site walk for a launch reading nvec vectors of vbytes per site: the
// largest divisor of Lz whose seven-slice window of input vectors (the +-3 t-hops) stays within 24 MB, the
// part of L2 the gathers can count on while the links stream through. Where the natural order already
// fits, the largest proper divisor (the walk is then a form for the tuner to reject, and for the tests).
inline int walk_zb_for(const hisq_ctx* ctx, int nvec, size_t vbytes) {
  const Geom& g = ctx->g;
  const double plane_bytes = (double)g.half_x * g.L[1] * nvec * vbytes;
  const double budget = 24.0 * (1 << 20);
  int cap = (int)(budget / (7.0 * plane_bytes));
  if (cap >= g.L[2]) cap = g.L[2] / 2;
  int zb = 1;
  for (int d = 1; d <= cap && d <= g.L[2]; ++d)
    if (g.L[2] % d == 0) zb = d;
  return zb;
}

// The tiled walk's parameters in the kernel arguments (reciprocals for the kernel's two divisions).
inline void set_walk(const hisq_ctx* ctx, DslashKArgs& a, int zb) {
  a.walk_zb = zb;
  a.walk_chunk = zb * ctx->g.half_x * ctx->g.L[1];
  a.walk_m_chunk = ~0ull / (unsigned long long)a.walk_chunk + 1;
  a.walk_m_lt = ~0ull / (unsigned long long)ctx->g.L[3] + 1;
}

// The launch forms of one group of vectors: kernels and their launchers, in the order the tuner numbers them.
struct DslashForms {
  static constexpr int CAP = 12;  // 8 vectors have 9 forms, the most
  const void* func[CAP];
  cudaError_t (*run[CAP])(hisq_ctx* ctx, const DslashKArgs& a, int block);
  int n = 0;
  void add(const void* f, cudaError_t (*r)(hisq_ctx*, const DslashKArgs&, int)) {
    func[n] = f;
    run[n++] = r;
  }
};

// One launch form: NR vectors per thread, TS threads per site (NR * TS vectors per launch); WALK: the
// output sites in the tiled walk (walk_zb_for) instead of cb order.
template <typename LR, typename SR, int NR, int EPI, bool COMP, int TS, bool WALK, bool PF>
static cudaError_t run_dslash(hisq_ctx* ctx, const DslashKArgs& a, int block) {
  int grid = (int)(((size_t)ctx->g.half * TS + block - 1) / block);
  // Plain launches in cb order: a grid of two resident waves with a grid-stride loop.
  // The tiled walk's plain launches take one site per thread: blocks are dispatched in
  // index order, so the sites in flight slide through the walk instead of each
  // resident wave of a grid-stride loop sweeping the whole lattice in turn (144^3x36:
  // DRAM traffic 1.13x -> 1.02x of the algorithmic bytes). Reducing launches: one wave
  // of the blocks that are resident together keeps the partials, and the finishing
  // block's sum over them, short (a grid of one site per thread made the per-vector
  // sums of the 8-vector form the launch's tail).
  int cap = WALK ? grid : max_grid_blocks(ctx, block);
  if (EPI == EPI_AXPY && a.partials) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, dslash_kernel<LR, SR, NR, EPI, COMP, TS, PF>, block, 0);
    cap = ctx->num_sms * (per_sm > 0 ? per_sm : 1);
  }
  if (grid > cap) grid = cap;
  DslashKArgs b = a;
  if (WALK) set_walk(ctx, b, walk_zb_for(ctx, NR * TS, 6 * sizeof(SR)));
  return launch_dependent(ctx, dslash_kernel<LR, SR, NR, EPI, COMP, TS, PF>, grid, block, b);
}

template <typename LR, typename SR, int NR, int EPI, bool COMP, int TS, bool WALK = false, bool PF = false>
static void add_dslash(DslashForms& f) {
  f.add((const void*)dslash_kernel<LR, SR, NR, EPI, COMP, TS, PF>, run_dslash<LR, SR, NR, EPI, COMP, TS, WALK, PF>);
}

// One launch form of dslash_split_kernel: the launch's vectors in groups of NR, HS threads per (site, group).
template <typename LR, typename SR, int NR, int EPI, int HS>
static cudaError_t run_split(hisq_ctx* ctx, const DslashKArgs& a, int block) {
  int grid = (int)(((size_t)ctx->g.half * HS + block - 1) / block);
  int cap = max_grid_blocks(ctx, block);
  if (EPI == EPI_AXPY && a.partials) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, dslash_split_kernel<LR, SR, NR, EPI, HS>, block, 0);
    cap = ctx->num_sms * (per_sm > 0 ? per_sm : 1);
  }
  if (grid > cap) grid = cap;
  return launch_dependent(ctx, dslash_split_kernel<LR, SR, NR, EPI, HS>, dim3(grid, a.nvec / NR), block, a);
}

template <typename LR, typename SR, int NR, int EPI, int HS>
static void add_split(DslashForms& f) {
  f.add((const void*)dslash_split_kernel<LR, SR, NR, EPI, HS>, run_split<LR, SR, NR, EPI, HS>);
}

// The split forms are offered where the site count times the shares fills the GPU at most twice (1024 threads
// per SM are one wave at 64 registers): beyond that one thread per site has warps enough and measured faster.
inline bool split_fits(const hisq_ctx* ctx, int shares) {
  return (double)ctx->g.half * shares <= 2.0 * ctx->num_sms * 1024;
}

static int launch_tuned(hisq_ctx* ctx, const char* key, const DslashForms& f, const DslashKArgs& a) {
  int vi = 0, block = 0;
  int rc = tuned_variant(ctx, key, f.func, f.n, [&](int i, int b) { return f.run[i](ctx, a, b); }, &vi, &block);
  if (rc != HISQ_OK) return rc;
  HISQ_CUDA(f.run[vi](ctx, a, block));
  note_launch(ctx);
  return HISQ_OK;
}

// The forms of a group of NR vectors in one thread per site, in cb order and (groups of 1 and 5 to 8) in the
// tiled walk, and, with few sites and uncompressed links, the split forms; added to f.
template <typename LR, typename SR, int NR, int EPI, bool COMP>
static void group_forms(DslashForms& f, const hisq_ctx* ctx) {
  add_dslash<LR, SR, NR, EPI, COMP, 1>(f);
  if (NR == 2) add_dslash<LR, SR, 1, EPI, COMP, 2>(f);
  if (NR == 4) {
    add_dslash<LR, SR, 2, EPI, COMP, 2>(f);
    add_dslash<LR, SR, 1, EPI, COMP, 4>(f);
  }
  if constexpr (NR == 8) {
    add_dslash<LR, SR, 4, EPI, COMP, 2>(f);
    add_dslash<LR, SR, 2, EPI, COMP, 4>(f);
    add_dslash<LR, SR, 8, EPI, COMP, 1, true>(f);
    add_dslash<LR, SR, 4, EPI, COMP, 2, true>(f);
    add_dslash<LR, SR, 2, EPI, COMP, 4, true>(f);
    add_dslash<LR, SR, 8, EPI, COMP, 1, false, true>(f);
    add_dslash<LR, SR, 8, EPI, COMP, 1, true, true>(f);
  }
  if (NR == 1 || (NR > 4 && NR < 8)) add_dslash<LR, SR, NR, EPI, COMP, 1, true>(f);
  if constexpr (!COMP) {
    if constexpr (NR == 1)
      if (split_fits(ctx, 2)) add_split<LR, SR, 1, EPI, 2>(f);
    if constexpr (sizeof(LR) < 8 || NR == 1)
      if (split_fits(ctx, 4)) add_split<LR, SR, NR, EPI, 4>(f);
    if constexpr (NR == 1)
      if (split_fits(ctx, 8)) add_split<LR, SR, 1, EPI, 8>(f);
  }
}

// A group of nr vectors shares each link read. The launch forms differ in how the group is spread
// over threads (vectors per thread x threads per site); the tuner times each and keeps the fastest.
template <typename LR, typename SR, int EPI, bool COMP>
static int launch_nr(hisq_ctx* ctx, const DslashKArgs& a, int nr) {
  char key[64];
  DslashForms f;
  snprintf(key, sizeof key, "dslash/l%d/s%d/nr%d/e%d/c%d", Real<LR>::prec, Real<SR>::prec, nr, EPI, (int)COMP);
  if constexpr (sizeof(LR) == 8) {
    if (nr > 1 && split_fits(ctx, 2 * nr)) {  // FP64 on few sites: each vector in its own row of blocks
      snprintf(key, sizeof key, "dslash/l%d/s%d/ny%d/e%d", Real<LR>::prec, Real<SR>::prec, nr, EPI);
      add_split<LR, SR, 1, EPI, 2>(f);
      if (split_fits(ctx, 4 * nr)) add_split<LR, SR, 1, EPI, 4>(f);
      if (split_fits(ctx, 8 * nr)) add_split<LR, SR, 1, EPI, 8>(f);
      // near the line the thread-per-site forms fill the FP64 pipe as well and read each link once for all the
      // vectors (8x10x14x34: two vectors 38.4 us, 39.1 split, four 74.2 and 75.7; 8^4: two vectors 21.2 and 7.2)
      if (nr == 2) group_forms<LR, SR, 2, EPI, COMP>(f, ctx);
      if (nr == 3) group_forms<LR, SR, 3, EPI, COMP>(f, ctx);
      if (nr == 4) group_forms<LR, SR, 4, EPI, COMP>(f, ctx);
      return launch_tuned(ctx, key, f, a);
    }
  }
  switch (nr) {
    case 1: group_forms<LR, SR, 1, EPI, COMP>(f, ctx); break;
    case 2: group_forms<LR, SR, 2, EPI, COMP>(f, ctx); break;
    case 3: group_forms<LR, SR, 3, EPI, COMP>(f, ctx); break;
    case 4: group_forms<LR, SR, 4, EPI, COMP>(f, ctx); break;
  }
  if constexpr (sizeof(LR) < 8) {
    switch (nr) {
      case 5: group_forms<LR, SR, 5, EPI, COMP>(f, ctx); break;
      case 6: group_forms<LR, SR, 6, EPI, COMP>(f, ctx); break;
      case 7: group_forms<LR, SR, 7, EPI, COMP>(f, ctx); break;
      case 8: group_forms<LR, SR, 8, EPI, COMP>(f, ctx); break;
    }
  }
  if (f.n == 0) return set_error(HISQ_EINVAL, "unsupported rhs group %d", nr);
  return launch_tuned(ctx, key, f, a);
}

// Largest rhs group per launch: 8, because a group of 16 needs more than the 255 registers a thread can hold
// and spills (measured 5x slower than two groups of 8). FP64 and double-float groups stop at 4, but where the
// split forms fit they take as many vectors as fit.
template <typename LR>
static int max_group(const hisq_ctx* ctx) {
  if (sizeof(LR) < 8) return 8;
  int n = 8;
  while (n > 4 && !split_fits(ctx, 2 * n)) --n;
  return n;
}

// Whether the context holds compressed long links (two rows, third reconstructed) of the precision.
template <typename LR>
static bool compressed(const hisq_ctx* ctx) {
  return sizeof(LR) < 8 && ctx->naik != 0.0 && ctx->long12[Real<LR>::prec] != nullptr;
}

// One launch per group of vectors, cut as given (LaunchCut).
template <typename LR, typename SR>
static int launch_groups(hisq_ctx* ctx, const DslashCall& c, int cut, int gmax) {
  const size_t site_bytes = 6 * sizeof(SR);
  int r0 = 0;
  while (r0 < c.nrhs) {
    const int nr = next_group(cut, c.nrhs - r0, gmax);
    DslashKArgs a;
    a.g = ctx->g;
    a.links = ctx->links[Real<LR>::prec];
    a.blk_bytes = link_block_bytes(Real<LR>::prec, ctx->g.half);
    a.out_parity = c.out_parity;
    a.out = (char*)c.out + (size_t)r0 * c.rhs_stride * site_bytes;
    a.in = (const char*)c.in + (size_t)r0 * c.rhs_stride * site_bytes;
    a.rhs_stride = c.rhs_stride;
    a.nvec = nr;
    a.y = c.y ? (const char*)c.y + (size_t)r0 * c.rhs_stride * site_bytes : nullptr;
    for (int r = 0; r < 16; ++r) {
      a.a[r] = (c.a_rhs && r0 + r < c.nrhs) ? c.a_rhs[r0 + r] : c.a;
      a.af[r] = (float)a.a[r];
    }
    a.partials = c.partials ? c.partials + (size_t)r0 * partial_stride(ctx) : nullptr;
    a.dot_out = c.dot_out ? c.dot_out + r0 : nullptr;
    a.counter = c.counter;
    a.skip = c.skip;
    const bool comp = compressed<LR>(ctx);
    a.long12 = comp ? ctx->long12[Real<LR>::prec] : nullptr;
    a.blk12 = long12_block_bytes(Real<LR>::prec, ctx->g.half);
    a.inv_naik = comp ? (float)(1.0 / ctx->naik) : 0.f;
    a.flags = ctx->load_flags;
    int rc;
    if constexpr (sizeof(LR) < 8) {
      if (comp)
        rc = c.epi == EPI_PLAIN ? launch_nr<LR, SR, EPI_PLAIN, true>(ctx, a, nr)
                                : launch_nr<LR, SR, EPI_AXPY, true>(ctx, a, nr);
      else
        rc = c.epi == EPI_PLAIN ? launch_nr<LR, SR, EPI_PLAIN, false>(ctx, a, nr)
                                : launch_nr<LR, SR, EPI_AXPY, false>(ctx, a, nr);
    } else {
      rc = c.epi == EPI_PLAIN ? launch_nr<LR, SR, EPI_PLAIN, false>(ctx, a, nr)
                              : launch_nr<LR, SR, EPI_AXPY, false>(ctx, a, nr);
    }
    if (rc != HISQ_OK) return rc;
    r0 += nr;
  }
  return HISQ_OK;
}

// D (or A's second half) on c.nrhs vectors. Where they can be cut in more than one way the tuner times each: no way is
// best everywhere. Measured, us: FP32, 12 vectors, 8+4 27.3 at 16^4 and 392 at 48^3x12, 6+6 34.7 and 416; FP32, 9
// vectors, 8+1 23.1 and 354, 5+4 26.9 and 342; double-float, 6 vectors at 32^3x8, 4+2 286, 3+3 371; FP64, 6 vectors,
// 4+2 258 at 16^4 and 734 at 32^3x8, 3+3 194 and 765. The powers of two (2+1 for 3) matter for FP64 and double-float,
// whose launch of three takes nearly as long as one of four.
template <typename LR, typename SR>
int dslash_launch_t(hisq_ctx* ctx, const DslashCall& c) {
  const int gmax = max_group<LR>(ctx);
  // few sites in FP64, where a launch is a row of blocks per vector: even groups (A of 10 vectors at 8^4: 59.5 us, 8+2 88)
  if (sizeof(LR) == 8 && gmax > 4) return launch_groups<LR, SR>(ctx, c, CUT_EVEN, gmax);
  int cuts[3], cut;
  const int n = launch_cuts(c.nrhs, gmax, sizeof(LR) == 8, cuts);
  if (n == 1) return launch_groups<LR, SR>(ctx, c, cuts[0], gmax);
  char key[64];
  snprintf(key, sizeof key, "dslash/l%d/s%d/cut%d/e%d/c%d", Real<LR>::prec, Real<SR>::prec, c.nrhs, c.epi, (int)compressed<LR>(ctx));
  int rc = tuned_way(ctx, key, cuts, n, [&](int w) { return launch_groups<LR, SR>(ctx, c, w, gmax); }, &cut);
  if (rc != HISQ_OK) return rc;
  return launch_groups<LR, SR>(ctx, c, cut, gmax);
}

}  // namespace hisq
