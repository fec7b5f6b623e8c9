// Instantiation of the persistent coarse-cycle kernel (coarse_cycle.cuh) for one precision
// form.  The including translation unit defines CC_TV (vectors, basis, residual
// minimisation), CC_T (smoother sweeps) and CC_TI (stored block inverses); one
// translation unit per form keeps the build parallel.  With CC_GROUP it is the kernel for
// several columns.
#pragma once
#include "coarse_cycle.cuh"

#include <algorithm>

namespace kcmg {

#define KCMG_CC_SWITCH(np, dim, ...)                                   \
  switch (np * 10 + dim) {                                             \
    case 32: { constexpr int NP = 3, DIM = 2; __VA_ARGS__; } break;    \
    case 62: { constexpr int NP = 6, DIM = 2; __VA_ARGS__; } break;    \
    case 102: { constexpr int NP = 10, DIM = 2; __VA_ARGS__; } break;  \
    case 43: { constexpr int NP = 4, DIM = 3; __VA_ARGS__; } break;    \
    case 103: { constexpr int NP = 10, DIM = 3; __VA_ARGS__; } break;  \
    case 203: { constexpr int NP = 20, DIM = 3; __VA_ARGS__; } break;  \
    default: break;                                                    \
  }

static void* coarse_kernel_ptr(int np, int dim) {
  void* f = nullptr;
#ifdef CC_GROUP
  KCMG_CC_SWITCH(np, dim, { f = (void*)k_coarse_group<CC_TV, CC_T, CC_TI, NP, DIM>; });
#else
  KCMG_CC_SWITCH(np, dim, { f = (void*)k_coarse_cycle<CC_TV, CC_T, CC_TI, NP, DIM>; });
#endif
  return f;
}

// FMAs of one operator application on a level
static long long cc_fmas(const CoarseArgs& a, int l) {
  return (long long)a.lv[l].N * (2 * a.dim + 1) * a.np;
}
// One block needs no grid barrier (about 1 us a phase with every SM taking part) but has one SM's
// FP64 FMA rate, two per clock: it wins while a sweep's FMAs take it less than that.  The same
// for the dense coarsest solve, which belongs to the block that runs the levels above it.
constexpr long long kCoarseSoloFmas = 6000, kCoarseSoloCoarsest = 12000;

// first level that block 0 runs alone: every level from there on, the coarsest included, is small
static int cc_solo_from(const CoarseArgs& a) {
  if ((long long)a.Nc * a.Nc > kCoarseSoloCoarsest) return a.nlev;
  int from = a.nlev - 1;
  while (from > a.lev0 && cc_fmas(a, from - 1) <= kCoarseSoloFmas) --from;
  return from < a.nlev - 1 ? from : a.nlev;
}

// blocks: one per SM and no more than the largest level's cells; one if that runs alone
static int cc_blocks(const CoarseArgs& a, int nsm) {
  if (a.solo_from <= a.lev0) return 1;
  const int cells = a.lv[a.lev0].N / a.np;
  return cells < nsm ? cells : nsm;
}

// longest basis whose coefficients are kept in shared memory (16 KB a level): the default 63
constexpr int kCoarseCoefMax = 63;

// shared-memory layout of a block (a multiple of 16 bytes for every piece)
static void coarse_cycle_layout(CoarseArgs* a, int grid) {
  int top = 0;
  auto take = [&](size_t bytes) {
    const int at = top;
    top += (int)((bytes + 15) / 16 * 16);
    return at;
  };
  const int nch = 1 << a->dim, segs = 2 * a->dim - 2;
  take((size_t)nch * a->np * a->np * sizeof(CC_TV));   // prolongation matrices
  size_t slab = 0, rows_max = 0;
  a->cols = 1;
  for (int l = a->lev0; l < a->nlev; ++l) {
    CoarseLevel& L = a->lv[l];
    const int parts = l >= a->solo_from ? 1 : grid;
    const int cells = L.N / a->np, own = (cells + parts - 1) / parts;
    const size_t rows = (size_t)own * a->np;
    if (l > a->lev0) slab = std::max(slab, rows * nch);                   // children of the own cells
    if (l == a->nlev - 1) break;
    const int pad = a->dim == 2 ? L.n[0] : L.n[0] * L.n[1];   // one block: zeros on both sides
    slab = std::max(slab, (size_t)(parts > 1 ? own + 2 + segs * own : own + 2 * pad) * a->np);
    rows_max = std::max(rows_max, rows);
    a->cols = std::max(a->cols, L.lcap);
    L.sm_r = take(rows * sizeof(CC_TV));
    L.coef_len = 2 * (size_t)L.lcap + (size_t)L.lcap * (L.lcap - 1) / 2;
    L.sm_gm = L.lcap <= kCoarseCoefMax ? take(L.coef_len * sizeof(double)) : -1;
  }
  a->sm_zv = take(slab * sizeof(CC_TV));
  a->sm_zs = sizeof(CC_TV) == sizeof(CC_T) ? a->sm_zv : take(slab * sizeof(CC_T));
  a->sm_ts = take(rows_max * sizeof(CC_T));
  a->sm_ws = take(rows_max * sizeof(CC_TV));
  a->sm_ps = take((size_t)kCoarseThreads * sizeof(double));
  a->sm_red = take((size_t)(2 * a->cols + 4) * sizeof(double));
  a->sm_as = a->smoother == 1 ? take((size_t)(kCoarseThreads / 32) * nch * a->np * sizeof(CC_T)) : 0;
  a->sm_bytes = top;
}

// whether a block's share fits beside the kernel's static shared memory; sets the kernel's limit
static cudaError_t cc_fits(void* f, const CoarseArgs& a, int dev) {
  cudaError_t e;
  int optin = 0, per_sm = 0;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  cudaFuncAttributes fa;
  if ((e = cudaFuncGetAttributes(&fa, f)) != cudaSuccess) return e;
  if (a.sm_bytes + (int)fa.sharedSizeBytes > optin) return cudaErrorInvalidConfiguration;
  if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                optin - (int)fa.sharedSizeBytes)) != cudaSuccess)   // the kernel's, not this context's
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kCoarseThreads, a.sm_bytes)) != cudaSuccess)
    return e;
  return per_sm < 1 ? cudaErrorInvalidConfiguration : cudaSuccess;
}

static cudaError_t cc_launch(void* f, int grid, int smem, void** args, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kCoarseThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, f, args);
}

#ifdef CC_GROUP
template <>
cudaError_t coarse_group_prepare<CC_TV, CC_T, CC_TI>(CoarseArgs* a, int ncol, int* blocks, int* groups) {
  void* f = coarse_kernel_ptr(a->np, a->dim);
  if (!f) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  a->solo_from = cc_solo_from(*a);
  const int cap = cc_blocks(*a, nsm);
  // an equal share of the SMs; more where a block's part does not fit in shared memory
  for (int g = std::max(1, std::min(cap, nsm / ncol)); g <= cap; ++g) {
    coarse_cycle_layout(a, g);
    e = cc_fits(f, *a, dev);
    if (e == cudaErrorInvalidConfiguration) continue;
    if (e != cudaSuccess) return e;
    *blocks = g;
    *groups = std::min(ncol, nsm / g);
    return cudaSuccess;
  }
  return cudaErrorInvalidConfiguration;
}

template <>
cudaError_t launch_coarse_group<CC_TV, CC_T, CC_TI>(const CoarseArgs& a, const CoarseArgs* cols, int ncol, int blocks,
                                                    int groups, cudaStream_t s) {
  void* f = coarse_kernel_ptr(a.np, a.dim);
  void* args[] = {&cols, &ncol, &blocks};
  return cc_launch(f, blocks * groups, a.sm_bytes, args, s);
}
#else
template <>
cudaError_t coarse_cycle_prepare<CC_TV, CC_T, CC_TI>(CoarseArgs* a, int* grid) {
  void* f = coarse_kernel_ptr(a->np, a->dim);
  if (!f) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  a->solo_from = cc_solo_from(*a);
  int g = cc_blocks(*a, nsm);
  if (*grid > 0 && *grid < g) g = *grid;   // the caller's cap
  coarse_cycle_layout(a, g);
  if ((e = cc_fits(f, *a, dev)) != cudaSuccess) return e;
  *grid = g;
  return cudaSuccess;
}

template <>
cudaError_t launch_coarse_cycle<CC_TV, CC_T, CC_TI>(const CoarseArgs& a, int grid, cudaStream_t s) {
  void* f = coarse_kernel_ptr(a.np, a.dim);
  if (!f) return cudaErrorInvalidValue;
  void* args[] = {const_cast<CoarseArgs*>(&a)};
  return cc_launch(f, grid, a.sm_bytes, args, s);
}
#endif

}  // namespace kcmg
