// Loop control, reductions and epilogues shared by the per-step kernels (kernels.cu,
// pattern_ops.cuh): the last block of a reduction takes the decisions of Alg. 1 and Alg. 2.
#pragma once
#include "kcmg_internal.h"
#include "reduce.cuh"

#include <cmath>

namespace kcmg {

// Sum over the block with a fixed shuffle/shared-memory tree (deterministic).
// Result valid in thread 0.  sh: >= 32 doubles of shared memory.
static __device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
  __syncthreads();
  if (ln == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    r = (ln < nw) ? sh[ln] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  return r;
}

// True in every thread of the block that finished last (all partials visible).
static __device__ __forceinline__ bool last_block(unsigned int* ticket) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Final reduction of few columns: out[c] = sum_b partial[b*ncol + c] (fixed order).
static __device__ void reduce_few(const double* partial, int nblk, int ncol, double* out, double* sh) {
  for (int c = 0; c < ncol; ++c) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += __ldcg(partial + (size_t)b * ncol + c);
    s = block_sum(s, sh);
    if (threadIdx.x == 0) out[c] = s;
  }
  __syncthreads();
}

static __device__ __forceinline__ void set_cond(const EpiArgs& e, int c) {
  e.st->cond = c;
  if (e.use_handle) cudaGraphSetConditional(e.handle, c ? 1u : 0u);
}

// Loop condition of Alg. 2 on a level.  The guard (loop bodies executed in this solve,
// counted outside the reductions) bounds every while loop independently of the rest.
static __device__ __forceinline__ int more_cycles(const LevelState* st) {
  return (st->rnorm > st->eps) && (st->it < st->maxit) && (st->status == KCMG_OK) &&
         (st->guard < st->guard_cap);
}

static __device__ __forceinline__ void record(const EpiArgs& e, int type) {
  LevelState* st = e.st;
  if (st->level == 0 && e.hist && st->hist_len < st->hist_cap) {
    e.hist[st->hist_len] = st->rnorm;
    e.hist_type_buf[st->hist_len] = type;
    st->hist_len++;
  }
}

// Epilogues run by thread 0 of the last block with the reduced sums.
static __device__ void epilogue(const EpiArgs& e, const double* sums) {
  LevelState* st = e.st;
  switch (e.kind) {
    case EPI_MG_BEGIN: {
      st->rnorm0 = st->rnorm = sqrt(sums[0]);
      st->eps = fmax(st->rtol * st->rnorm0, st->atol);
      st->l = 0; st->it = 0; st->flags = 0; st->breakdowns = 0; st->restart_req = 0; st->left = 0.0;
      if (!isfinite(st->rnorm)) st->status = KCMG_NONFINITE;
      record(e, 0);
      set_cond(e, more_cycles(st));
    } break;
    // W^T w, ||w||^2 and w . r decide the whole step: the norm of w_hat = w - W h by Pythagoras
    // (kPythagoras; else the second Gram-Schmidt pass is requested, "twice is enough"), and
    // alpha = w_hat . r = w . r - h . (W^T r).  r is orthogonal to W but for what its last update has
    // left of the last column: alpha of that step was taken this way, too, and its error would come
    // back multiplied with every h, until r grows (FP64, 12 x 12 x 8, p = 2, lmax 400: from 1e-16 to
    // 1e-8 of ||b|| in 60 cycles).  The update measures it, and the next one takes it out.
    case EPI_GRAM1: {
      const int l = st->l;
      const double naz2 = sums[l], nw2 = naz2 - sums[l + 2];   // [l + 2]: sum of the squared coefficients
      st->naz2 = naz2;
      int f = 0;
      if (!isfinite(naz2) || !(naz2 > 0.0)) f |= F_DISCARD;
      else if (l > 0 && nw2 < kPythagoras * naz2) f |= F_REORTH;
      else {
        st->gamma = 1.0 / sqrt(nw2);
        st->alpha = st->gamma * (sums[l + 1] - (l > 0 ? sums[l - 1] * st->left : 0.0));
      }
      if (!isfinite(naz2) && st->level == 0) st->status = KCMG_NONFINITE;
      st->flags = f;
    } break;
    // the second pass: w' = w - W h
    case EPI_GRAM2: {
      const int l = st->l;
      const double n2 = sums[l], nw2 = n2 - sums[l + 2];
      if (!isfinite(nw2)) {
        st->flags |= F_DISCARD;
        if (!isfinite(n2) && st->level == 0) st->status = KCMG_NONFINITE;
      } else if (nw2 < kPythagoras * n2) {
        st->flags |= F_OWN_NORM;
      } else if (!(nw2 > st->brk * st->brk * st->naz2)) {
        st->flags |= F_DISCARD;
      } else {
        st->gamma = 1.0 / sqrt(nw2);
        st->alpha = st->gamma * (sums[l + 1] - sums[l - 1] * st->left);   // l > 0 here
      }
    } break;
    case EPI_FINISH: {
      if (!(st->flags & F_DISCARD)) {
        st->l++;
        st->left = sums[1];
        st->breakdowns = 0;
      } else if (st->level == 0) {
        if (++st->breakdowns >= 2 && st->status == KCMG_OK) st->status = KCMG_BREAKDOWN;
      }
      st->rnorm = sqrt(sums[0]);
      if (!isfinite(st->rnorm) && st->status == KCMG_OK) st->status = KCMG_NONFINITE;
      record(e, e.hist_type);
      if (e.end_iter) {
        st->it++;
        st->iters_total++;
        const int cap = (st->lmax > 0 && st->lmax < st->lcap) ? st->lmax : st->lcap;
        if (st->level == 0 && !(st->rnorm > st->eps) && st->l > 0) st->restart_req = 1;
        if (st->l + st->per_cycle > cap) st->restart_req = 1;
      }
    } break;
    case EPI_RESTART: {
      st->rnorm = sqrt(sums[0]);
      st->l = 0;
      st->left = 0.0;
      st->restart_req = 0;
      st->nrestart++;
      if (!isfinite(st->rnorm) && st->status == KCMG_OK) st->status = KCMG_NONFINITE;
      record(e, 4);
      set_cond(e, more_cycles(st));
    } break;
    case EPI_NORM: {
      if (e.out) *e.out = sqrt(sums[0]);
    } break;
    default: break;
  }
}

// Write this block's partial sums, and if last, reduce and run the epilogue.
template <int NC>
static __device__ __forceinline__ void finish_reduction(double (&v)[NC], double* partial, const EpiArgs& e,
                                                 double* sh) {
  bsum_n<NC>(v, sh);
  if (threadIdx.x == 0)
#pragma unroll
    for (int c = 0; c < NC; ++c) partial[(size_t)blockIdx.x * NC + c] = v[c];
  if (last_block(&e.st->ticket)) {
    __shared__ double sums[NC];
    reduce_few(partial, gridDim.x, NC, sums, sh);
    if (threadIdx.x == 0) {
      epilogue(e, sums);
      e.st->ticket = 0u;
    }
  }
}

// Start of the restart kernel that ends a loop body: true if the level restarts (the caller then
// computes the residual); otherwise the body is counted and the loop condition set.
static __device__ __forceinline__ bool restart_begin(const EpiArgs& e) {
  if (!e.st->restart_req) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      e.st->guard++;
      set_cond(e, more_cycles(e.st));
    }
    return false;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&e.st->guard, 1);
  return true;
}

}  // namespace kcmg
