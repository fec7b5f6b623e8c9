// Persistent cooperative kernel for the coarse part of the K-cycle: MG(lambda) of Alg. 2
// on the small levels below the finest (and, for small problems, on all levels), with the block-Jacobi smoother (Alg. BJ), residual
// minimisation (Alg. 1), transfers, the level-local criteria of Sec. 4.2 and the dense
// coarsest solve, all in one launch per finest-level cycle.
//
// Coarse levels are small (here 200-330K unknowns), so a phase is bound by latency (a grid
// barrier, an L2 round trip, a dependent chain of FP64 FMAs) and, from about 5K unknowns, by the
// FP64 FMA rate of the SMs that take part.  What follows from that:
//   - Every block owns a contiguous range of each level's cells, the same in every phase, so that
//     the work spreads over all SMs even on a level of a few hundred cells, and r, the basis W
//     and the coefficients never leave the SM: r and w are in shared memory, W is read through L1
//     (only its own block writes it).
//   - What blocks exchange is the iterate of a sweep (and r, b, x at a transfer).  Before the
//     sum, a block copies its neighbours' slabs of the iterate (the ranges shifted by the grid's
//     strides) to shared memory: one L2 round trip a phase in place of one per use.
//   - A row's products are split over several threads where a block has fewer rows than threads.
//   - One reduction per residual minimisation: W^T w, ||w||^2, w.r, ||r||^2 and the last column's
//     product with r together give the coefficients, the new column's norm (Pythagoras, guarded by
//     the reorthogonalisation test) and alpha, so the column is normalised as it is formed and no
//     second reduction is needed.
//     The next smoother's first sweep needs own rows only: no barrier in between.
//   - Corrections are stored as they come; x = sum_k y_k z_k with R y = alpha (R: the
//     orthogonalisation coefficients) is formed when the level returns or restarts, so Alg. 1's
//     second recurrence costs one pass over the corrections per visit, not one per correction.
//   - Levels too small to pay for a grid barrier run in one block while the others wait for it
//     (cc_solo_from()); a reduction sums over the blocks that have cells of the level.
//   - A small problem's finest level is part of the launch too (Alg. 2 on level 0, below), and
//     several columns of one run side by side (k_coarse_group).
//   - FP64 instructions are scarce (one of a warp takes its SM 16 clocks), so scalars are computed
//     by one warp, sums over lanes are transposed (several columns at a time) and bytes are
//     counted in integers.
// Measured (GB300, one launch; first the kernel whose blocks took whole 320-row tiles, read every
// neighbour value through L2 and reduced three times a minimisation): levels 16^3 and 8^3 at
// np = 10 beside the finest level's kernels 971 -> 553 us; 64 x 48 and two levels below at
// np = 10, 2-D, 16.7 -> 8.2 ms; 16^3 and 8^3 alone, 16 visits, 5.0 -> 2.7 ms; 192 unknowns
// 749 -> 257 us.  Whole solves: whole_solve() (engine.cu).
// Every control decision is taken by all blocks from the same reduced values (fixed reduction
// order), so all blocks follow the same path.  The grid barrier spins with a bound: if it ever
// times out it raises an error flag and every block leaves the kernel, so a fault becomes a
// status, not a hang.
#pragma once
#include "barrier_count.h"
#include "kcmg_internal.h"
#include "reduce.cuh"
#include "schwarz.cuh"

#include <cuda/atomic>

#include <cmath>

namespace kcmg {

extern __shared__ __align__(16) unsigned char smem_cc[];   // layout: CoarseArgs / CoarseLevel offsets

namespace {

template <typename T> struct V2T;
template <> struct V2T<double> { using type = double2; };
template <> struct V2T<float> { using type = float2; };

template <typename TI> __device__ __forceinline__ float2 inv_pair_f(const TI* p, size_t i);
template <> __device__ __forceinline__ float2 inv_pair_f<float>(const float* p, size_t i) {
  return __ldg(reinterpret_cast<const float2*>(p) + i);
}
template <> __device__ __forceinline__ float2 inv_pair_f<__nv_bfloat16>(const __nv_bfloat16* p, size_t i) {
  return __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(p)[i]);
}
template <typename T, typename TI> struct InvLoad {
  static __device__ __forceinline__ void get(const TI* p, size_t i, T& a, T& b) {
    const float2 v = inv_pair_f<TI>(p, i);
    a = (T)v.x;
    b = (T)v.y;
  }
};
template <> struct InvLoad<double, double> {
  static __device__ __forceinline__ void get(const double* p, size_t i, double& a, double& b) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p) + i);
    a = v.x;
    b = v.y;
  }
};

template <typename T> __device__ __forceinline__ T ldv(const T* p) { return __ldcg(p); }

}  // namespace

// Grid barrier with a bounded wait.  Every block adds one to a counter (a release, which
// publishes the block's writes, and without waiting for the old value) and polls until the
// counter reaches the total for this generation.  blocks: how many share the barrier (the grid, or
// one group of it).  gen: this block's barrier count so far in the
// launch; the last block to leave the kernel clears the counter (cc_leave), the host at the start
// of every solve.  Returns false (in every thread of the block) once the error flag is set;
// callers then leave the kernel.
static __device__ __forceinline__ bool cc_barrier(const CoarseArgs& a, unsigned int& gen, unsigned int blocks) {
  __shared__ int s_ok;
  __syncthreads();
  if (blocks == 1) return true;
  if (threadIdx.x == 0) {
    cuda::atomic_ref<unsigned int, cuda::thread_scope_device> cnt(*a.bar_count);
    cuda::atomic_ref<int, cuda::thread_scope_device> err(*a.err);
    const unsigned int target = (gen + 1) * blocks;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar_count) : "memory");
    cuda::atomic_ref<unsigned int, cuda::thread_scope_device> progress(*a.bar_progress);
    unsigned int polls = 0, seen = 0;
    int ok = 1;
    while (!count_reached(cnt.load(cuda::memory_order_acquire), target)) {
      if ((++polls & 1023) == 0) {
        if (err.load(cuda::memory_order_relaxed)) { ok = 0; break; }
        if (give_up(polls, seen, progress.load(cuda::memory_order_relaxed))) {
          err.store(1, cuda::memory_order_relaxed);
          ok = 0;
          break;
        }
      }
    }
    s_ok = ok;
  }
  ++gen;
  __syncthreads();
  return s_ok != 0;
}

// Called by every block after its last barrier: the last one clears the counters for the next
// launch.  No block polls any more, since all have passed the barrier.
static __device__ __forceinline__ void cc_leave(const CoarseArgs& a, unsigned int blocks) {
  if (blocks == 1 || threadIdx.x != 0) return;
  if (atomicAdd(a.bar_gen, 1u) == blocks - 1) {
    *a.bar_count = 0u;
    *a.bar_gen = 0u;
    __threadfence();
  }
}

namespace {

// Per-level scalars, held identically by every block.
struct LvScal {
  int l, it, first;      // first: no reduction done yet on this visit (||b|| unknown)
  double r2, eps2;       // ||r||^2 and the squared tolerance
};

// Scalars of a residual minimisation, computed by warp 0 and read by the block: FP64 instructions
// are scarce (16 clocks an SM for one of a warp), so what is the same for all threads is done once.
struct RmScal {
  double rr, naz2, gam, alp, r2new;
  int verdict;           // 0 take the correction, 1 another Gram-Schmidt pass, 2 discard it
};

// Vectors, basis W, Z, the Alg. 1 operator and the transfers are in TV (FP64, or FP32 in
// the inner solve of the iterative-refinement forms); the smoother sweeps run in TS with
// inverses stored as TI.  Reductions over lanes and blocks, norms and alpha are FP64 in every form;
// a lane's share of W^T w is summed in TV.
template <typename TV, typename TS, typename TI, int NP, int DIM, bool GROUP>
struct CoarseCycle {
  using T = TV;
  using V2 = typename V2T<TV>::type;
  using VS2 = typename V2T<TS>::type;
  static constexpr int S = 2 * DIM + 1;
  static constexpr int JP = (NP + 1) / 2;
  static constexpr int NCH = 1 << DIM;

  const CoarseArgs& a;
  double* sh;            // 32 * 8 doubles
  double* red_s;         // reduced sums, a.cols + 4
  double* cf;            // coefficients of the minimisation, a.cols
  RmScal* rms;
  int* nbs;              // neighbour slab of each slot: cell offset in the slab buffer
  long long* tph;        // clocks per phase kind, then per level (thread 0 of block 0)
  T* Ps;                 // NCH*NP*NP (prolongation matrices)
  int bid_ = 0, nall_ = 0;   // with GROUP: this block among those that share the cycle, and their number
  int rcount = 0;        // reductions done (selects the partial buffer)
  unsigned int gen = 0;  // grid barriers passed (identical in every block)
  bool ok = true;
  long long bytes = 0;   // algorithmic bytes of this launch (kept by thread 0 of block 0)

  // blocks that take part in the current level (all, or block 0 alone on the smallest levels) and
  // this block's range of it (set by enter())
  int nblk = 1, lev = 0, K0 = 0, nc = 0, rows = 0, row0 = 0;
  int lpr = 1, part = 0, lrow = 0;   // threads per row; this thread's part and row (rows < blockDim)
  int rs_off = 0;                    // residual, own rows (byte offset)
  int own0 = 0;                      // the own rows' place in the slab buffer
  double *R = nullptr, *gm = nullptr, *al = nullptr;   // packed columns of R, 1 / R_kk, alpha

  // the whole grid's: read where they are used, which keeps no registers
  __device__ int bid() const { return GROUP ? bid_ : (int)blockIdx.x; }
  __device__ int nall() const { return GROUP ? nall_ : (int)gridDim.x; }
  __device__ bool grid_bar() { return cc_barrier(a, gen, nall()); }
  // barrier of the blocks that take part in the current level
  __device__ bool bar() {
    if (nblk > 1) return grid_bar();
    __syncthreads();
    return true;
  }
  __device__ int blocks_of(int l) const { return l >= a.solo_from ? 1 : nall(); }
  __device__ void count(long long b) {
    if (bid() == 0 && threadIdx.x == 0) bytes += b;
  }
  // unique operator bytes of n slots on a level with this element size
  __device__ long long opbytes(const CoarseLevel& C, int slots, int elem) const {
    return (long long)slots * C.N * NP * elem;
  }
  __device__ const CoarseLevel& L(int l) const { return a.lv[l]; }
  __device__ T* vec(void* p) const { return static_cast<T*>(p); }
  __device__ T* zsV() const { return reinterpret_cast<T*>(smem_cc + a.sm_zv); }
  __device__ TS* zsS() const { return reinterpret_cast<TS*>(smem_cc + a.sm_zs); }
  __device__ TS* ts() const { return reinterpret_cast<TS*>(smem_cc + a.sm_ts); }
  __device__ T* ws() const { return reinterpret_cast<T*>(smem_cc + a.sm_ws); }
  __device__ T* rs_() const { return reinterpret_cast<T*>(smem_cc + rs_off); }
  __device__ double* ps() const { return reinterpret_cast<double*>(smem_cc + a.sm_ps); }

  // first of C cells of block b out of n; with fewer cells than blocks the first C have one each
  __device__ static int first_cell(int C, int b, int n) {
    n = min(n, C);
    return b >= n ? C : (int)(((long long)C * b) / n);
  }

  __device__ void enter(int l) {
    lev = l;
    nblk = blocks_of(l);
    const CoarseLevel& C = L(l);
    const int cells = C.N / NP;
    K0 = first_cell(cells, bid(), nblk);
    nc = first_cell(cells, bid() + 1, nblk) - K0;
    rows = nc * NP;
    row0 = K0 * NP;
    // threads per row: 8, 4, 2 or 1, as many as the block has
    lpr = 1;
    while (rows > 0 && lpr < 8 && 2 * lpr * rows <= (int)blockDim.x) lpr *= 2;
    part = 0;
    lrow = threadIdx.x;
    if (lpr > 1) {
      part = threadIdx.x / rows;
      lrow = threadIdx.x - part * rows;
    }
    rs_off = C.sm_r;
    gm = C.sm_gm >= 0 ? reinterpret_cast<double*>(smem_cc + C.sm_gm) : C.coef;
    al = gm + C.lcap;
    R = al + C.lcap;
    // slab buffer: [own cells with one more on each side | -y | +y | -z | +z]; one block owns all
    // cells, and its own slab, with the largest stride of zeros on each side, serves every slot
    const int pad = nblk == 1 ? (DIM == 2 ? C.n[0] : C.n[0] * C.n[1]) : 1;
    own0 = pad * NP;
    __syncthreads();
    if (threadIdx.x < S) {
      const int s = threadIdx.x, k = (s - 1) / 2, side = (s - 1) & 1;
      const int st = k == 0 ? 1 : k == 1 ? C.n[0] : C.n[0] * C.n[1];
      nbs[s] = s == 0 ? pad
               : (k == 0 || nblk == 1) ? pad + (side ? st : -st)
                                            : (nc + 2) + (2 * (k - 1) + side) * nc;
    }
    __syncthreads();
  }

  // ---------------------------------------------------------------- slabs
  // The neighbours' cells of the iterate z (global) into the slab buffer; with own: the block's
  // own cells too.  All loads of a thread are in flight together: one L2 round trip.  Cells past
  // the grid's ends read as zero.  Cells that are in range but not neighbours (across a face of
  // the grid) need no mask: a Galerkin block towards a missing neighbour is exactly zero.
  template <typename TX>
  __device__ void load_slabs(const TX* z, TX* buf, bool own) {
    const CoarseLevel& C = L(lev);
    constexpr int NS = 2 * DIM - 2;
    if (own)
      for (int i = threadIdx.x; i < rows; i += blockDim.x) buf[own0 + i] = ldv(z + row0 + i);
    if (nblk > 1) {
      const int st[2] = {C.n[0] * NP, C.n[0] * C.n[1] * NP};
      for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        TX v[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          const int g = row0 + i + (k & 1 ? st[k / 2] : -st[k / 2]);
          v[k] = (g >= 0 && g < C.N) ? ldv(z + g) : TX(0);
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) buf[(nc + 2 + k * nc) * NP + i] = v[k];
      }
      const int q = (int)blockDim.x - 1 - (int)threadIdx.x;   // the x neighbours of the range's ends
      if (q < 2 * NP) {
        const int g = q < NP ? row0 - NP + q : row0 + rows + q - NP;
        buf[q < NP ? q : (nc + 1) * NP + q - NP] = (g >= 0 && g < C.N) ? ldv(z + g) : TX(0);
      }
    } else {   // one block: zeros on both sides (the transfers use the buffer too)
      for (int i = threadIdx.x; i < own0; i += blockDim.x) buf[i] = buf[own0 + rows + i] = TX(0);
    }
    __syncthreads();
  }

  // pairs of operator entries of a row over slots FROM.. and how many a thread takes with LPR
  // threads a row; with eight they are kept in registers over the sweeps of a smoother call
  template <int FROM, int LPR> struct Trips { static constexpr int N = ((S - FROM) * JP + LPR - 1) / LPR; };
  static constexpr int kKeep = Trips<1, 8>::N;

  template <typename TX, int FROM, int LPR, int B, int U>
  __device__ __forceinline__ void load_pairs(const void* Aop, int lr, int q, typename V2T<TX>::type (&av)[U]) const {
    using VX = typename V2T<TX>::type;
    const CoarseLevel& C = L(lev);
    const int row = row0 + lr, g = row >> 5, lane = row & 31;
    const VX* Ap = reinterpret_cast<const VX*>(Aop) + (size_t)g * JP * 32 + lane;
    const size_t sl = (size_t)C.G * JP * 32;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = FROM * JP + q + (B + u) * LPR;
      if (LPR == 1 ? B + u < Trips<FROM, LPR>::N : e < S * JP) {
        const int s = e / JP, jp = e - s * JP;
        av[u] = __ldg(Ap + s * sl + jp * 32);
      } else {
        av[u].x = TX(0);
        av[u].y = TX(0);
      }
    }
  }
  template <typename TX, int FROM, int LPR, int B, int U>
  __device__ __forceinline__ void apply_pairs(const TX* buf, int c, int q, const typename V2T<TX>::type (&av)[U],
                                              TX (&acc)[4]) const {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = FROM * JP + q + (B + u) * LPR;
      if (LPR == 1 ? B + u < Trips<FROM, LPR>::N : e < S * JP) {
        const int s = e / JP, jp = e - s * JP, k = LPR >= 4 ? 0 : (u & 1) << 1;   // chains
        const TX* zp = buf + (nbs[s] + c) * NP + 2 * jp;
        acc[k] = fma(av[u].x, zp[0], acc[k]);
        if (NP % 2 == 0 || jp + 1 < JP) acc[k + 1] = fma(av[u].y, zp[1], acc[k + 1]);
      }
    }
  }
  // sum over slots FROM.. of A_{K,s} z_{nbr(K,s)} for own row lr: this thread's share
  template <typename TX, int FROM, int LPR, int B = 0>
  __device__ __forceinline__ void row_share(const void* Aop, const TX* buf, int lr, int q, TX (&acc)[4]) const {
    constexpr int T0 = Trips<FROM, LPR>::N, U = T0 - B < 8 ? T0 - B : 8;
    typename V2T<TX>::type av[U];
    load_pairs<TX, FROM, LPR, B, U>(Aop, lr, q, av);
    apply_pairs<TX, FROM, LPR, B, U>(buf, lr / NP, q, av, acc);
    if constexpr (B + U < T0) row_share<TX, FROM, LPR, B + U>(Aop, buf, lr, q, acc);
  }

  // f(own row, sum) in one thread per row, over slots FROM..; ends with every thread past the
  // reads of the slab buffer
  template <typename TX, int FROM, int LPR, typename F>
  __device__ __forceinline__ void for_rows_l(const void* Aop, const TX* buf, F&& f) {
    TX* p = reinterpret_cast<TX*>(ps());
    if (part < LPR) {
      TX acc[4] = {TX(0), TX(0), TX(0), TX(0)};
      row_share<TX, FROM, LPR>(Aop, buf, lrow, part, acc);
      p[part * rows + lrow] = LPR >= 4 ? acc[0] + acc[1] : (acc[0] + acc[1]) + (acc[2] + acc[3]);
    }
    sum_shares<TX, LPR>(f);
  }
  template <typename TX, int LPR, typename F>
  __device__ __forceinline__ void sum_shares(F&& f) {
    const TX* p = reinterpret_cast<const TX*>(ps());
    __syncthreads();
    if (threadIdx.x < rows) {
      TX v[LPR];
#pragma unroll
      for (int q = 0; q < LPR; ++q) v[q] = p[q * rows + threadIdx.x];
#pragma unroll
      for (int o = LPR / 2; o; o >>= 1)
#pragma unroll
        for (int q = 0; q < o; ++q) v[q] += v[q + o];
      f((int)threadIdx.x, v[0]);
    }
  }
  template <typename TX, int FROM, typename F>
  __device__ __forceinline__ void for_rows(const void* Aop, const TX* buf, F&& f) {
    if (lpr == 1) {
      for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
        TX acc[4] = {TX(0), TX(0), TX(0), TX(0)};   // independent FMA chains (latency)
        row_share<TX, FROM, 1>(Aop, buf, lr, 0, acc);
        f(lr, (acc[0] + acc[1]) + (acc[2] + acc[3]));
      }
    } else if (lpr == 2) {
      for_rows_l<TX, FROM, 2>(Aop, buf, f);
    } else if (lpr == 4) {
      for_rows_l<TX, FROM, 4>(Aop, buf, f);
    } else {
      for_rows_l<TX, FROM, 8>(Aop, buf, f);
    }
    __syncthreads();
  }

  // ---------------------------------------------------------------- smoother
  // One sweep of Alg. BJ in TS on the own cells: t = r - A_off zo (skipped on the first sweep
  // from z = 0), zn = (1 - omega) zo + omega D^{-1} t.  The own iterate is in the slab buffer; the
  // new one goes to global memory for the neighbours and, in TO, to the slab buffer out.  With
  // KEEP > 1 the thread's operator entries are in av (KEEP threads a row).
  template <int KEEP, typename TO>
  __device__ __forceinline__ void sweep(const TS* zo, TO* zn, TO* out, bool first, const VS2 (&av)[kKeep]) {
    const CoarseLevel& C = L(lev);
    count(opbytes(C, first ? 0 : S - 1, a.smoother_bytes) + opbytes(C, 1, a.inverse_bytes) +
          (long long)C.N * (sizeof(T) + sizeof(TO) + (first ? 0 : sizeof(TS))));
    TS* t = ts();
    TS* zb = zsS();
    const T* rs = rs_();
    if (first) {
      for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) t[lr] = (TS)rs[lr];
      __syncthreads();
    } else {
      load_slabs<TS>(zo, zb, false);
      auto residual = [&](int lr, TS v) { t[lr] = (TS)rs[lr] - v; };
      if constexpr (KEEP > 1) {
        if (part < KEEP) {
          TS acc[4] = {TS(0), TS(0), TS(0), TS(0)};
          apply_pairs<TS, 1, KEEP, 0, kKeep>(zb, lrow / NP, part, av, acc);
          reinterpret_cast<TS*>(ps())[part * rows + lrow] = acc[0] + acc[1];
        }
        sum_shares<TS, KEEP>(residual);
        __syncthreads();
      } else {
        for_rows<TS, 1>(C.As, zb, residual);
      }
    }
    const TI* D = static_cast<const TI*>(C.Dinv);
    const TS om = (TS)a.omega, om1 = (TS)a.omega1;
    for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
      const int row = row0 + lr, g = row >> 5, lane = row & 31, base = (lr / NP) * NP;
      TS d0s = TS(0), d1s = TS(0);
#pragma unroll
      for (int jp = 0; jp < JP; ++jp) {
        TS d0, d1;
        InvLoad<TS, TI>::get(D, ((size_t)g * JP + jp) * 32 + lane, d0, d1);
        d0s = fma(d0, t[base + 2 * jp], d0s);
        if (2 * jp + 1 < NP) d1s = fma(d1, t[base + 2 * jp + 1], d1s);
      }
      const TS dz = d0s + d1s;
      const TS v = first ? om * dz : fma(om1, zb[own0 + lr], om * dz);
      zn[row] = (TO)v;
      out[own0 + lr] = (TO)v;
    }
  }

  // Alg. AS phases on a level (schwarz.cuh): the sweep's residual in TS, both partitions'
  // patch solves (one warp per patch), and the combination z_new = z_old + omega (z_0 + z_1)
  __device__ void as_residual(const TS* zo, bool first) {
    const CoarseLevel& C = L(lev);
    count((long long)C.N * (sizeof(T) + sizeof(TS)) + (first ? 0ll : opbytes(C, S, a.smoother_bytes) + (long long)C.N * sizeof(TS)));
    TS* res = static_cast<TS*>(C.as_r);
    if (first) {
      for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) res[row0 + lr] = (TS)rs_()[lr];
    } else {
      load_slabs<TS>(zo, zsS(), true);
      for_rows<TS, 0>(C.As, zsS(), [&](int lr, TS v) { res[row0 + lr] = (TS)rs_()[lr] - v; });
    }
  }
  __device__ void as_patches() {
    const CoarseLevel& C = L(lev);
    constexpr int M = NCH * NP;
    const int np0 = as_npatch(C.n, DIM, 0), np1 = as_npatch(C.n, DIM, 1);
    count((long long)(np0 + np1) * M * M * a.inverse_bytes + (long long)(np0 + np1) * M * 2 * sizeof(TS));
    const TI* inv0 = static_cast<const TI*>(C.as_inv0);
    const TI* inv1 = static_cast<const TI*>(C.as_inv1);
    const TS* res = static_cast<const TS*>(C.as_r);
    TS* zP = static_cast<TS*>(C.as_z);
    const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    TS* prs = reinterpret_cast<TS*>(smem_cc + a.sm_as) + (size_t)warp * M;
    // a warp takes 32 rows of a patch; units over blocks first, so that few patches use every SM
    constexpr int JT = (M + 31) / 32;
    const int units = (np0 + np1) * JT;
    for (int u = bid() + nblk * warp; u < units; u += nblk * wpb) {
      const int w = u / JT, t = u - w * JT;
      if (w < np0) as_patch_rows_warp<TS, TI, NP, DIM>(C.n, 0, w, t, inv0, res, zP, prs);
      else as_patch_rows_warp<TS, TI, NP, DIM>(C.n, 1, w - np0, t, inv1, res, zP + (size_t)np0 * M, prs);
    }
  }
  template <typename TO>
  __device__ void as_combine(const TS* zo, TO* zn, TO* out, bool first) {
    const CoarseLevel& C = L(lev);
    count((long long)C.N * (2 * sizeof(TS) + sizeof(TO)));
    const int np0 = as_npatch(C.n, DIM, 0);
    const TS* zP = static_cast<const TS*>(C.as_z);
    for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
      const TO v = (TO)as_combine_row<TS, NP, DIM>(C.n, row0 + lr, zP, np0, zo, (TS)a.omega, first);
      zn[row0 + lr] = v;
      out[own0 + lr] = v;
    }
  }

  // z = BJ(r) or AS(r) from z = 0 (a.sweeps sweeps): own rows in zsV(), all rows in C.z
  __device__ __forceinline__ void smooth() {
    if (a.smoother == 1) {
      TS* sb[2] = {static_cast<TS*>(L(lev).s0), static_cast<TS*>(L(lev).s1)};
      for (int k = 0; k < a.sweeps && ok; ++k) {
        const TS* zo = sb[(k + 1) & 1];
        as_residual(zo, k == 0);
        if (!(ok = bar())) break;
        as_patches();
        if (!(ok = bar())) break;
        if (k == a.sweeps - 1) as_combine<T>(zo, vec(L(lev).z), zsV(), k == 0);
        else as_combine<TS>(zo, sb[k & 1], zsS(), k == 0);
        ok = bar();
        ph(PH_SWEEP);
      }
    } else if (lpr == 8) {
      bj_sweeps<8>();
    } else {
      bj_sweeps<1>();
    }
  }
  template <int KEEP>
  __device__ __forceinline__ void bj_sweeps() {
    const CoarseLevel& C = L(lev);
    TS* sb[2] = {static_cast<TS*>(C.s0), static_cast<TS*>(C.s1)};
    VS2 av[kKeep];
    if constexpr (KEEP > 1) {
      if (part < KEEP && a.sweeps > 1) load_pairs<TS, 1, KEEP, 0, kKeep>(C.As, lrow, part, av);
    }
    for (int k = 0; k < a.sweeps && ok; ++k) {
      const TS* zo = sb[(k + 1) & 1];
      if (k == a.sweeps - 1) sweep<KEEP, T>(zo, vec(C.z), zsV(), k == 0, av);
      else sweep<KEEP, TS>(zo, sb[k & 1], zsS(), k == 0, av);
      ok = bar();
      ph(PH_SWEEP);
    }
  }

  // ---------------------------------------------------------------- reductions
  // partial[c][b] of every block b -> red_s[0..n): few columns are summed by every block, more
  // columns by one owner each (a second barrier)
  __device__ bool reduce_cols(double* pt, int n) {
    if (nblk == 1) {   // the sums are the block's own, in red_s already
      __syncthreads();
      return true;
    }
    if (!bar()) return false;
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5, nsum = summands();
    if (n * nsum <= 4096) {
      // four columns a warp: their loads are in flight together, and the transposed sum takes
      // fewer FP64 additions than one column at a time
      for (int c0 = 4 * warp; c0 < n; c0 += 4 * nw) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = ln; b < nsum; b += 32)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            v[k] += c0 + k < n ? __ldcg(pt + (size_t)(c0 + k) * nsum + b) : 0.0;
        int k;
        const double t = warp_sum_t<4>(v, ln, k);
        if ((ln & 7) == 0 && c0 + k < n) red_s[c0 + k] = t;
      }
      __syncthreads();
      return true;
    }
    for (int c = bid() + nblk * warp; c < n; c += nblk * nw) {
      double v = 0.0;
      for (int b = ln; b < nsum; b += 32) v += __ldcg(pt + (size_t)c * nsum + b);
#pragma unroll
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (ln == 0) a.red[c] = v;
    }
    if (!bar()) return false;
    for (int c = threadIdx.x; c < n; c += blockDim.x) red_s[c] = __ldcg(a.red + c);
    __syncthreads();
    return true;
  }
  // blocks with cells of the level, the first of all: the others only keep step
  __device__ int summands() const { return min(nblk, L(lev).N / NP); }
  __device__ double* next_partial() {
    if (nblk == 1) return nullptr;   // alone: no partial sums, and the others' count must not differ
    double* pt = a.partial + (size_t)(rcount & 1) * a.partial_stride;
    rcount++;
    return pt;
  }

  // this block's sums of column c < l: W_c . w, l: w . w, l + 1: w . r, l + 2: r . r, l + 3 (l > 0):
  // W_{l-1} . r over the own rows; LPC lanes of a warp share a column.  The columns' per-thread sums are in T (coefficients of
  // the size of ||w||); those of norms and w . r are FP64 products and sums in every form.
  template <int LPC>
  __device__ void dots_lpc(const T* W, int N, int l, double* pt) {
    constexpr int CPW = 32 / LPC;
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int sub = ln / LPC, lc = ln - sub * LPC, n = sums_of(l), nsum = summands();
    const T* w = ws();
    const T* rs = rs_();
    for (int c0 = warp * CPW; c0 < n; c0 += nw * CPW) {
      const int c = c0 + sub;
      T s0 = T(0), s1 = T(0);
      double d = 0.0;
      if (sizeof(T) == 4 && c >= l && c < n) {
        const T* u = c == l + 3 ? W + (size_t)(l - 1) * N + row0 : c == l + 2 ? rs : w;
        const T* v = c == l ? w : rs;
        for (int j = lc; j < rows; j += LPC) d = fma((double)u[j], (double)v[j], d);
      } else if (c < n) {
        const T* u = c < l || c == l + 3 ? W + (size_t)(c < l ? c : l - 1) * N + row0 : c == l + 2 ? rs : w;
        const T* v = c <= l ? w : rs;
        int j = lc;
        for (; j + LPC < rows; j += 2 * LPC) {
          s0 = fma(u[j], v[j], s0);
          s1 = fma(u[j + LPC], v[j + LPC], s1);
        }
        if (j < rows) s0 = fma(u[j], v[j], s0);
      }
      d += (double)(s0 + s1);
#pragma unroll
      for (int o = LPC / 2; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      if (lc == 0 && c < n) {
        if (nblk == 1) red_s[c] = d;
        else if (rows > 0) pt[(size_t)c * nsum + bid()] = d;
      }
    }
  }
  __device__ bool dots(const T* W, int N, int l) {
    double* pt = next_partial();
    dots_lpc<8>(W, N, l, pt);   // few lanes a column: fewer FP64 instructions in the lanes' sum
    return reduce_cols(pt, sums_of(l));
  }
  __device__ static int sums_of(int l) { return l > 0 ? l + 4 : 3; }

  // v[row] - sum_c W[c][row] cf[c] -> f(own row, value), columns split over lpr threads a row
  template <typename F>
  __device__ void project(const T* W, int N, int l, const T* v, F&& f) {
    auto share = [&](int lr, int q, int np) {
      const T* Wp = W + row0 + lr;
      T s[4] = {T(0), T(0), T(0), T(0)};
      int i = q;
      for (; i + 3 * np < l; i += 4 * np)
#pragma unroll
        for (int t = 0; t < 4; ++t) s[t] = fma((T)(-cf[i + t * np]), Wp[(size_t)(i + t * np) * N], s[t]);
      for (; i < l; i += np) s[0] = fma((T)(-cf[i]), Wp[(size_t)i * N], s[0]);
      return (s[0] + s[1]) + (s[2] + s[3]);
    };
    if (lpr == 1 || l < 8) {
      for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) f(lr, v[lr] + share(lr, 0, 1));
    } else {
      T* p = reinterpret_cast<T*>(ps());
      if (part < lpr) p[part * rows + lrow] = share(lrow, part, lpr);
      __syncthreads();
      if (threadIdx.x < rows) {
        T s = p[threadIdx.x];
        for (int q = 1; q < lpr; ++q) s += p[q * rows + threadIdx.x];
        f((int)threadIdx.x, v[threadIdx.x] + s);
      }
    }
    __syncthreads();
  }

  // whether this block keeps the level's coefficients: every block in shared memory, block 0 where
  // a long basis puts them in global memory (read by all after a barrier)
  __device__ bool own_coef() const { return L(lev).sm_gm >= 0 || bid() == 0; }

  // ---------------------------------------------------------------- Alg. 1
  // with the correction zg: own rows in zsV(), all rows in zg; returns false on a barrier error
  __device__ bool rm(LvScal& sc, const T* zg) {
    const CoarseLevel& C = L(lev);
    const int N = C.N, l = sc.l;
    T* W = vec(C.W);
    T* w = ws();
    const T* zown = zsV() + own0;
    T* rs = rs_();
    load_slabs<T>(zg, zsV(), false);
    for_rows<T, 0>(C.A, zsV(), [&](int lr, T v) { w[lr] = v; });
    count(opbytes(C, S, sizeof(T)) + (long long)N * sizeof(T) * 2 + (long long)(l + 1) * N * sizeof(T));
    if (!dots(W, N, l)) return false;
    ph(PH_RM_GRAM1);
    // w_hat = w - W W^T w: its norm by Pythagoras; another pass whenever that leaves too little
    // of it (kPythagoras; classical Gram-Schmidt, "twice is enough" but for a few columns of FP32 forms)
    double* Rc = R + (size_t)l * (l - 1) / 2;
    // r is orthogonal to W but for what the last step has left of its column (epilogue.cuh, EPI_GRAM1):
    // out of r now, by the warps that do not decide, and into that step's alpha
    if (l > 0) {
      const int q = (int)blockDim.x - 1 - (int)threadIdx.x;
      const T left = (T)red_s[l + 3];
      const T* Wp = W + (size_t)(l - 1) * N + row0;
      for (int lr = q; lr < rows; lr += blockDim.x) rs[lr] = fma(-left, Wp[lr], rs[lr]);
      if (q == 0 && own_coef()) al[l - 1] += red_s[l + 3];
    }
    for (int pass = 0;; ++pass) {
      decide(l, pass);
      for (int i = threadIdx.x; i < l; i += blockDim.x) {
        cf[i] = red_s[i];
        if (own_coef()) Rc[i] = pass == 0 ? red_s[i] : Rc[i] + red_s[i];
      }
      __syncthreads();
      if (pass == 0 && sc.first) {
        sc.r2 = rms->rr;
        sc.eps2 = C.rtol * C.rtol * sc.r2;
        sc.first = 0;
      }
      if (rms->verdict != 1) break;
      project(W, N, l, w, [&](int lr, T v) { w[lr] = v; });
      count((long long)(l + 2) * N * sizeof(T) + (long long)(l + 1) * N * sizeof(T));   // apply + second dots
      if (!dots(W, N, l)) return false;
      ph(PH_RM_REORTH);
    }
    if (rms->verdict == 2) {
      sc.r2 = rms->rr;
      return true;
    }
    const T g = (T)rms->gam, al_t = (T)rms->alp;
    T* Wl = W + (size_t)l * N + row0;
    T* Zl = vec(C.Z) + (size_t)l * N + row0;
    project(W, N, l, w, [&](int lr, T v) {
      const T wv = v * g;
      Wl[lr] = wv;
      Zl[lr] = zown[lr];
      rs[lr] = fma(-al_t, wv, rs[lr]);
    });
    if (threadIdx.x == 0 && own_coef()) {
      gm[l] = rms->gam;
      al[l] = rms->alp;
    }
    count((long long)(l + 4) * N * sizeof(T));   // W columns; w, r in; new columns and r out
    // ||r - alpha w||^2 = ||r||^2 - alpha^2 for unit w with alpha = w . r; reduce the
    // updated vector explicitly only if that cancels more than four digits
    sc.l++;
    sc.r2 = rms->r2new;
    if (!(sc.r2 > 1e-4 * rms->rr) && !residual_norm(sc)) return false;
    ph(PH_RM_UPDATE);
    return true;
  }

  static constexpr int kMaxPasses = 48;   // 4^-48 < brk^2 = 1e-28
  // warp 0: the scalars of a Gram pass with l columns from red_s into rms (the caller's
  // __syncthreads publishes them)
  __device__ void decide(int l, int pass) {
    if (threadIdx.x >= 32) return;
    double hh = 0.0;
    for (int i = threadIdx.x; i < l; i += 32) hh = fma(red_s[i], red_s[i], hh);
    if (l > 0)
#pragma unroll
      for (int o = 16; o; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
    if (threadIdx.x != 0) return;
    const double n2 = red_s[l], nw2 = n2 - hh, left = pass == 0 && l > 0 ? red_s[l + 3] : 0.0;
    if (pass == 0) {
      rms->naz2 = n2;
      const double rr = red_s[l + 2] - left * left;
      rms->rr = rr < 0.0 ? 0.0 : rr;   // (a NaN stays one)
    }
    const double tiny = a.brk * a.brk * rms->naz2;
    // n2 is the sum over the vector as the passes have left it, so it tells what is rounding; every
    // pass takes at least 1 - kPythagoras of it, which ends within kMaxPasses
    int v = 0;
    if (!isfinite(nw2) || !(n2 > (pass > 0 ? tiny : 0.0))) v = 2;
    else if (l > 0 && nw2 < kPythagoras * n2) v = pass < kMaxPasses ? 1 : 2;
    else if (!(nw2 > tiny)) v = 2;
    rms->verdict = v;
    if (v == 0) {
      const double gam = rsqrt(nw2), alp = gam * (red_s[l + 1] - (l > 0 ? red_s[l - 1] * left : 0.0));
      rms->gam = gam;
      rms->alp = alp;
      rms->r2new = rms->rr - alp * alp;
    }
  }

  // sc.r2 = ||r||^2 from the own rows of every block
  __device__ bool residual_norm(LvScal& sc) {
    double* pt = next_partial();
    double s = 0.0;
    const T* rs = rs_();
    for (int j = threadIdx.x; j < rows; j += blockDim.x) s = fma((double)rs[j], (double)rs[j], s);
    double v[1] = {s};
    __syncthreads();
    bsum_n<1>(v, sh);
    if (threadIdx.x == 0 && rows > 0) *(nblk == 1 ? red_s : pt + bid()) = v[0];
    if (!reduce_cols(pt, 1)) return false;
    sc.r2 = red_s[0];
    return true;
  }

  // x += sum_k y_k z_k over the level's corrections, with R y = alpha (back substitution by one
  // warp of every block); returns false on a barrier error
  __device__ bool update_x(const LvScal& sc) {
    const CoarseLevel& C = L(lev);
    const int l = sc.l, N = C.N;
    if (C.sm_gm < 0 && !bar()) return false;
    __syncthreads();
    if (threadIdx.x < 32) {
      // coefficients in global memory are another block's: read through L2
      const bool far = C.sm_gm < 0;
      auto get = [&](const double* q) { return far ? __ldcg(q) : *q; };
      for (int i = threadIdx.x; i < l; i += 32) cf[i] = get(al + i);
      __syncwarp();
      double g = l > 0 ? get(gm + l - 1) : 0.0;
      for (int k = l - 1; k >= 0; --k) {
        const double y = cf[k] * g;
        if (k > 0) g = get(gm + k - 1);
        __syncwarp();
        const double* Rk = R + (size_t)k * (k - 1) / 2;
#pragma unroll 4
        for (int i = threadIdx.x; i < k; i += 32) cf[i] = fma(-get(Rk + i), y, cf[i]);
        if (threadIdx.x == 0) cf[k] = y;
        __syncwarp();
      }
    }
    __syncthreads();
    const T* Z = vec(C.Z);
    T* x = vec(C.x);
    for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
      T s[4] = {T(0), T(0), T(0), T(0)};
      int i = 0;
      for (; i + 3 < l; i += 4)
#pragma unroll
        for (int t = 0; t < 4; ++t) s[t] = fma((T)cf[i + t], Z[(size_t)(i + t) * N + row0 + lr], s[t]);
      for (; i < l; ++i) s[0] = fma((T)cf[i], Z[(size_t)i * N + row0 + lr], s[0]);
      x[row0 + lr] = ldv(x + row0 + lr) + ((s[0] + s[1]) + (s[2] + s[3]));
    }
    count((long long)(l + 2) * N * sizeof(T));
    return true;
  }

  // ---------------------------------------------------------------- transfers
  // b of level lev + 1 = R r (own rows of that level); with start: its r = b and x = 0.  Needs
  // C.r of this level complete in global memory.
  __device__ void restrict_(bool start) {
    const CoarseLevel &F = L(lev), &C = L(lev + 1);
    count((long long)F.N * sizeof(T) + (long long)C.N * sizeof(T) * (start ? 3 : 1));
    const int cells = C.N / NP;
    const int nb = blocks_of(lev + 1);
    const int J0 = first_cell(cells, bid(), nb), nJ = first_cell(cells, bid() + 1, nb) - J0;
    const T* rf = vec(F.r);
    T* stage = zsV();   // children of the own coarse cells: [cell][child][NP]
    for (int i = threadIdx.x; i < nJ * NCH * NP; i += blockDim.x) {
      const int q = i % NP, k = (i / NP) % NCH, J = J0 + i / (NP * NCH);
      const int jx = J % C.n[0], jy = (J / C.n[0]) % C.n[1], jz = DIM == 3 ? J / (C.n[0] * C.n[1]) : 0;
      const int fx = 2 * jx + (k & 1), fy = 2 * jy + ((k >> 1) & 1), fz = DIM == 3 ? 2 * jz + ((k >> 2) & 1) : 0;
      stage[i] = ldv(rf + (size_t)(fx + F.n[0] * (fy + F.n[1] * fz)) * NP + q);
    }
    __syncthreads();
    T* rc = reinterpret_cast<T*>(smem_cc + C.sm_r);
    for (int lr = threadIdx.x; lr < nJ * NP; lr += blockDim.x) {
      const int c = lr / NP, i = lr - c * NP;
      T s[NCH];
#pragma unroll
      for (int k = 0; k < NCH; ++k) s[k] = T(0);
#pragma unroll 2
      for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int k = 0; k < NCH; ++k) s[k] = fma(Ps[(k * NP + q) * NP + i], stage[(c * NCH + k) * NP + q], s[k]);
      T v = T(0);
#pragma unroll
      for (int k = 0; k < NCH; ++k) v += s[k];
      vec(C.b)[J0 * NP + lr] = v;
      if (start) {
        rc[lr] = v;
        vec(C.x)[J0 * NP + lr] = T(0);
      }
    }
    __syncthreads();
  }

  // z = P x_{lev + 1} on the own rows: zsV() and zf
  __device__ void prolong(T* zf) {
    const CoarseLevel &F = L(lev), &C = L(lev + 1);
    count((long long)F.N * sizeof(T) + (long long)C.N * sizeof(T));
    const T* xc = vec(C.x);
    T* own = zsV() + own0;
    for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) {
      const int K = K0 + lr / NP, q = lr % NP;
      const int ix = K % F.n[0], iy = (K / F.n[0]) % F.n[1], iz = DIM == 3 ? K / (F.n[0] * F.n[1]) : 0;
      const int k = (ix & 1) | ((iy & 1) << 1) | (DIM == 3 ? ((iz & 1) << 2) : 0);
      const int J = (ix >> 1) + C.n[0] * ((iy >> 1) + C.n[1] * (iz >> 1));
      T xv[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) xv[i] = ldv(xc + (size_t)J * NP + i);
      T s = T(0);
#pragma unroll
      for (int i = 0; i < NP; ++i) s = fma(Ps[(k * NP + q) * NP + i], xv[i], s);
      zf[row0 + lr] = s;
      own[lr] = s;
    }
  }

  // x_c = A_c^{-1} b_c (FP64 dense inverse), one warp per row, rows over blocks first
  __device__ void coarse_solve(int l) {
    const CoarseLevel& C = L(l);
    count((long long)a.Nc * a.Nc * 8 + (long long)a.Nc * 2 * sizeof(T));
    const T* bc = vec(C.b);
    T* xc = vec(C.x);
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, ln = threadIdx.x & 31;
    for (int row = bid() + nblk * warp; row < a.Nc; row += nblk * nw) {
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      const double* Ar = a.Ainv + (size_t)row * a.Nc;
      int j = ln;
      for (; j + 96 < a.Nc; j += 128)
#pragma unroll
        for (int t = 0; t < 4; ++t) s[t] = fma(__ldg(Ar + j + 32 * t), (double)ldv(bc + j + 32 * t), s[t]);
      for (; j < a.Nc; j += 32) s[0] = fma(__ldg(Ar + j), (double)ldv(bc + j), s[0]);
      double v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (ln == 0) xc[row] = (T)v;
    }
  }

  // ---------------------------------------------------------------- timing
  // SM clocks per phase kind (the interval since the previous phase boundary, closing barrier
  // included) and per level, by thread 0 of block 0; the clock counter is read in a few cycles,
  // the global timer only at the kernel's ends, which give the scale
  long long t_ph = 0, t_mark = 0;
  __device__ void ph(int kind) {
    if (bid() == 0 && threadIdx.x == 0) {
      const long long t = clock64();
      if (t_ph) tph[kind] += t - t_ph;
      t_ph = t;
      if (nblk < nall()) *static_cast<volatile unsigned int*>(a.bar_progress) = (unsigned int)t;   // the others wait
    }
  }
  __device__ void mark(int l) {
    if (bid() == 0 && threadIdx.x == 0) {
      const long long t = clock64();
      if (t_mark) tph[kCoarsePhases + l] += t - t_mark;
      t_mark = t;
    }
  }

  // ---------------------------------------------------------------- Alg. 2
  // The recursion MG(lev) -> MG(lev + 1) of Alg. 2 runs as a loop over an explicit
  // per-level state (the levels form a chain, so a phase per level suffices).  On entry b, r = b
  // and x = 0 of level lev0 are set, r also in shared memory.  ||b|| comes with the first
  // reduction of a visit.
  // Level 0 is part of the kernel when the whole hierarchy is small (a.lev0 == 0): its loop, its
  // tolerance and iteration cap, the history, restarts on a compensated residual and the
  // breakdown count follow the per-step kernels (EPI_* in epilogue.cuh); its tolerance and
  // ||r0|| are set by the residual kernel before the launch.  Alg. AsyncMG's cycle runs its coarse path
  // first: it reads only the cycle-start residual, so the iterates are those of the concurrent
  // form.
  enum Phase { PRE, CORRECT, POST, STEP };   // what comes next on the level

  __device__ static void start(LvScal& sc, double rtol) {
    sc.l = 0;
    sc.it = 0;
    sc.first = 1;
    sc.r2 = rtol < 1.0 ? 1.0 : 0.0;   // stands for ||b|| > rtol ||b|| until ||b|| is known
    sc.eps2 = 0.0;
  }

  // level 0's scalars of Alg. 1 and 2 beside LvScal (identical in every block)
  struct Top { int status, breakdowns, hist_len, bodies, steps; };
  __device__ void record(Top& t, double r2, int type) {
    const LevelState* st = L(0).st;
    if (t.hist_len >= st->hist_cap || !a.hist) return;
    if (bid() == 0 && threadIdx.x == 0) {
      a.hist[t.hist_len] = sqrt(r2);
      a.hist_type[t.hist_len] = type;
    }
    ++t.hist_len;
  }

  // r = b - A x on the level (compensated on an FP64 finest level), its norm, empty basis
  __device__ bool restart(LvScal& s) {
    const CoarseLevel& C = L(lev);
    if (!update_x(s) || !bar()) return false;
    load_slabs<T>(vec(C.x), zsV(), true);
    const T* b = vec(C.b);
    if constexpr (sizeof(T) == 8) {
      if (lev == 0) {
        for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) rs_()[lr] = row_residual_dd(lr, ldv(b + row0 + lr));
        __syncthreads();
      }
    }
    if (sizeof(T) != 8 || lev > 0)
      for_rows<T, 0>(C.A, zsV(), [&](int lr, T v) { rs_()[lr] = ldv(b + row0 + lr) - v; });
    count(opbytes(C, S, sizeof(T)) + (long long)C.N * sizeof(T) * 3);
    s.l = 0;
    return residual_norm(s);
  }
  // b - A x of own row lr with products and sums in double-double, rounded once; a missing
  // neighbour's block is not applied (the finest level's blocks are the caller's)
  __device__ double row_residual_dd(int lr, double bv) const {
    const CoarseLevel& C = L(lev);
    const int c = lr / NP, K = K0 + c, row = row0 + lr, g = row >> 5, lane = row & 31;
    const double2* Ap = reinterpret_cast<const double2*>(C.A) + (size_t)g * JP * 32 + lane;
    const double* x = reinterpret_cast<const double*>(smem_cc + a.sm_zv);
    double hi = 0.0, lo = 0.0;
    for (int s = 0; s < S; ++s) {
      if (s > 0 && __ldg(C.nbr + (size_t)K * (S - 1) + s - 1) < 0) continue;
      const double* xp = x + (nbs[s] + c) * NP;
      for (int j = 0; j < NP; ++j) {
        const double2 a2 = __ldg(Ap + ((size_t)s * C.G * JP + j / 2) * 32);
        const double av = (j & 1) ? a2.y : a2.x, p = av * xp[j], pe = fma(av, xp[j], -p);
        const double sm = hi + p, bb = sm - hi;
        lo += ((hi - (sm - bb)) + (p - bb)) + pe;
        hi = sm;
      }
    }
    const double t = bv - hi, bb = t - bv;
    return t + (((bv - (t - bb)) + (-hi - bb)) - lo);
  }

  __device__ void run(int lev0) {
    LvScal sc[KCMG_MAX_LEVELS];
    int phase[KCMG_MAX_LEVELS];
    int restarts[KCMG_MAX_LEVELS];
    int guard[KCMG_MAX_LEVELS];
    for (int i = 0; i < KCMG_MAX_LEVELS; ++i) { phase[i] = PRE; restarts[i] = 0; guard[i] = 0; }
    Top top{KCMG_OK, 0, 0, 0, 0};
    mark(lev);
    ph(PH_CONTROL);
    start(sc[lev], lev0 == 0 ? 0.0 : L(lev).rtol);
    int maxit0 = 0;
    if constexpr (GROUP) {   // r = b - A x0 and its norm
      const LevelState* st = L(0).st;
      if (!(ok = restart(sc[0]))) return;
      sc[0].first = 0;
      const double n0 = sqrt(sc[0].r2), eps = fmax(st->rtol * n0, st->atol);
      sc[0].eps2 = eps * eps;
      if (!isfinite(n0)) top.status = KCMG_NONFINITE;
      maxit0 = st->maxit;
      if (bid() == 0 && threadIdx.x == 0) L(0).st->rnorm0 = n0;
    } else if (lev0 == 0) {   // set by the residual kernel
      const LevelState* st = L(0).st;
      sc[0].first = 0;
      sc[0].r2 = st->rnorm * st->rnorm;
      sc[0].eps2 = st->eps * st->eps;
      top.status = st->status;
      top.hist_len = st->hist_len;
      maxit0 = st->maxit;
    }
    // one smoother call or prolongation and one residual minimisation per pass
    while (ok) {
      const CoarseLevel& C = L(lev);
      LvScal& s = sc[lev];
      const bool top0 = lev == 0, async = top0 && a.async_smooth > 0;
      const T* z = vec(C.z);
      bool minimise = true;
      if (phase[lev] == CORRECT) {
        prolong(async ? vec(a.zc) : vec(C.z));                     // z = P z_c
        if (!(ok = bar())) break;
        ph(PH_TRANSFER);
        if (async) {
          phase[lev] = STEP;
          top.steps = 0;
          continue;
        }
      } else if (phase[lev] == STEP && top.steps == a.async_smooth) {
        z = vec(a.zc);                                             // the coarse correction closes the cycle
        for (int i = threadIdx.x; i < rows; i += blockDim.x) zsV()[own0 + i] = ldv(z + row0 + i);
      } else {
        // while ||r|| > eps (level-local criteria of Sec. 4.2)
        if (phase[lev] == PRE &&
            !(s.r2 > s.eps2 && s.it < (top0 ? maxit0 : C.maxit) && guard[lev] < (1 << 24) &&
              (!top0 || top.status == KCMG_OK))) {
          if (!top0 && bid() == 0 && threadIdx.x == 0 && C.st) {
            C.st->iters_total += s.it;
            C.st->nrestart += restarts[lev];
          }
          if (!(ok = update_x(s))) break;
          mark(lev);
          if (lev == lev0) break;
          restarts[lev] = 0;
          // x complete everywhere: the caller's blocks, of which only this one may have been here
          if (!(ok = blocks_of(lev - 1) > 1 ? grid_bar() : bar())) break;
          ph(PH_CONTROL);
          enter(lev - 1);                                          // return to the caller
          continue;
        }
        if (phase[lev] == PRE && async) minimise = false;          // the coarse path comes first
        else smooth();                                             // pre- or post-smoother
        if (!ok) break;
      }
      if (minimise) {
        const int l0 = s.l;
        if (!(ok = rm(s, z))) break;
        if (top0) {
          if (s.l > l0) {
            top.breakdowns = 0;
          } else {
            if (!isfinite(rms->naz2) && top.status == KCMG_OK) top.status = KCMG_NONFINITE;
            if (++top.breakdowns >= 2 && top.status == KCMG_OK) top.status = KCMG_BREAKDOWN;
          }
          if (!isfinite(s.r2) && top.status == KCMG_OK) top.status = KCMG_NONFINITE;
          record(top, s.r2, phase[0] == CORRECT || z != vec(C.z) ? 2 : phase[0] == POST ? 3 : 1);
        }
      }
      if (phase[lev] == PRE) {
        ++guard[lev];
        if (!top0 && s.it == 0 && s.l == 0 && !(s.r2 > 0.0)) {     // b = 0 (or not finite): x = 0
          s.r2 = 0.0;
          continue;
        }
        T* rg = vec(C.r);
        for (int lr = threadIdx.x; lr < rows; lr += blockDim.x) rg[row0 + lr] = rs_()[lr];
        if (!(ok = bar())) break;                                  // r complete everywhere
        phase[lev] = CORRECT;
        const bool direct = (lev + 1 == a.nlev - 1), alone = blocks_of(lev + 1) < nblk;
        if (!alone || bid() == 0) restrict_(!direct);         // r_c = R r
        ph(PH_TRANSFER);
        mark(lev);
        if (alone && bid() != 0) {                            // block 0 solves the rest
          if (!(ok = grid_bar())) break;
        } else if (direct) {
          const int nb = nblk;
          nblk = blocks_of(lev + 1);
          if (!(ok = bar())) break;
          coarse_solve(lev + 1);                                   // z_c = A_c \ r_c
          nblk = nb;
          if (!(ok = bar())) break;
          ph(PH_COARSEST);
          mark(lev + 1);
        } else {
          enter(lev + 1);                                          // z_c = MG(A_c, r_c, 0)
          start(sc[lev], L(lev).rtol);
          phase[lev] = PRE;
        }
      } else if (phase[lev] == CORRECT) {
        phase[lev] = POST;
      } else if (phase[lev] == STEP && top.steps < a.async_smooth) {
        ++top.steps;
      } else {
        s.it++;
        const int cap = (a.lmax > 0 && a.lmax < C.lcap) ? a.lmax : C.lcap, per = async ? a.async_smooth + 1 : 3;
        const bool converged = top0 && !(s.r2 > s.eps2) && s.l > 0;
        if (s.l + per > cap || converged) {                        // restart: r = b - A x
          if (!(ok = restart(s))) break;
          ph(PH_RESTART);
          ++restarts[lev];
          if (top0) {
            if (!isfinite(s.r2) && top.status == KCMG_OK) top.status = KCMG_NONFINITE;
            record(top, s.r2, 4);
          }
        }
        phase[lev] = PRE;
      }
    }
    if constexpr (GROUP) {   // true residual, and the column to the caller's array
      if (!ok) return;
      const int l = sc[0].l;
      sc[0].l = 0;
      if (!(ok = restart(sc[0]))) return;
      sc[0].l = l;
      for (int lr = threadIdx.x; lr < rows; lr += blockDim.x)
        a.io_x[(size_t)(row0 + lr) * a.io_stride] = (double)ldv(vec(L(0).x) + row0 + lr);
    }
    if (lev0 == 0 && ok && bid() == 0 && threadIdx.x == 0) {
      LevelState* st = L(0).st;
      st->it = sc[0].it;
      st->iters_total += sc[0].it;
      st->l = sc[0].l;
      st->rnorm = sqrt(sc[0].r2);
      st->nrestart += restarts[0];
      st->status = top.status;
      st->breakdowns = top.breakdowns;
      st->hist_len = top.hist_len;
    }
  }
};

// Registers: a bound of 512 threads allows 128, with which nothing spills; 320 threads then take
// under two thirds of the register file, so that level-0 kernels of the task-parallel cycle run
// on the same SMs beside this one.
template <typename TV, typename TS, typename TI, int NP, int DIM>
__global__ void __launch_bounds__(512) k_coarse_cycle(const __grid_constant__ CoarseArgs a) {
  using T = TV;
  __shared__ double sh[32 * 8];
  double* red_s = reinterpret_cast<double*>(smem_cc + a.sm_red);   // cols + 4 sums
  double* cf = red_s + a.cols + 4;                                  // cols coefficients
  __shared__ RmScal rms;
  __shared__ int nbs[2 * DIM + 1];
  __shared__ long long tph[kCoarsePhases + KCMG_MAX_LEVELS];
  if (threadIdx.x < kCoarsePhases + KCMG_MAX_LEVELS) tph[threadIdx.x] = 0;
  constexpr int NCH = 1 << DIM;
  T* Ps = reinterpret_cast<T*>(smem_cc);   // prolongation matrices first
  const double* P = static_cast<const double*>(a.P);   // FP64 prolongation matrices
  for (int i = threadIdx.x; i < NCH * NP * NP; i += blockDim.x) Ps[i] = (T)P[i];
  CoarseCycle<TV, TS, TI, NP, DIM, false> cc{a, sh, red_s, cf, &rms, nbs, tph, Ps};
  unsigned long long t0 = 0;
  long long c0 = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    c0 = clock64();
  }
  // start of MG on the first level: on a coarse level r = b, set by the restriction kernel with
  // x = 0; on level 0 r = b - A x0 by the residual kernel.  Blocks without a part in the first
  // level go to the end.
  if (blockIdx.x < cc.blocks_of(a.lev0)) {
    cc.enter(a.lev0);
    const CoarseLevel& C = a.lv[a.lev0];
    for (int lr = threadIdx.x; lr < cc.rows; lr += blockDim.x)
      cc.rs_()[lr] = ldv(static_cast<const T*>(a.lev0 == 0 ? C.r : C.b) + cc.row0 + lr);
    __syncthreads();
    cc.count((long long)C.N * sizeof(T));
    cc.run(a.lev0);
  }
  // device time of this launch: every block has passed the last barrier of the cycle
  if (cc.ok) cc.ok = cc.grid_bar();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    unsigned long long t1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    const double scale = (double)(t1 - t0) / (double)max(1ll, clock64() - c0);   // ns per clock
    for (int k = 0; k < kCoarsePhases; ++k) atomicAdd(a.stat_phase_ns + k, (unsigned long long)(tph[k] * scale));
    for (int l = 0; l < a.nlev; ++l)
      atomicAdd(a.stat_level_ns + l, (unsigned long long)(tph[kCoarsePhases + l] * scale));
    atomicAdd(a.stat_ns, t1 - t0);
    atomicAdd(a.stat_launches, 1ull);
    atomicAdd(a.stat_bytes, (double)cc.bytes);
  }
  cc_leave(a, gridDim.x);
}

// Several right-hand sides: group g of gb blocks solves columns g, g + groups, ... one after
// another, each as k_coarse_cycle does with the whole grid, and the groups run side by side.  A
// phase of a small level is mostly latency (a barrier, an L2 round trip), which the columns'
// phases then spend at the same time; the groups need no barrier with one another.  Measured
// (GB300) against the batched kernels, one launch a step for all columns and the loop on the host:
// 8^3, np = 10, to 1e-11, 8 columns of 19 blocks 182 -> 34 ms, 32 columns of 4 blocks 242 -> 58 ms.
template <typename TV, typename TS, typename TI, int NP, int DIM>
__global__ void __launch_bounds__(512) k_coarse_group(const CoarseArgs* __restrict__ cols, int ncol, int gb) {
  using T = TV;
  __shared__ CoarseArgs a;
  __shared__ double sh[32 * 8];
  __shared__ RmScal rms;
  __shared__ int nbs[2 * DIM + 1];
  __shared__ long long tph[kCoarsePhases + KCMG_MAX_LEVELS];
  constexpr int NCH = 1 << DIM;
  const int bid = blockIdx.x % gb, groups = gridDim.x / gb;
  T* Ps = reinterpret_cast<T*>(smem_cc);
  unsigned int gen = 0;
  for (int col = blockIdx.x / gb; col < ncol; col += groups) {
    __syncthreads();
    static_assert(sizeof(CoarseArgs) % 4 == 0, "copied in words");
    for (int i = threadIdx.x; i < (int)(sizeof(CoarseArgs) / 4); i += blockDim.x)
      reinterpret_cast<unsigned int*>(&a)[i] = reinterpret_cast<const unsigned int*>(cols + col)[i];
    if (threadIdx.x < kCoarsePhases + KCMG_MAX_LEVELS) tph[threadIdx.x] = 0;
    __syncthreads();
    const double* P = static_cast<const double*>(a.P);
    for (int i = threadIdx.x; i < NCH * NP * NP; i += blockDim.x) Ps[i] = (T)P[i];
    double* red_s = reinterpret_cast<double*>(smem_cc + a.sm_red);
    CoarseCycle<TV, TS, TI, NP, DIM, true> cc{a, sh, red_s, red_s + a.cols + 4, &rms, nbs, tph, Ps, bid, gb};
    cc.gen = gen;
    cc.enter(0);
    const CoarseLevel& C = a.lv[0];
    for (int lr = threadIdx.x; lr < cc.rows; lr += blockDim.x) {
      const size_t row = cc.row0 + lr;
      static_cast<T*>(C.b)[row] = (T)a.io_b[row * a.io_stride];
      static_cast<T*>(C.x)[row] = (T)a.io_x[row * a.io_stride];
    }
    cc.run(0);
    gen = cc.gen;
    if (!cc.ok) break;
  }
  cc_leave(a, gb);
}

}  // namespace

}  // namespace kcmg
