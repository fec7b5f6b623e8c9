// Device kernels of the K-cycle orthonormalization multigrid solve (sm_103a).
//
// Operator application, block-Jacobi sweeps, transfers, the coarsest solve, the Gram /
// residual-minimisation kernels of Alg. 1, the device-side loop control of Alg. 2 and
// the setup kernels (Galerkin product, block inverses, dense coarsest inverse).
#include "epilogue.cuh"

#include <cmath>

namespace kcmg {

// ------------------------------------------------------------------ small helpers
template <typename T> struct Vec2;
template <> struct Vec2<double> { using type = double2; };
template <> struct Vec2<float> { using type = float2; };

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename TI> struct InvPair;
template <> struct InvPair<double> {
  using type = double2;
  static __device__ __forceinline__ double2 load(const double* p, size_t i) {
    return __ldg(reinterpret_cast<const double2*>(p) + i);
  }
};
template <> struct InvPair<float> {
  using type = float2;
  static __device__ __forceinline__ float2 load(const float* p, size_t i) {
    return __ldg(reinterpret_cast<const float2*>(p) + i);
  }
};
template <> struct InvPair<__nv_bfloat16> {
  using type = float2;
  static __device__ __forceinline__ float2 load(const __nv_bfloat16* p, size_t i) {
    __nv_bfloat162 v = reinterpret_cast<const __nv_bfloat162*>(p)[i];
    return __bfloat1622float2(v);
  }
};

// ------------------------------------------------------------------ operator kernels
// y = A x (or y = b - A x), one thread per DOF row, optional ||y||^2 with an epilogue.
// conditional: run only if the level requested a restart; otherwise thread 0 of block 0
// re-evaluates the loop condition and every block returns.
// Error-free transformations for the compensated residual (Knuth's two-sum; the product
// error from a fused multiply-add).
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// r = b - A x with the products and sums of each row carried in double-double and rounded
// once: the correctly rounded residual of the FP64 iterate, so that convergence tests near
// the attainable accuracy are not decided by summation noise.  ||r||^2 with an epilogue.
template <int NP, int S>
__device__ __forceinline__ double residual_dd_row(const double* __restrict__ A, const int* __restrict__ nbr,
                                                  int G, int row, const double* __restrict__ x,
                                                  double bv) {
  constexpr int JP = (NP + 1) / 2;
  constexpr int NF = S - 1;
  const int g = row >> 5, lane = row & 31, K = row / NP;
  double hi = 0.0, lo = 0.0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int J = (s == 0) ? K : __ldg(nbr + (size_t)K * NF + s - 1);
    if (J < 0) continue;
    const double2* Ap = reinterpret_cast<const double2*>(A) + ((size_t)(s * G + g) * JP) * 32 + lane;
    const double* xp = x + (size_t)J * NP;
#pragma unroll
    for (int jp = 0; jp < JP; ++jp) {
      const double2 a = __ldg(Ap + jp * 32);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (2 * jp + q >= NP) continue;
        const double av = q ? a.y : a.x, xv = __ldg(xp + 2 * jp + q);
        const double p = av * xv, pe = fma(av, xv, -p);
        double sh, se;
        two_sum(hi, p, sh, se);
        hi = sh;
        lo += se + pe;
      }
    }
  }
  double t, te;
  two_sum(bv, -hi, t, te);
  return t + (te - lo);
}

template <int NP, int S>
__global__ void __launch_bounds__(320)
k_residual_dd(const double* __restrict__ A, const int* __restrict__ nbr, int N, int G,
              const double* __restrict__ x, double* __restrict__ r, const double* __restrict__ b,
              double* partial, EpiArgs e, int conditional) {
  if (conditional && !restart_begin(e)) return;
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  double out = 0.0;
  if (row < N) {
    out = residual_dd_row<NP, S>(A, nbr, G, row, x, b[row]);
    r[row] = out;
  }
  double v[1] = {out * out};
  finish_reduction<1>(v, partial, e, sh);
}

template <typename T, int NP, int S, bool RESID, bool NORM>
__global__ void __launch_bounds__(320)
k_spmv(const T* __restrict__ A, const int* __restrict__ nbr, int N, int G,
       const T* __restrict__ x, T* __restrict__ y, const T* __restrict__ b, double* partial,
       EpiArgs e, int conditional) {
  using V2 = typename Vec2<T>::type;
  constexpr int JP = (NP + 1) / 2;
  constexpr int NF = S - 1;
  if (conditional && !restart_begin(e)) return;
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = row >> 5, lane = row & 31;
  T acc = T(0);
  if (row < N) {
    const int K = row / NP;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int J = (s == 0) ? K : __ldg(nbr + (size_t)K * NF + s - 1);
      if (J < 0) continue;
      const V2* Ap = reinterpret_cast<const V2*>(A) + ((size_t)(s * G + g) * JP) * 32 + lane;
      const T* xp = x + (size_t)J * NP;
#pragma unroll
      for (int jp = 0; jp < JP; ++jp) {
        const V2 a = __ldg(Ap + jp * 32);
        acc = fma(a.x, __ldg(xp + 2 * jp), acc);
        if (2 * jp + 1 < NP) acc = fma(a.y, __ldg(xp + 2 * jp + 1), acc);
      }
    }
    const T out = RESID ? (b[row] - acc) : acc;
    y[row] = out;
    acc = out;
  }
  if (NORM) {
    double v[1] = {row < N ? (double)acc * (double)acc : 0.0};
    finish_reduction<1>(v, partial, e, sh);
  }
}

// One damped block-Jacobi sweep (Alg. BJ): t = r - A_off z_old (skipped on the first
// sweep from z = 0), z_new = (1 - omega) z_old + omega D^{-1} t.  A block holds whole
// cells; t is exchanged through shared memory for the inverse-block product.
template <typename T, typename TI, int NP, int S, bool FIRST>
__global__ void __launch_bounds__(320)
k_bj_sweep(const T* __restrict__ A, const TI* __restrict__ Dinv, const int* __restrict__ nbr,
           int N, int G, const T* __restrict__ r, const T* __restrict__ zold,
           T* __restrict__ znew, double omega) {
  using V2 = typename Vec2<T>::type;
  constexpr int JP = (NP + 1) / 2;
  constexpr int NF = S - 1;
  extern __shared__ unsigned char smem_raw[];
  T* ts = reinterpret_cast<T*>(smem_raw);
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  const int g = row >> 5, lane = row & 31;
  T tv = T(0);
  if (row < N) {
    tv = r[row];
    if (!FIRST) {
      const int K = row / NP;
      T acc = T(0);
#pragma unroll
      for (int s = 1; s < S; ++s) {
        const int J = __ldg(nbr + (size_t)K * NF + s - 1);
        if (J < 0) continue;
        const V2* Ap = reinterpret_cast<const V2*>(A) + ((size_t)(s * G + g) * JP) * 32 + lane;
        const T* zp = zold + (size_t)J * NP;
#pragma unroll
        for (int jp = 0; jp < JP; ++jp) {
          const V2 a = __ldg(Ap + jp * 32);
          acc = fma(a.x, zp[2 * jp], acc);
          if (2 * jp + 1 < NP) acc = fma(a.y, zp[2 * jp + 1], acc);
        }
      }
      tv -= acc;
    }
  }
  ts[threadIdx.x] = tv;
  __syncthreads();
  if (row < N) {
    const int base = (row / NP) * NP - blockIdx.x * blockDim.x;
    T dz = T(0);
#pragma unroll
    for (int jp = 0; jp < JP; ++jp) {
      const auto d = InvPair<TI>::load(Dinv, ((size_t)g * JP + jp) * 32 + lane);
      dz = fma((T)d.x, ts[base + 2 * jp], dz);
      if (2 * jp + 1 < NP) dz = fma((T)d.y, ts[base + 2 * jp + 1], dz);
    }
    const T om = (T)omega;
    znew[row] = FIRST ? om * dz : fma(T(1) - om, zold[row], om * dz);
  }
}

// ------------------------------------------------------------------ transfers
struct Dims { int n[3]; };

// r_c[J][i] = sum_k sum_a P_k[a][i] r_f[child_k(J)][a]  (R = P^T).  With b/r/x given this
// also starts the next level's MG call: b = r = r_c, x = 0, ||r_c||^2 -> MG_BEGIN.
template <typename T, typename TIN, int NP, int DIM>
__global__ void __launch_bounds__(256)
k_restrict(Dims nf, Dims nc, const T* __restrict__ P, const TIN* __restrict__ rf, T* bout,
           T* rout, T* xout, int Nc, double* partial, EpiArgs e) {
  constexpr int NCH = 1 << DIM;
  __shared__ T Ps[NCH * NP * NP];
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  for (int i = threadIdx.x; i < NCH * NP * NP; i += blockDim.x) Ps[i] = P[i];
  __syncthreads();
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  T s = T(0);
  if (row < Nc) {
    const int J = row / NP, i = row - J * NP;
    const int jx = J % nc.n[0], jy = (J / nc.n[0]) % nc.n[1], jz = DIM == 3 ? J / (nc.n[0] * nc.n[1]) : 0;
#pragma unroll
    for (int k = 0; k < NCH; ++k) {
      const int fx = 2 * jx + (k & 1), fy = 2 * jy + ((k >> 1) & 1), fz = DIM == 3 ? 2 * jz + ((k >> 2) & 1) : 0;
      const int K = fx + nf.n[0] * (fy + nf.n[1] * fz);
      const TIN* rp = rf + (size_t)K * NP;
#pragma unroll
      for (int a = 0; a < NP; ++a) s = fma(Ps[(k * NP + a) * NP + i], (T)rp[a], s);
    }
    bout[row] = s;
    if (rout) { rout[row] = s; xout[row] = T(0); }
  }
  if (e.kind != EPI_NONE) {
    double v[1] = {row < Nc ? (double)s * (double)s : 0.0};
    finish_reduction<1>(v, partial, e, sh);
  }
}

// z_f[child_k(J)][a] = sum_i P_k[a][i] z_c[J][i]
template <typename T, typename TOUT, int NP, int DIM>
__global__ void __launch_bounds__(256)
k_prolong(Dims nf, Dims nc, const T* __restrict__ P, const T* __restrict__ zc, TOUT* __restrict__ zf,
          int Nf) {
  constexpr int NCH = 1 << DIM;
  __shared__ T Ps[NCH * NP * NP];
  for (int i = threadIdx.x; i < NCH * NP * NP; i += blockDim.x) Ps[i] = P[i];
  __syncthreads();
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= Nf) return;
  const int K = row / NP, a = row - K * NP;
  const int ix = K % nf.n[0], iy = (K / nf.n[0]) % nf.n[1], iz = DIM == 3 ? K / (nf.n[0] * nf.n[1]) : 0;
  const int k = (ix & 1) | ((iy & 1) << 1) | (DIM == 3 ? ((iz & 1) << 2) : 0);
  const int J = (ix >> 1) + nc.n[0] * ((iy >> 1) + nc.n[1] * (iz >> 1));
  const T* zp = zc + (size_t)J * NP;
  T s = T(0);
#pragma unroll
  for (int i = 0; i < NP; ++i) s = fma(Ps[(k * NP + a) * NP + i], zp[i], s);
  zf[row] = (TOUT)s;
}

// x = A_c^{-1} b with the dense FP64 inverse; one warp per row.
template <typename T>
__global__ void k_coarse_gemv(const double* __restrict__ Ainv, int n, const T* __restrict__ b,
                              T* __restrict__ x) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), ln = threadIdx.x & 31;
  if (row >= n) return;
  double s = 0.0;
  for (int j = ln; j < n; j += 32) s = fma(__ldg(Ainv + (size_t)row * n + j), (double)b[j], s);
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (ln == 0) x[row] = (T)s;
}

// ------------------------------------------------------------------ Gram / RM (Alg. 1)
// partial[k][c] = sum over element chunk k of W_c . w for c < l, ||w||^2 at c = l, w . r at l + 1.
// Work items are (group of kDotCols columns) x (element chunk); the fixed grid takes them
// round-robin with K = grid / groups chunks per group, so a block reduces its sums once
// per item and the reduction order depends only on N, l and the grid.  With PAIR (N even)
// a thread takes two consecutive elements per step with one 16-byte (FP64) or 8-byte
// (FP32) load per column.  The last partial column group reads a valid column in place of
// the missing ones and drops those sums, so every step issues the same FMAs (no
// predicated arithmetic).  ||w||^2 and w . r ride with group 0 as separate accumulators.
constexpr int kDotCols = 8;

template <typename T> struct Pair;
template <> struct Pair<double> { using type = double2; };
template <> struct Pair<float> { using type = float2; };

template <typename T, bool PAIR, bool NORM>
__device__ __forceinline__ void dots_item(const T* __restrict__ W, int N, const T* __restrict__ w,
                                          const T* __restrict__ r, int l, int c0, int u0, int u1,
                                          T (&acc)[kDotCols], T& ww, T& wr) {
  using T2 = typename Pair<T>::type;
  const T* Wc[kDotCols];
#pragma unroll
  for (int c = 0; c < kDotCols; ++c) Wc[c] = W + (size_t)min(c0 + c, l - 1) * N;
  for (int u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
    if (PAIR) {
      const T2 wv = __ldg(reinterpret_cast<const T2*>(w) + u);
#pragma unroll
      for (int c = 0; c < kDotCols; ++c) {
        const T2 a = __ldg(reinterpret_cast<const T2*>(Wc[c]) + u);
        acc[c] = fma(a.x, wv.x, acc[c]);
        acc[c] = fma(a.y, wv.y, acc[c]);
      }
      if (NORM) {
        const T2 rv = __ldg(reinterpret_cast<const T2*>(r) + u);
        ww = fma(wv.x, wv.x, ww);
        ww = fma(wv.y, wv.y, ww);
        wr = fma(wv.x, rv.x, wr);
        wr = fma(wv.y, rv.y, wr);
      }
    } else {
      const T wv = __ldg(w + u);
#pragma unroll
      for (int c = 0; c < kDotCols; ++c) acc[c] = fma(__ldg(Wc[c] + u), wv, acc[c]);
      if (NORM) {
        ww = fma(wv, wv, ww);
        wr = fma(wv, __ldg(r + u), wr);
      }
    }
  }
}

// At most 64 registers: two of this kernel's warps then fit an SM sub-partition beside three of
// the coarse cycle's at 128 (64K registers a SM, a quarter to each), so that in the task-parallel
// cycle it runs beside that kernel; with 68 the whole smoother path waited for its end (24^3,
// p = 3, Schwarz, m = 12, one cycle: 11.6 -> 10.0 ms).
template <typename T, bool PAIR>
__global__ void __launch_bounds__(kVecThreads, 4)
k_gram_dots(const T* __restrict__ W, int N, const T* __restrict__ w, const T* __restrict__ r, double* partial,
            EpiArgs e, int conditional) {
  LevelState* st = e.st;
  if (conditional && !(st->flags & F_REORTH)) return;
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  const int l = st->l;
  const int ncol = l + 2;
  const int groups = l > 0 ? (l + kDotCols - 1) / kDotCols : 1;   // l = 0: ||w||^2 and w . r only
  const int K = max(1, (int)gridDim.x / groups);
  const int units = PAIR ? N / 2 : N;
  const int chunk = (units + K - 1) / K;
  for (int item = blockIdx.x; item < groups * K; item += gridDim.x) {
    const int g = item / K, k = item - g * K;
    const int c0 = g * kDotCols;
    const int u0 = min(units, k * chunk), u1 = min(units, u0 + chunk);
    T acct[kDotCols];
#pragma unroll
    for (int c = 0; c < kDotCols; ++c) acct[c] = T(0);
    T ww = T(0), wr = T(0);
    if (l == 0) {
      for (int u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
        if (PAIR) {
          using T2 = typename Pair<T>::type;
          const T2 wv = __ldg(reinterpret_cast<const T2*>(w) + u), rv = __ldg(reinterpret_cast<const T2*>(r) + u);
          ww = fma(wv.x, wv.x, ww);
          ww = fma(wv.y, wv.y, ww);
          wr = fma(wv.x, rv.x, wr);
          wr = fma(wv.y, rv.y, wr);
        } else {
          const T wv = __ldg(w + u);
          ww = fma(wv, wv, ww);
          wr = fma(wv, __ldg(r + u), wr);
        }
      }
    } else if (g == 0) {
      dots_item<T, PAIR, true>(W, N, w, r, l, c0, u0, u1, acct, ww, wr);
    } else {
      dots_item<T, PAIR, false>(W, N, w, r, l, c0, u0, u1, acct, ww, wr);
    }
    // the block's sums in FP64 (FP32 vectors: FP32 products and per-thread sums)
    double acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = (double)acct[c];
    bsum_n<8>(acc, sh);
    if (threadIdx.x == 0)
#pragma unroll
      for (int c = 0; c < kDotCols; ++c)
        if (c0 + c < l) partial[(size_t)k * ncol + c0 + c] = acc[c];
    if (g == 0) {
      double v[2] = {(double)ww, (double)wr};
      bsum_n<2>(v, sh);
      if (threadIdx.x == 0) {
        partial[(size_t)k * ncol + l] = v[0];
        partial[(size_t)k * ncol + l + 1] = v[1];
      }
    }
  }
  if (last_block(&st->ticket)) {
    // one warp per column: lanes read independent partials, then a fixed shuffle tree
    extern __shared__ double sums[];  // [ncol], then the sum of the squared coefficients
    const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int c = wid; c < ncol; c += nw) {
      double s = 0.0;
      for (int b = ln; b < K; b += 32) s += __ldcg(partial + (size_t)b * ncol + c);
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (ln == 0) sums[c] = s;
    }
    __syncthreads();
    // the coefficients and the sum of their squares, in parallel: one thread's loop over the basis
    // would take 60 clocks a column
    double* h = e.kind == EPI_GRAM2 ? e.h2 : e.h;
    for (int i = threadIdx.x; i < l; i += blockDim.x) h[i] = sums[i];
    if (wid == 0) {
      double hh = 0.0;
      for (int i = ln; i < l; i += 32) hh = fma(sums[i], sums[i], hh);
#pragma unroll
      for (int o = 16; o; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
      if (ln == 0) {
        sums[ncol] = hh;
        epilogue(e, sums);
        st->ticket = 0u;
      }
    }
  }
}

// w_out = w - W h (first pass of the reorthogonalisation; runs only when requested)
template <typename T>
__global__ void __launch_bounds__(kVecThreads)
k_gram_apply(const T* __restrict__ W, int N, const T* __restrict__ w, T* __restrict__ wout,
             const LevelState* st, const double* __restrict__ h) {
  if (!(st->flags & F_REORTH)) return;
  extern __shared__ double hs[];
  const int l = st->l;
  for (int i = threadIdx.x; i < l; i += blockDim.x) hs[i] = h[i];
  __syncthreads();
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    T s = w[j];
#pragma unroll 4
    for (int i = 0; i < l; ++i) s = fma((T)(-hs[i]), __ldg(W + (size_t)i * N + j), s);
    wout[j] = s;
  }
}

// The step of Alg. 1: w_l = gamma (w_src - W c) as column l of W, r -= alpha w_l + left w_{l-1} (what
// the last step has left of its column); ||r||^2 and w_l . r -> EPI_FINISH.  gamma and alpha are known from the Gram pass, so the column is normalised and applied
// as it is formed.  Without reorthogonalisation w_src = w, c = h; with it w_src = w' = w - W h,
// c = h2.  The correction itself is stored as it comes, with its column of R (h, or h + h2):
// A Z = W R with R_ll = 1 / gamma_l, so x follows from R y = alpha when it is needed (k_solve_y,
// k_x_update), and the second recurrence z - Z h of Alg. 1, as much FP64 work as the first, is
// gone: 64^3, np = 10, m = 12, five cycles 195.4 -> 182.7 ms.
// A discarded correction leaves W, Z, r unchanged.  With PAIR (N even) a thread takes two
// consecutive elements with one 16-byte (FP64) / 8-byte (FP32) load per column.
// With F_OWN_NORM the column is formed as it is, and the last block takes its norm and w_hat . r
// from it, normalises and applies it (own_norm): one block's bandwidth, which is rare enough not to
// matter, in place of two more launches in every minimisation.
template <typename T>
__device__ __noinline__ void own_norm(T* Wl, int N, T* r, const RmCoef& co, LevelState* st, double* sums, double* sh) {
  __shared__ double sc[3];
  double v[2] = {0.0, 0.0};
  for (int j = threadIdx.x; j < N; j += blockDim.x) {   // written by other blocks: through L2
    const double a = __ldcg(Wl + j);
    v[0] = fma(a, a, v[0]);
    v[1] = fma(a, (double)__ldcg(r + j), v[1]);
  }
  bsum_n<2>(v, sh);
  if (threadIdx.x == 0) {
    const double nw = sqrt(v[0]);
    sc[0] = sc[1] = 0.0;
    if (!isfinite(nw) || !(nw > st->brk * sqrt(st->naz2))) {
      st->flags |= F_DISCARD;
      if (!isfinite(nw) && st->level == 0) st->status = KCMG_NONFINITE;
    } else {
      st->gamma = sc[0] = 1.0 / nw;
      st->alpha = sc[1] = v[1] / nw;
      co.gm[st->l] = sc[0];
      co.al[st->l] = sc[1];
      if (st->l > 0) co.al[st->l - 1] += st->left;
    }
    sc[2] = st->left;
  }
  __syncthreads();
  if (sc[0] == 0.0) return;   // discarded: r and its norm stay
  const T gam = (T)sc[0], al = (T)sc[1], lf = (T)sc[2];
  const T* Wp = Wl - (st->l > 0 ? N : 0);
  v[0] = v[1] = 0.0;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    const T wp = lf != T(0) ? Wp[j] : T(0);
    const T a = __ldcg(Wl + j) * gam, rv = fma(-al, a, fma(-lf, wp, __ldcg(r + j)));
    Wl[j] = a;
    r[j] = rv;
    v[0] = fma((double)rv, (double)rv, v[0]);
    v[1] = fma((double)a, (double)rv, v[1]);
  }
  bsum_n<2>(v, sh);
  if (threadIdx.x == 0) {
    sums[0] = v[0];
    sums[1] = v[1];
  }
}

// Registers for six blocks an SM with FP32 vectors and four with FP64 (64^3, np = 10, l = 206: 0.92
// -> 0.59 ms with FP32 vectors, which own_norm alone would give five; 0.98 ms with FP64).
template <typename T, bool PAIR>
__global__ void __launch_bounds__(kVecThreads, sizeof(T) == 4 ? 6 : 4)
k_gram_update(T* W, T* Z, int N, const T* __restrict__ w, const T* __restrict__ wre,
              const T* __restrict__ z, RmCoef co, T* __restrict__ r, double* partial, EpiArgs e) {
  using T2 = typename Pair<T>::type;
  LevelState* st = e.st;
  extern __shared__ double cs[];  // [l]
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  const int l = st->l;
  const bool re = (st->flags & F_REORTH) != 0, keep = !(st->flags & F_DISCARD), own = (st->flags & F_OWN_NORM) != 0;
  const T gam = own ? T(1) : (T)st->gamma, al = own ? T(0) : (T)st->alpha, lf = (T)st->left;
  if (keep)
    for (int i = threadIdx.x; i < l; i += blockDim.x) {
      cs[i] = re ? e.h2[i] : e.h[i];
      if (blockIdx.x == 0) co.R[(size_t)l * (l - 1) / 2 + i] = re ? e.h[i] + e.h2[i] : e.h[i];
    }
  if (keep && blockIdx.x == 0 && threadIdx.x == 0) {
    co.gm[l] = st->gamma;
    co.al[l] = st->alpha;
    if (!own && l > 0) co.al[l - 1] += st->left;
  }
  __syncthreads();
  const T* ws = re ? wre : w;
  T* Wl = W + (size_t)l * N;
  T* Zl = Z + (size_t)l * N;
  // ||r||^2 with FP64 products and sums also of FP32 vectors (two FMAs a pair and the conversions, 2
  // clocks of an SM beside the 3 of l = 200 columns); w_l . r, itself of the size of a rounding, in T
  double r2 = 0.0;
  T wr = T(0);
  if (PAIR) {
    const int units = N / 2;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < units; u += gridDim.x * blockDim.x) {
      T2 rv = reinterpret_cast<const T2*>(r)[u];
      if (keep) {
        T2 a = __ldg(reinterpret_cast<const T2*>(ws) + u);
        reinterpret_cast<T2*>(Zl)[u] = __ldg(reinterpret_cast<const T2*>(z) + u);
        T2 wi = {T(0), T(0)};
#pragma unroll 4
        for (int i = 0; i < l; ++i) {
          wi = __ldg(reinterpret_cast<const T2*>(W + (size_t)i * N) + u);
          const T cw = (T)(-cs[i]);
          a.x = fma(cw, wi.x, a.x);
          a.y = fma(cw, wi.y, a.y);
        }
        a.x *= gam;
        a.y *= gam;
        reinterpret_cast<T2*>(Wl)[u] = a;
        if (!own) {
          rv.x = fma(-al, a.x, fma(-lf, wi.x, rv.x));
          rv.y = fma(-al, a.y, fma(-lf, wi.y, rv.y));
          reinterpret_cast<T2*>(r)[u] = rv;
        }
        wr = fma(a.x, rv.x, wr);
        wr = fma(a.y, rv.y, wr);
      }
      r2 = fma((double)rv.x, (double)rv.x, r2);
      r2 = fma((double)rv.y, (double)rv.y, r2);
    }
  } else {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
      T rv = r[j];
      if (keep) {
        T a = ws[j];
        Zl[j] = z[j];
        T wi = T(0);
#pragma unroll 4
        for (int i = 0; i < l; ++i) {
          wi = __ldg(W + (size_t)i * N + j);
          a = fma((T)(-cs[i]), wi, a);
        }
        a *= gam;
        Wl[j] = a;
        if (!own) {
          rv = fma(-al, a, fma(-lf, wi, rv));
          r[j] = rv;
        }
        wr = fma(a, rv, wr);
      }
      r2 = fma((double)rv, (double)rv, r2);
    }
  }
  double v[2] = {r2, (double)wr};
  bsum_n<2>(v, sh);
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = v[0];
    partial[2 * blockIdx.x + 1] = v[1];
  }
  if (last_block(&st->ticket)) {
    __shared__ double sums[2];
    reduce_few(partial, gridDim.x, 2, sums, sh);
    if (own && keep) own_norm<T>(Wl, N, r, co, st, sums, sh);
    if (threadIdx.x == 0) {
      epilogue(e, sums);
      st->ticket = 0u;
    }
  }
}

// R y = alpha by back substitution, one block; conditional: only if the level restarts.  One column
// of R a step, the next one's entries loaded meanwhile: about an L2 round trip a step.
constexpr int kSolveThreads = 512;
__global__ void __launch_bounds__(kSolveThreads) k_solve_y(const LevelState* st, RmCoef co, int conditional) {
  if (conditional && !st->restart_req) return;
  extern __shared__ double cf[];
  constexpr int PER = kLcapMax / kSolveThreads;
  const int l = st->l;
  for (int i = threadIdx.x; i < l; i += kSolveThreads) cf[i] = co.al[i];
  double nx[PER], g = l > 0 ? co.gm[l - 1] : 0.0;
  auto column = [&](int k) {
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int i = threadIdx.x + p * kSolveThreads;
      nx[p] = i < k ? co.R[(size_t)k * (k - 1) / 2 + i] : 0.0;
    }
  };
  if (l > 0) column(l - 1);
  __syncthreads();
  for (int k = l - 1; k >= 0; --k) {
    const double y = cf[k] * g;
    double cur[PER];
#pragma unroll
    for (int p = 0; p < PER; ++p) cur[p] = nx[p];
    if (k > 0) {
      g = co.gm[k - 1];
      column(k - 1);
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int i = threadIdx.x + p * kSolveThreads;
      if (i < k) cf[i] = fma(-cur[p], y, cf[i]);
    }
    if (threadIdx.x == 0) co.y[k] = y;
    __syncthreads();
  }
}

// x += Z y (FP64 coefficients, vectors in T)
template <typename T, bool PAIR>
__global__ void __launch_bounds__(kVecThreads)
k_x_update(const T* __restrict__ Z, int N, T* __restrict__ x, const LevelState* st, RmCoef co, int conditional) {
  using T2 = typename Pair<T>::type;
  if (conditional && !st->restart_req) return;
  extern __shared__ double ys[];
  const int l = st->l;
  if (l == 0) return;
  for (int i = threadIdx.x; i < l; i += blockDim.x) ys[i] = co.y[i];
  __syncthreads();
  const int units = PAIR ? N / 2 : N;
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < units; u += gridDim.x * blockDim.x) {
    if (PAIR) {
      T2 s = {T(0), T(0)};
#pragma unroll 4
      for (int i = 0; i < l; ++i) {
        const T2 zi = __ldg(reinterpret_cast<const T2*>(Z + (size_t)i * N) + u);
        const T y = (T)ys[i];
        s.x = fma(y, zi.x, s.x);
        s.y = fma(y, zi.y, s.y);
      }
      T2 xv = reinterpret_cast<const T2*>(x)[u];
      xv.x += s.x;
      xv.y += s.y;
      reinterpret_cast<T2*>(x)[u] = xv;
    } else {
      T s = T(0);
#pragma unroll 4
      for (int i = 0; i < l; ++i) s = fma((T)ys[i], __ldg(Z + (size_t)i * N + u), s);
      x[u] += s;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kVecThreads)
k_norm(const T* __restrict__ v, int N, double* partial, EpiArgs e) {
  __shared__ double sh[32 * 8];   // bsum_n<NC> needs 32 * NC
  double s = 0.0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
    const double a = (double)v[j];
    s = fma(a, a, s);
  }
  double vv[1] = {s};
  finish_reduction<1>(vv, partial, e, sh);
}

__global__ void k_control(EpiArgs e) { set_cond(e, more_cycles(e.st)); }

template <typename Ts, typename Td>
__global__ void k_convert(const Ts* __restrict__ a, Td* __restrict__ b, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = (Td)a[i];
}
__global__ void k_scale_to_float(const double* __restrict__ a, float* __restrict__ b, double s, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = (float)(s * a[i]);
}
__global__ void k_axpy_scaled_to_double(const float* __restrict__ e, double* __restrict__ x, double s,
                                        size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    x[i] = fma(s, (double)e[i], x[i]);
}
template <typename T>
__global__ void k_axpy_to_double(const T* __restrict__ e, double* __restrict__ x, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    x[i] += (double)e[i];
}

// ------------------------------------------------------------------ setup kernels
__global__ void k_build_nbr(int dim, Dims n, int* nbr) {
  const int C = n.n[0] * n.n[1] * (dim == 3 ? n.n[2] : 1);
  const int K = blockIdx.x * blockDim.x + threadIdx.x;
  if (K >= C) return;
  const int c[3] = {K % n.n[0], (K / n.n[0]) % n.n[1], dim == 3 ? K / (n.n[0] * n.n[1]) : 0};
  const int stride[3] = {1, n.n[0], n.n[0] * n.n[1]};
  for (int j = 0; j < dim; ++j) {
    nbr[K * 2 * dim + 2 * j] = c[j] > 0 ? K - stride[j] : -1;
    nbr[K * 2 * dim + 2 * j + 1] = c[j] < n.n[j] - 1 ? K + stride[j] : -1;
  }
}

// Galerkin product A_c = P^T A P, one block per (coarse cell, coarse slot), np*np threads.
// Contributions: every child K of J and fine slot s whose neighbour K2 lies in the coarse
// cell addressed by the coarse slot: C += P_k^T A[s][K] P_k2.
template <int NP, int DIM>
__global__ void k_galerkin(const double* __restrict__ Af, const int* __restrict__ nbrf, Dims nf,
                           Dims nc, const double* __restrict__ P, double* __restrict__ Ac) {
  constexpr int S = 2 * DIM + 1, NCH = 1 << DIM;
  __shared__ double Ps[NCH * NP * NP];
  __shared__ double Ts[NP * NP];
  const int J = blockIdx.x, cs = blockIdx.y;
  const int Cc = nc.n[0] * nc.n[1] * (DIM == 3 ? nc.n[2] : 1);
  const int Cf = nf.n[0] * nf.n[1] * (DIM == 3 ? nf.n[2] : 1);
  for (int i = threadIdx.x; i < NCH * NP * NP; i += blockDim.x) Ps[i] = P[i];
  const int ti = threadIdx.x / NP, tj = threadIdx.x % NP;
  const bool act = threadIdx.x < NP * NP;
  const int jx = J % nc.n[0], jy = (J / nc.n[0]) % nc.n[1], jz = DIM == 3 ? J / (nc.n[0] * nc.n[1]) : 0;
  double acc = 0.0;
  __syncthreads();
  for (int k = 0; k < NCH; ++k) {
    const int fx = 2 * jx + (k & 1), fy = 2 * jy + ((k >> 1) & 1), fz = DIM == 3 ? 2 * jz + ((k >> 2) & 1) : 0;
    const int K = fx + nf.n[0] * (fy + nf.n[1] * fz);
    for (int s = 0; s < S; ++s) {
      const int K2 = (s == 0) ? K : nbrf[K * (S - 1) + s - 1];
      if (K2 < 0) continue;
      const int x2 = K2 % nf.n[0], y2 = (K2 / nf.n[0]) % nf.n[1], z2 = DIM == 3 ? K2 / (nf.n[0] * nf.n[1]) : 0;
      const int J2 = (x2 >> 1) + nc.n[0] * ((y2 >> 1) + nc.n[1] * (z2 >> 1));
      const int target = (J2 == J) ? 0 : s;  // crossing a coarse face keeps the direction
      if (target != cs) continue;
      const int k2 = (x2 & 1) | ((y2 & 1) << 1) | (DIM == 3 ? ((z2 & 1) << 2) : 0);
      const double* Ab = Af + ((size_t)s * Cf + K) * NP * NP;
      // T = A_b P_k2 : T[a][j] = sum_m A[a][m] P_k2[m][j]
      if (act) {
        double t = 0.0;
        for (int m = 0; m < NP; ++m) t = fma(Ab[ti * NP + m], Ps[(k2 * NP + m) * NP + tj], t);
        Ts[ti * NP + tj] = t;
      }
      __syncthreads();
      if (act)
        for (int a = 0; a < NP; ++a) acc = fma(Ps[(k * NP + a) * NP + ti], Ts[a * NP + tj], acc);
      __syncthreads();
    }
  }
  if (act) Ac[((size_t)cs * Cc + J) * NP * NP + threadIdx.x] = acc;
}

// Gauss-Jordan inverse with partial pivoting of every diagonal block; one warp per cell,
// lane j holds columns j and j + 32 of the augmented matrix [A | I].
template <int NP>
__global__ void k_block_inverse(const double* __restrict__ diag, int ncell, double* __restrict__ inv,
                                int* fail) {
  const int K = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), ln = threadIdx.x & 31;
  if (K >= ncell) return;
  double c0[NP], c1[NP];  // column ln and column ln+32 of [A | I]
  const double* A = diag + (size_t)K * NP * NP;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int j0 = ln, j1 = ln + 32;
    c0[i] = j0 < NP ? A[i * NP + j0] : (j0 - NP == i ? 1.0 : 0.0);
    c1[i] = j1 < NP ? A[i * NP + j1] : (j1 - NP == i ? 1.0 : 0.0);
  }
  bool bad = false;
#pragma unroll
  for (int c = 0; c < NP; ++c) {
    // pivot search in column c (held by lane c in c0)
    int p = c;
    double best = -1.0;
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (i >= c && fabs(c0[i]) > best) { best = fabs(c0[i]); p = i; }
    p = __shfl_sync(0xffffffffu, p, c);
    best = __shfl_sync(0xffffffffu, best, c);
    if (!(best > 0.0)) bad = true;
    // swap rows c and p
    double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (i == c) { a0 = c0[i]; a1 = c1[i]; }
      if (i == p) { b0 = c0[i]; b1 = c1[i]; }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (i == c) { c0[i] = b0; c1[i] = b1; }
      else if (i == p) { c0[i] = a0; c1[i] = a1; }
    }
    double d = 0.0;
#pragma unroll
    for (int i = 0; i < NP; ++i) if (i == c) d = c0[i];
    d = __shfl_sync(0xffffffffu, d, c);
    const double inv_d = bad ? 0.0 : 1.0 / d;
    double pr0 = 0, pr1 = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (i == c) { c0[i] *= inv_d; c1[i] *= inv_d; pr0 = c0[i]; pr1 = c1[i]; }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const double f = __shfl_sync(0xffffffffu, c0[i], c);
      if (i != c) { c0[i] = fma(-f, pr0, c0[i]); c1[i] = fma(-f, pr1, c1[i]); }
    }
  }
  if (bad && ln == 0) atomicExch(fail, 1);
  double* out = inv + (size_t)K * NP * NP;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (ln >= NP && ln < 2 * NP) out[i * NP + ln - NP] = c0[i];
    if (ln + 32 >= NP && ln + 32 < 2 * NP) out[i * NP + ln + 32 - NP] = c1[i];
  }
}

// dense augmented matrix M = [A_c | I] (n x 2n) of the coarsest operator
__global__ void k_assemble_dense(int np, int dim, const double* __restrict__ blk,
                                 const int* __restrict__ nbr, int ncell, double* M) {
  const int n = ncell * np, S = 2 * dim + 1;
  const size_t tot = (size_t)n * 2 * n;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(idx / (2 * n)), j = (int)(idx % (2 * n));
    double v = 0.0;
    if (j >= n) {
      v = (j - n == i) ? 1.0 : 0.0;
    } else {
      const int K = i / np, a = i % np, J = j / np, m = j % np;
      for (int s = 0; s < S; ++s) {
        const int K2 = s == 0 ? K : nbr[K * (S - 1) + s - 1];
        if (K2 == J) v += blk[((size_t)s * ncell + K) * np * np + a * np + m];
      }
    }
    M[idx] = v;
  }
}

// Gauss-Jordan step c on M (n x 2n): pick the pivot, swap, scale (single block)
__global__ void k_gj_pivot(double* M, int n, int c, double* fcol, int* fail) {
  __shared__ double bv[1024];
  __shared__ int bi[1024];
  double best = -1.0;
  int p = c;
  for (int i = c + threadIdx.x; i < n; i += blockDim.x) {
    const double v = fabs(M[(size_t)i * 2 * n + c]);
    if (v > best) { best = v; p = i; }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = p;
  __syncthreads();
  for (int o = blockDim.x / 2; o; o >>= 1) {
    if (threadIdx.x < o) {
      const double v2 = bv[threadIdx.x + o];
      const int i2 = bi[threadIdx.x + o];
      if (v2 > bv[threadIdx.x] || (v2 == bv[threadIdx.x] && i2 < bi[threadIdx.x])) {
        bv[threadIdx.x] = v2;
        bi[threadIdx.x] = i2;
      }
    }
    __syncthreads();
  }
  p = bi[0];
  if (!(bv[0] > 0.0)) {
    if (threadIdx.x == 0) atomicExch(fail, 1);
    return;
  }
  for (int j = threadIdx.x; j < 2 * n; j += blockDim.x) {
    const double a = M[(size_t)c * 2 * n + j], b = M[(size_t)p * 2 * n + j];
    M[(size_t)c * 2 * n + j] = b;
    M[(size_t)p * 2 * n + j] = a;
  }
  __syncthreads();
  const double d = M[(size_t)c * 2 * n + c];
  __syncthreads();
  for (int j = threadIdx.x; j < 2 * n; j += blockDim.x) M[(size_t)c * 2 * n + j] /= d;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) fcol[i] = (i == c) ? 0.0 : M[(size_t)i * 2 * n + c];
}

// elimination of column c from every other row: M[i][j] -= f_i M[c][j]
__global__ void k_gj_elim(double* M, int n, int c, const double* __restrict__ fcol, const int* fail) {
  if (*fail) return;
  const size_t tot = (size_t)n * 2 * n;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(idx / (2 * n)), j = (int)(idx % (2 * n));
    if (i == c) continue;
    M[idx] = fma(-fcol[i], M[(size_t)c * 2 * n + j], M[idx]);
  }
}

__global__ void k_extract_inverse(const double* __restrict__ M, int n, double* Ainv) {
  const size_t tot = (size_t)n * n;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(idx / n), j = (int)(idx % n);
    Ainv[idx] = M[(size_t)i * 2 * n + n + j];
  }
}

// natural [nslot][C][np][np] FP64 -> row-interleaved T; with nbr [C][nslot - 1], blocks towards a
// missing neighbour become zero (no kernel applies them; some need not test for them then)
template <typename T>
__global__ void k_interleave(int np, int nslot, const double* __restrict__ nat, const int* __restrict__ nbr,
                             int ncell, int G,
                             T* __restrict__ out) {
  const int JP = (np + 1) / 2;
  const size_t tot = (size_t)nslot * G * JP * 64;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(idx & 1);
    const int lane = (int)((idx >> 1) & 31);
    size_t q = idx >> 6;
    const int jp = (int)(q % JP);
    q /= JP;
    const int g = (int)(q % G);
    const int s = (int)(q / G);
    const int row = g * 32 + lane, j = 2 * jp + e;
    double v = 0.0;
    if (row < ncell * np && j < np) {
      const int K = row / np, i = row % np;
      if (s == 0 || !nbr || nbr[(size_t)K * (nslot - 1) + s - 1] >= 0)
        v = nat[((size_t)s * ncell + K) * np * np + i * np + j];
    }
    out[idx] = (T)v;
  }
}

// transposed operator: out[s][K] = (in[opp(s)][nbr(K, s)])^T
__global__ void k_transpose_blocks(int np, int dim, const double* __restrict__ in,
                                   const int* __restrict__ nbr, int ncell, double* __restrict__ out) {
  const int S = 2 * dim + 1;
  const size_t tot = (size_t)S * ncell * np * np;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(idx % np), i = (int)((idx / np) % np);
    const int K = (int)((idx / ((size_t)np * np)) % ncell), s = (int)(idx / ((size_t)np * np * ncell));
    const int J = s == 0 ? K : nbr[K * (S - 1) + s - 1];
    const int opp = s == 0 ? 0 : (((s - 1) ^ 1) + 1);
    out[idx] = J < 0 ? 0.0 : in[((size_t)opp * ncell + J) * np * np + j * np + i];
  }
}

__global__ void k_count_diff(const double* __restrict__ a, const double* __restrict__ b, size_t n,
                             unsigned int* cnt) {
  unsigned int c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    c += (a[i] != b[i]);
  if (c) atomicAdd(cnt, c);
}

// g_K = -lambda^T (dA/d log nu_K) u (SWIP operator with harmonic face coefficients)
template <int NP>
__device__ double bil(const double* M, const double* l, const double* u) {
  double s = 0.0;
  for (int i = 0; i < NP; ++i) {
    double t = 0.0;
    for (int j = 0; j < NP; ++j) t = fma(M[i * NP + j], u[j], t);
    s = fma(l[i], t, s);
  }
  return s;
}
template <int NP>
__global__ void k_grad_lognu(int dim, Dims n, const double* __restrict__ nu, const double* __restrict__ V,
                             const double* __restrict__ F, const double* __restrict__ B,
                             const double* __restrict__ lam, const double* __restrict__ u, double* g) {
  const int C = n.n[0] * n.n[1] * (dim == 3 ? n.n[2] : 1);
  const int K = blockIdx.x * blockDim.x + threadIdx.x;
  if (K >= C) return;
  constexpr int BS = NP * NP;
  const int c[3] = {K % n.n[0], (K / n.n[0]) % n.n[1], dim == 3 ? K / (n.n[0] * n.n[1]) : 0};
  const int stride[3] = {1, n.n[0], n.n[0] * n.n[1]};
  const double* lK = lam + (size_t)K * NP;
  const double* uK = u + (size_t)K * NP;
  double s = bil<NP>(V, lK, uK);
  for (int k = 0; k < dim; ++k) {
    const double* Fk = F + (size_t)k * 4 * BS;
    const double* Bk = B + (size_t)k * 2 * BS;
    if (c[k] < n.n[k] - 1) {
      const int R = K + stride[k];
      const double a = nu[K], b = nu[R], dg = 2.0 * b * b / ((a + b) * (a + b));
      const double* lR = lam + (size_t)R * NP;
      const double* uR = u + (size_t)R * NP;
      s += dg * (bil<NP>(Fk, lK, uK) + bil<NP>(Fk + BS, lK, uR) + bil<NP>(Fk + 2 * BS, lR, uK) +
                 bil<NP>(Fk + 3 * BS, lR, uR));
    } else {
      s += bil<NP>(Bk + BS, lK, uK);
    }
    if (c[k] > 0) {
      const int L = K - stride[k];
      const double a = nu[K], b = nu[L], dg = 2.0 * b * b / ((a + b) * (a + b));
      const double* lL = lam + (size_t)L * NP;
      const double* uL = u + (size_t)L * NP;
      s += dg * (bil<NP>(Fk, lL, uL) + bil<NP>(Fk + BS, lL, uK) + bil<NP>(Fk + 2 * BS, lK, uL) +
                 bil<NP>(Fk + 3 * BS, lK, uK));
    } else {
      s += bil<NP>(Bk, lK, uK);
    }
  }
  g[K] = -nu[K] * s;
}

// ------------------------------------------------------------------ launchers
// total-degree DG spaces: 2-D p = 1, 2, 3 (3, 6, 10 modes); 3-D p = 1, 2, 3 (4, 10, 20)
bool np_supported(int np, int dim) {
  return dim == 2 ? (np == 3 || np == 6 || np == 10) : dim == 3 ? (np == 4 || np == 10 || np == 20) : false;
}

int block_rows_for(int np) {
  switch (np) {
    case 3: return 288;   // 3 * 96
    case 4: return 256;
    case 6: return 288;
    case 10: return 320;  // 2 * lcm(32, 10)
    case 20: return 320;
    default: return 0;
  }
}

static inline int nblocks(size_t n, int t, int cap = 4096) {
  size_t b = (n + t - 1) / t;
  if (b < 1) b = 1;
  return (int)(b > (size_t)cap ? cap : b);
}

static Dims mkdims(const int* n) { Dims d; d.n[0] = n[0]; d.n[1] = n[1]; d.n[2] = n[2]; return d; }

// dispatch over the supported (np, dim) pairs; the body sees NP, DIM and S = 2 DIM + 1
#define KCMG_ND_SWITCH(np, dim, ...)                                                      \
  switch (np * 10 + dim) {                                                                \
    case 32: { constexpr int NP = 3, DIM = 2, S = 5; (void)S; (void)DIM; __VA_ARGS__; } break;       \
    case 62: { constexpr int NP = 6, DIM = 2, S = 5; (void)S; (void)DIM; __VA_ARGS__; } break;       \
    case 102: { constexpr int NP = 10, DIM = 2, S = 5; (void)S; (void)DIM; __VA_ARGS__; } break;     \
    case 43: { constexpr int NP = 4, DIM = 3, S = 7; (void)S; (void)DIM; __VA_ARGS__; } break;       \
    case 103: { constexpr int NP = 10, DIM = 3, S = 7; (void)S; (void)DIM; __VA_ARGS__; } break;     \
    case 203: { constexpr int NP = 20, DIM = 3, S = 7; (void)S; (void)DIM; __VA_ARGS__; } break;     \
    default: break;                                                                       \
  }
#define KCMG_NP_SWITCH(np, ...)                               \
  switch (np) {                                               \
    case 3: { constexpr int NP = 3; __VA_ARGS__; } break;     \
    case 4: { constexpr int NP = 4; __VA_ARGS__; } break;     \
    case 6: { constexpr int NP = 6; __VA_ARGS__; } break;     \
    case 10: { constexpr int NP = 10; __VA_ARGS__; } break;   \
    case 20: { constexpr int NP = 20; __VA_ARGS__; } break;   \
    default: break;                                           \
  }

template <typename T>
void launch_spmv(int np, int dim, const T* A, const int* nbr, int N, int G, int rows_pad,
                 int block_rows, const T* x, T* y, const T* b, double* partial,
                 const EpiArgs& e, int conditional, cudaStream_t s) {
  const int grid = rows_pad / block_rows;
  const bool resid = b != nullptr, norm = e.kind != EPI_NONE;
  KCMG_ND_SWITCH(np, dim, {
    if (resid && norm) k_spmv<T, NP, S, true, true><<<grid, block_rows, 0, s>>>(A, nbr, N, G, x, y, b, partial, e, conditional);
    else if (resid) k_spmv<T, NP, S, true, false><<<grid, block_rows, 0, s>>>(A, nbr, N, G, x, y, b, partial, e, conditional);
    else if (norm) k_spmv<T, NP, S, false, true><<<grid, block_rows, 0, s>>>(A, nbr, N, G, x, y, b, partial, e, conditional);
    else k_spmv<T, NP, S, false, false><<<grid, block_rows, 0, s>>>(A, nbr, N, G, x, y, b, partial, e, conditional);
  });
}

void launch_residual_dd(int np, int dim, const double* A, const int* nbr, int N, int G, int rows_pad,
                        int block_rows, const double* x, double* r, const double* b, double* partial,
                        const EpiArgs& e, int conditional, cudaStream_t s) {
  const int grid = rows_pad / block_rows;
  KCMG_ND_SWITCH(np, dim, {
    k_residual_dd<NP, S><<<grid, block_rows, 0, s>>>(A, nbr, N, G, x, r, b, partial, e, conditional);
  });
}

template <typename T, typename TI>
void launch_bj_sweep(int np, int dim, const T* A, const TI* Dinv, const int* nbr, int N, int G,
                     int rows_pad, int block_rows, const T* r, const T* zold, T* znew,
                     double omega, int first, cudaStream_t s) {
  const int grid = rows_pad / block_rows;
  const size_t sm = (size_t)block_rows * sizeof(T);
  KCMG_ND_SWITCH(np, dim, {
    if (first) k_bj_sweep<T, TI, NP, S, true><<<grid, block_rows, sm, s>>>(A, Dinv, nbr, N, G, r, zold, znew, omega);
    else k_bj_sweep<T, TI, NP, S, false><<<grid, block_rows, sm, s>>>(A, Dinv, nbr, N, G, r, zold, znew, omega);
  });
}

template <typename T, typename TIN>
void launch_restrict(int np, int dim, const int* nf, const int* nc, const T* P, const TIN* rf,
                     T* b, T* r, T* x, double* partial, const EpiArgs& e, cudaStream_t s) {
  const int Nc = nc[0] * nc[1] * (dim == 3 ? nc[2] : 1) * np;
  const int grid = nblocks(Nc, 256, 1 << 30);
  KCMG_ND_SWITCH(np, dim, {
    k_restrict<T, TIN, NP, DIM><<<grid, 256, 0, s>>>(mkdims(nf), mkdims(nc), P, rf, b, r, x, Nc, partial, e);
  });
}

template <typename T, typename TOUT>
void launch_prolong(int np, int dim, const int* nf, const int* nc, const T* P, const T* zc,
                    TOUT* zf, cudaStream_t s) {
  const int Nf = nf[0] * nf[1] * (dim == 3 ? nf[2] : 1) * np;
  const int grid = nblocks(Nf, 256, 1 << 30);
  KCMG_ND_SWITCH(np, dim, {
    k_prolong<T, TOUT, NP, DIM><<<grid, 256, 0, s>>>(mkdims(nf), mkdims(nc), P, zc, zf, Nf);
  });
}

template <typename T>
void launch_coarse_gemv(const double* Ainv, int n, const T* b, T* x, cudaStream_t s) {
  const int rows_per_block = 8;
  k_coarse_gemv<T><<<(n + rows_per_block - 1) / rows_per_block, 32 * rows_per_block, 0, s>>>(Ainv, n, b, x);
}

// dynamic shared memory: the final sums (lcap + 3 doubles) or the coefficients
// (lcap doubles); lcap <= kLcapMax keeps it within the default 48 KB
template <typename T>
void launch_gram_dots(const T* W, int N, const T* w, const T* r, int lcap, int nblk, double* partial,
                      const EpiArgs& e, int conditional, cudaStream_t s) {
  const size_t sm = (lcap + 3) * sizeof(double);
  if (N % 2 == 0)   // pairs of elements: every column base is 16-byte (FP64) / 8-byte (FP32) aligned
    k_gram_dots<T, true><<<nblk, kVecThreads, sm, s>>>(W, N, w, r, partial, e, conditional);
  else
    k_gram_dots<T, false><<<nblk, kVecThreads, sm, s>>>(W, N, w, r, partial, e, conditional);
}

template <typename T>
void launch_gram_apply(const T* W, int N, const T* w, T* wout, int lcap, int nblk, LevelState* st,
                       const double* h, cudaStream_t s) {
  k_gram_apply<T><<<nblk, kVecThreads, lcap * sizeof(double), s>>>(W, N, w, wout, st, h);
}

template <typename T>
void launch_gram_update(T* W, T* Z, int N, const T* w, const T* wre, const T* z, const RmCoef& co, T* r, int lcap,
                        int nblk, double* partial, const EpiArgs& e, cudaStream_t s) {
  const size_t sm = lcap * sizeof(double);
  if (N % 2 == 0)   // pairs of elements (aligned column bases), half the grid
    k_gram_update<T, true><<<(nblk + 1) / 2, kVecThreads, sm, s>>>(W, Z, N, w, wre, z, co, r, partial, e);
  else
    k_gram_update<T, false><<<nblk, kVecThreads, sm, s>>>(W, Z, N, w, wre, z, co, r, partial, e);
}

template <typename T>
void launch_x_update(const T* Z, int N, T* x, const LevelState* st, const RmCoef& co, int lcap, int nblk,
                     int conditional, cudaStream_t s) {
  const size_t sm = lcap * sizeof(double);
  k_solve_y<<<1, kSolveThreads, sm, s>>>(st, co, conditional);
  if (N % 2 == 0)
    k_x_update<T, true><<<(nblk + 1) / 2, kVecThreads, sm, s>>>(Z, N, x, st, co, conditional);
  else
    k_x_update<T, false><<<nblk, kVecThreads, sm, s>>>(Z, N, x, st, co, conditional);
}

template <typename T>
void launch_norm(const T* v, int N, int nblk, double* partial, const EpiArgs& e, cudaStream_t s) {
  k_norm<T><<<nblk, kVecThreads, 0, s>>>(v, N, partial, e);
}

void launch_control(const EpiArgs& e, cudaStream_t s) { k_control<<<1, 1, 0, s>>>(e); }

template <typename Ts, typename Td>
void launch_convert(const Ts* src, Td* dst, size_t n, cudaStream_t s) {
  k_convert<Ts, Td><<<nblocks(n, 256), 256, 0, s>>>(src, dst, n);
}
template <typename T>
void launch_axpy_to_double(const T* e, double* x, size_t n, cudaStream_t s) {
  k_axpy_to_double<T><<<nblocks(n, 256), 256, 0, s>>>(e, x, n);
}
void launch_scale_to_float(const double* src, float* dst, double a, size_t n, cudaStream_t s) {
  k_scale_to_float<<<nblocks(n, 256), 256, 0, s>>>(src, dst, a, n);
}
void launch_axpy_scaled_to_double(const float* e, double* x, double a, size_t n, cudaStream_t s) {
  k_axpy_scaled_to_double<<<nblocks(n, 256), 256, 0, s>>>(e, x, a, n);
}

int launch_galerkin(int np, int dim, const double* Af, const int* nbrf, const int* nf,
                    const int* nc, const double* P, double* Ac, cudaStream_t s) {
  const int Cc = nc[0] * nc[1] * (dim == 3 ? nc[2] : 1);
  dim3 grid(Cc, 2 * dim + 1);
  const int threads = ((np * np + 31) / 32) * 32;
  int ok = 0;
  KCMG_ND_SWITCH(np, dim, {
    ok = 1;
    k_galerkin<NP, DIM><<<grid, threads, 0, s>>>(Af, nbrf, mkdims(nf), mkdims(nc), P, Ac);
  });
  return ok;
}

int launch_block_inverse(int np, const double* diag, int ncell, double* inv, int* fail,
                         cudaStream_t s) {
  const int wpb = 4;
  int ok = 0;
  KCMG_NP_SWITCH(np, {
    ok = 1;
    k_block_inverse<NP><<<(ncell + wpb - 1) / wpb, 32 * wpb, 0, s>>>(diag, ncell, inv, fail);
  });
  return ok;
}

void launch_dense_gj_step(double* M, int n, int c, double* fcol, int* fail, cudaStream_t s) {
  k_gj_pivot<<<1, 1024, 0, s>>>(M, n, c, fcol, fail);
  k_gj_elim<<<nblocks((size_t)n * 2 * n, 256, 2048), 256, 0, s>>>(M, n, c, fcol, fail);
}

void launch_assemble_dense(int np, int dim, const double* blk, const int* nbr, int ncell,
                           double* M, cudaStream_t s) {
  const size_t n = (size_t)ncell * np;
  k_assemble_dense<<<nblocks(n * 2 * n, 256), 256, 0, s>>>(np, dim, blk, nbr, ncell, M);
}

void launch_extract_inverse(const double* M, int n, double* Ainv, cudaStream_t s) {
  k_extract_inverse<<<nblocks((size_t)n * n, 256), 256, 0, s>>>(M, n, Ainv);
}

template <typename T>
void launch_interleave(int np, int nslot, const double* nat, const int* nbr, int ncell, int G, T* out,
                       cudaStream_t s) {
  const size_t tot = (size_t)nslot * G * ((np + 1) / 2) * 64;
  k_interleave<T><<<nblocks(tot, 256, 1 << 16), 256, 0, s>>>(np, nslot, nat, nbr, ncell, G, out);
}

void launch_transpose_blocks(int np, int dim, const double* in, const int* nbr, int ncell,
                             double* out, cudaStream_t s) {
  const size_t tot = (size_t)(2 * dim + 1) * ncell * np * np;
  k_transpose_blocks<<<nblocks(tot, 256, 1 << 16), 256, 0, s>>>(np, dim, in, nbr, ncell, out);
}

void launch_count_diff(const double* a, const double* b, size_t n, unsigned int* cnt,
                       cudaStream_t s) {
  k_count_diff<<<nblocks(n, 256, 1 << 14), 256, 0, s>>>(a, b, n, cnt);
}

void launch_build_nbr(int dim, const int* n, int* nbr, cudaStream_t s) {
  const int C = n[0] * n[1] * (dim == 3 ? n[2] : 1);
  k_build_nbr<<<nblocks(C, 256, 1 << 30), 256, 0, s>>>(dim, mkdims(n), nbr);
}

void launch_grad_lognu(int np, int dim, const int* n, const double* nu, const double* V,
                       const double* F, const double* B, const double* lam, const double* u,
                       double* g, cudaStream_t s) {
  const int C = n[0] * n[1] * (dim == 3 ? n[2] : 1);
  KCMG_NP_SWITCH(np, {
    k_grad_lognu<NP><<<nblocks(C, 128, 1 << 30), 128, 0, s>>>(dim, mkdims(n), nu, V, F, B, lam, u, g);
  });
}

// explicit instantiations
#define KCMG_INST_T(T)                                                                        \
  template void launch_spmv<T>(int, int, const T*, const int*, int, int, int, int, const T*, T*, \
                               const T*, double*, const EpiArgs&, int, cudaStream_t);            \
  template void launch_restrict<T, T>(int, int, const int*, const int*, const T*, const T*, T*,   \
                                      T*, T*, double*, const EpiArgs&, cudaStream_t);            \
  template void launch_prolong<T, T>(int, int, const int*, const int*, const T*, const T*, T*,    \
                                     cudaStream_t);                                              \
  template void launch_coarse_gemv<T>(const double*, int, const T*, T*, cudaStream_t);           \
  template void launch_gram_dots<T>(const T*, int, const T*, const T*, int, int, double*,          \
                                    const EpiArgs&, int, cudaStream_t);                          \
  template void launch_gram_apply<T>(const T*, int, const T*, T*, int, int, LevelState*,         \
                                     const double*, cudaStream_t);                               \
  template void launch_gram_update<T>(T*, T*, int, const T*, const T*, const T*, const RmCoef&, T*, int, \
                                      int, double*, const EpiArgs&, cudaStream_t);               \
  template void launch_x_update<T>(const T*, int, T*, const LevelState*, const RmCoef&, int, int, int, cudaStream_t); \
  template void launch_norm<T>(const T*, int, int, double*, const EpiArgs&, cudaStream_t);       \
  template void launch_interleave<T>(int, int, const double*, const int*, int, int, T*, cudaStream_t); \
  template void launch_axpy_to_double<T>(const T*, double*, size_t, cudaStream_t);

KCMG_INST_T(double)
KCMG_INST_T(float)
template void launch_bj_sweep<double, double>(int, int, const double*, const double*, const int*, int,
                                              int, int, int, const double*, const double*, double*,
                                              double, int, cudaStream_t);
template void launch_bj_sweep<float, float>(int, int, const float*, const float*, const int*, int, int,
                                            int, int, const float*, const float*, float*, double, int,
                                            cudaStream_t);
template void launch_bj_sweep<float, __nv_bfloat16>(int, int, const float*, const __nv_bfloat16*,
                                                    const int*, int, int, int, int, const float*,
                                                    const float*, float*, double, int, cudaStream_t);
template void launch_interleave<__nv_bfloat16>(int, int, const double*, const int*, int, int, __nv_bfloat16*,
                                               cudaStream_t);
template void launch_restrict<float, double>(int, int, const int*, const int*, const float*,
                                             const double*, float*, float*, float*, double*,
                                             const EpiArgs&, cudaStream_t);
template void launch_prolong<float, double>(int, int, const int*, const int*, const float*,
                                            const float*, double*, cudaStream_t);
template void launch_convert<double, float>(const double*, float*, size_t, cudaStream_t);
template void launch_convert<double, __nv_bfloat16>(const double*, __nv_bfloat16*, size_t, cudaStream_t);
template void launch_convert<float, double>(const float*, double*, size_t, cudaStream_t);

}  // namespace kcmg
