// Operator application and block-Jacobi sweeps of the finest level for operators whose blocks
// have the zero pattern of a tensor basis (tensor_pattern.cuh).
//
// The dense kernels multiply every entry of a block, (S np) FMAs and (S np) stored values per
// unknown.  At np = 10 in three dimensions 160 of a cell's 700 operator entries are nonzero (at
// np = 20, 410 of 2800), so the FP64 kernels, bound by the FP64 FMA rate (two per SM and clock),
// and the FP32 kernels, bound by HBM, both do 3 to 5 times more than the operator needs.  Here
// only the pattern's entries are stored and multiplied.
//
// Layout: 32 consecutive cells form a group, one lane per cell, so every lane of a warp applies
// the same entries: the pattern is unrolled at compile time, no index is loaded and no lane
// idles, and each stored pair of entries is one coalesced 512-byte (FP64) load of the warp.
// PARTS warps share a group, each with every PARTS-th row: one warp per group leaves too few
// warps and too many registers at np >= 6 (TensorPattern::PARTS).  Neighbours' iterates are read
// straight from L1 with 16-byte loads (a cell's np values are contiguous).
//
// Measured (GB300, whole calls on device vectors): y = A x at 64^3, np = 10, FP64 355 -> 113 us
// (355: dense blocks and staged vectors); r = b - A x with its norm at 96 x 80 x 72, np = 4,
// 192 -> 108 us; five FP32 sweeps with BF16 inverses at 64^3 561 -> 231 us; the 64^3 FP64 solve's
// first five cycles 289 -> 223 ms (with the dense kernels' Alg. 1, which has changed since).
//
// Results are those of the dense kernels bit for bit: a row sees its nonzero entries in the
// dense kernels' order, and the products left out are exact zeros.  A vector entry that is
// infinite or NaN makes the dense kernels' zero products NaN; poison_rows() keeps that.
#pragma once
#include "pattern_device.cuh"

namespace kcmg {

namespace {

// y = A x or y = b - A x on the finest level, ||y||^2 with an epilogue
template <typename T, int NP, int DIM, bool RESID, bool NORM>
__global__ void __launch_bounds__(kPatThreads)
k_pat_spmv(const T* __restrict__ V, PatGrid gr, const T* __restrict__ x, T* __restrict__ y,
           const T* __restrict__ b, double* partial, EpiArgs e, int conditional) {
  constexpr int PARTS = TensorPattern<NP, DIM>::PARTS;
  if (conditional && !restart_begin(e)) return;
  __shared__ double sh[32 * 8];
  double nrm = 0.0;
  const PatLane L = pat_lane<PARTS>(gr);
  pat_dispatch<PARTS>(L.part, [&](auto Qc) {
    constexpr int Q = decltype(Qc)::value;
    using Part = typename TensorPattern<NP, DIM>::template Part<PARTS, Q>;
    T acc[Part::ROWS];
#pragma unroll
    for (int r = 0; r < Part::ROWS; ++r) acc[r] = T(0);
    if (L.group < gr.groups) pat_apply<T, NP, DIM, PARTS, Q, 0>(V, gr, L, x, acc);
    if (L.cell < gr.C) {
#pragma unroll
      for (int r = 0; r < Part::ROWS; ++r) {
        const size_t row = (size_t)L.cell * NP + Q + r * PARTS;
        const T out = RESID ? (b[row] - acc[r]) : acc[r];
        y[row] = out;
        if (NORM) nrm = fma((double)out, (double)out, nrm);
      }
    }
  });
  if (NORM) {
    double v[1] = {nrm};
    finish_reduction<1>(v, partial, e, sh);
  }
}

// r = b - A x in double-double, rounded once (as k_residual_dd); ||r||^2 with an epilogue
template <int NP, int DIM>
__global__ void __launch_bounds__(kPatThreads)
k_pat_residual_dd(const double* __restrict__ V, PatGrid gr, const double* __restrict__ x, double* __restrict__ r,
                  const double* __restrict__ b, double* partial, EpiArgs e, int conditional) {
  constexpr int PARTS = TensorPattern<NP, DIM>::PARTS;
  if (conditional && !restart_begin(e)) return;
  __shared__ double sh[32 * 8];
  double nrm = 0.0;
  const PatLane L = pat_lane<PARTS>(gr);
  pat_dispatch<PARTS>(L.part, [&](auto Qc) {
    constexpr int Q = decltype(Qc)::value;
    using Part = typename TensorPattern<NP, DIM>::template Part<PARTS, Q>;
    DD acc[Part::ROWS];
#pragma unroll
    for (int k = 0; k < Part::ROWS; ++k) acc[k] = DD{0.0, 0.0};
    if (L.group < gr.groups) pat_apply<double, NP, DIM, PARTS, Q, 0>(V, gr, L, x, acc);
    if (L.cell < gr.C) {
#pragma unroll
      for (int k = 0; k < Part::ROWS; ++k) {
        const size_t row = (size_t)L.cell * NP + Q + k * PARTS;
        double t, te;
        two_sum(b[row], -acc[k].hi, t, te);
        const double out = t + (te - acc[k].lo);
        r[row] = out;
        nrm = fma(out, out, nrm);
      }
    }
  });
  double v[1] = {nrm};
  finish_reduction<1>(v, partial, e, sh);
}

// One damped block-Jacobi sweep (Alg. BJ, as k_bj_sweep): t = r - A_off z_old (skipped when
// FIRST, z_old = 0), z_new = (1 - omega) z_old + omega D^{-1} t.  The warps of a group exchange
// their rows of t through shared memory ([mode][lane]: conflict-free); the inverse is dense.
// FP32 sweeps of an FP64 level: the first sweep rounds the FP64 residual (TR) itself and leaves
// the FP32 copy in r_lo for the others, the last writes the FP64 correction (TZ), so no pass
// over the vectors only converts them.
template <typename T, typename TI, typename TR, typename TZ, int NP, int DIM, bool FIRST>
__global__ void __launch_bounds__(kPatThreads)
k_pat_sweep(const T* __restrict__ V, const TI* __restrict__ D, PatGrid gr, const TR* __restrict__ r,
            T* __restrict__ r_lo, const T* __restrict__ zold, TZ* __restrict__ znew, double omega) {
  constexpr int PARTS = TensorPattern<NP, DIM>::PARTS;
  constexpr int GPB = kPatThreads / 32 / PARTS;
  constexpr bool SHARE = !FIRST && PARTS > 1;
  __shared__ T ts[SHARE ? GPB : 1][SHARE ? NP : 1][32];
  const PatLane L = pat_lane<PARTS>(gr);
  const bool act = L.cell < gr.C;
  T t[NP];
  if (FIRST) {
    TR tr[NP];
    load_cell<TR, NP>(r, act ? L.cell : gr.C - 1, tr);
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = (T)tr[i];
    if (!std::is_same<T, TR>::value && act) {
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (PARTS == 1 || i % PARTS == L.part) r_lo[(size_t)L.cell * NP + i] = t[i];
    }
  } else {
    pat_dispatch<PARTS>(L.part, [&](auto Qc) {
      constexpr int Q = decltype(Qc)::value;
      using Part = typename TensorPattern<NP, DIM>::template Part<PARTS, Q>;
      T acc[Part::ROWS];
#pragma unroll
      for (int k = 0; k < Part::ROWS; ++k) acc[k] = T(0);
      if (L.group < gr.groups) pat_apply<T, NP, DIM, PARTS, Q, 1>(V, gr, L, zold, acc);
#pragma unroll
      for (int k = 0; k < Part::ROWS; ++k) {
        const int i = Q + k * PARTS;
        const T tv = (act ? (T)r[(size_t)L.cell * NP + i] : T(0)) - acc[k];
        if (PARTS == 1) t[i] = tv;
        else ts[L.slot][i][L.lane] = tv;
      }
    });
    if (PARTS > 1) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < NP; ++i) t[i] = ts[L.slot][i][L.lane];
    }
  }
  if (!act) return;
  const T om = (T)omega;
  const TI* Dp = D + ((size_t)L.group * PARTS + L.part) * (TensorPattern<NP, DIM>::INV_PAIRS * 64) + 2 * L.lane;
  pat_dispatch<PARTS>(L.part, [&](auto Qc) {
    constexpr int Q = decltype(Qc)::value;
    constexpr int ROWS = (NP - Q + PARTS - 1) / PARTS;
    typename PairLoad<TI>::type d{};
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
      T dz = T(0);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const int q = k * NP + j;
        if ((q & 1) == 0) d = PairLoad<TI>::get(Dp + (q >> 1) * 64);
        dz = fma((T)((q & 1) ? d.y : d.x), t[j], dz);
      }
      const size_t row = (size_t)L.cell * NP + Q + k * PARTS;
      znew[row] = (TZ)(FIRST ? om * dz : fma(T(1) - om, zold[row], om * dz));
    }
  });
}

// residual of the no-allocation call (noalloc.cu): r = b - A x, ||r|| to *norm through the
// caller's scratch: [0, blocks) partial sums, a counter at count_at
template <int NP, int DIM, bool VEC>
__global__ void __launch_bounds__(kPatThreads)
k_pat_residual_scratch(const double* __restrict__ V, PatGrid gr, const double* __restrict__ x,
                       const double* __restrict__ b, double* __restrict__ r, double* scratch, int count_at,
                       double* norm) {
  constexpr int PARTS = TensorPattern<NP, DIM>::PARTS;
  __shared__ double sh[32 * 8];
  __shared__ int s_last;
  double nrm[1] = {0.0};
  const PatLane L = pat_lane<PARTS>(gr);
  pat_dispatch<PARTS>(L.part, [&](auto Qc) {
    constexpr int Q = decltype(Qc)::value;
    using Part = typename TensorPattern<NP, DIM>::template Part<PARTS, Q>;
    double acc[Part::ROWS];
#pragma unroll
    for (int k = 0; k < Part::ROWS; ++k) acc[k] = 0.0;
    if (L.group < gr.groups) pat_apply<double, NP, DIM, PARTS, Q, 0, VEC>(V, gr, L, x, acc);
    if (L.cell < gr.C) {
#pragma unroll
      for (int k = 0; k < Part::ROWS; ++k) {
        const size_t row = (size_t)L.cell * NP + Q + k * PARTS;
        const double out = b[row] - acc[k];
        r[row] = out;
        nrm[0] = fma(out, out, nrm[0]);
      }
    }
  });
  bsum_n<1>(nrm, sh);
  unsigned int* counter = reinterpret_cast<unsigned int*>(scratch + count_at);
  if (threadIdx.x == 0) {
    scratch[blockIdx.x] = nrm[0];
    __threadfence();
    s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (s_last) {   // last block: fixed-order sum of the partials, then reset the counter
    double t[1] = {0.0};
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t[0] += __ldcg(scratch + i);
    bsum_n<1>(t, sh);
    if (threadIdx.x == 0) {
      *norm = sqrt(t[0]);
      *counter = 0u;
    }
  }
}

// ------------------------------------------------------------------ setup
// *outside becomes nonzero if a block of nat [S][C][NP][NP] has an entry outside the pattern
// (a NaN or infinity there included).  Blocks towards a missing neighbour are not applied and
// not looked at.
template <int NP, int DIM>
__global__ void k_pat_check(const double* __restrict__ nat, const int* __restrict__ nbr, int C,
                            typename TensorPattern<NP, DIM>::Zeros zeros, int* outside) {
  constexpr int S = TensorPattern<NP, DIM>::S;
  const size_t total = (size_t)S * C * NP * NP;
  int bad = 0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int ij = (int)(e % (NP * NP)), i = ij / NP, j = ij - i * NP;
    const int K = (int)((e / (NP * NP)) % C), s = (int)(e / ((size_t)NP * NP * C));
    if (!((zeros.m[s][i] >> j) & 1u)) continue;
    if (!(nat[e] == 0.0) && (s == 0 || nbr[(size_t)K * (S - 1) + s - 1] >= 0)) bad = 1;
  }
  if (bad) atomicOr(outside, 1);
}

// one part of nat [S][C][NP][NP] -> the pattern's entries [group][part][pair][lane][2]; zero
// beyond the last cell, towards missing neighbours and in the padding
template <typename T, int NP, int DIM, typename TAB>
__global__ void k_pat_pack(const double* __restrict__ nat, const int* __restrict__ nbr, int C, int groups,
                           const __grid_constant__ TAB tab, int part, T* __restrict__ V) {
  using TP = TensorPattern<NP, DIM>;
  const size_t total = (size_t)groups * TP::PAIRS * 64;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const int lane = (int)((q >> 1) & 31), e = (int)((q >> 6) % TP::PAIRS) * 2 + (int)(q & 1);
    const size_t g = (q >> 6) / TP::PAIRS;
    const int K = (int)(g * 32) + lane;
    double v = 0.0;
    if (K < C && e < tab.n && tab.i[e] >= 0) {
      int s = 0;
      while (e >= tab.begin[s + 1]) ++s;
      if (s == 0 || nbr[(size_t)K * (TP::S - 1) + s - 1] >= 0)
        v = nat[(((size_t)s * C + K) * NP + tab.i[e]) * NP + tab.j[e]];
    }
    V[(g * TP::PARTS + part) * (TP::PAIRS * 64) + (q % (TP::PAIRS * 64))] = (T)v;
  }
}

// natural inverses [C][NP][NP] -> [group][part][pair][lane][2], the part's rows one after another
template <typename TI, int NP, int DIM>
__global__ void k_pat_pack_inverse(const double* __restrict__ inv, int C, int groups, TI* __restrict__ D) {
  constexpr int PARTS = TensorPattern<NP, DIM>::PARTS, PAIRS = TensorPattern<NP, DIM>::INV_PAIRS;
  const size_t total = (size_t)groups * PARTS * PAIRS * 64;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const int lane = (int)((q >> 1) & 31), e = (int)((q >> 6) % PAIRS) * 2 + (int)(q & 1);
    const size_t gp = (q >> 6) / PAIRS;
    const int part = (int)(gp % PARTS), K = (int)(gp / PARTS) * 32 + lane;
    const int i = part + (e / NP) * PARTS, j = e % NP;
    D[q] = (TI)((K < C && i < NP) ? inv[((size_t)K * NP + i) * NP + j] : 0.0);
  }
}

template <typename F>
bool pat_switch(int np, int dim, F&& f) {
  switch (np * 10 + dim) {
    case 32: f(std::integral_constant<int, 3>{}, std::integral_constant<int, 2>{}); return true;
    case 62: f(std::integral_constant<int, 6>{}, std::integral_constant<int, 2>{}); return true;
    case 102: f(std::integral_constant<int, 10>{}, std::integral_constant<int, 2>{}); return true;
    case 43: f(std::integral_constant<int, 4>{}, std::integral_constant<int, 3>{}); return true;
    case 103: f(std::integral_constant<int, 10>{}, std::integral_constant<int, 3>{}); return true;
    case 203: f(std::integral_constant<int, 20>{}, std::integral_constant<int, 3>{}); return true;
    default: return false;
  }
}

PatGrid pat_grid(const int* n, int dim) {
  PatGrid g;
  g.n0 = n[0];
  g.n1 = n[1];
  g.n2 = dim == 3 ? n[2] : 1;
  g.C = g.n0 * g.n1 * g.n2;
  g.groups = (g.C + 31) / 32;
  return g;
}

}  // namespace

#define KCMG_PAT(np, dim, ...)                                                      \
  pat_switch(np, dim, [&](auto NPc, auto DIMc) {                                    \
    constexpr int NP = decltype(NPc)::value, DIM = decltype(DIMc)::value;           \
    (void)DIM;                                                                      \
    __VA_ARGS__;                                                                    \
  })

template <typename T, int NP, int DIM, int Q>
static void pack_part(const double* nat, const int* nbr, int C, T* V, cudaStream_t s) {
  using TP = TensorPattern<NP, DIM>;
  if constexpr (Q < TP::PARTS) {
    static constexpr auto tab = TP::template Part<TP::PARTS, Q>::make();
    using Tab = typename TP::template Part<TP::PARTS, Q>::Tab;
    k_pat_pack<T, NP, DIM, Tab><<<152 * 8, 256, 0, s>>>(nat, nbr, C, (C + 31) / 32, tab, Q, V);
    pack_part<T, NP, DIM, Q + 1>(nat, nbr, C, V, s);
  }
}

template <typename T>
void launch_pattern_pack(int np, int dim, const double* nat, const int* nbr, int C, T* V, cudaStream_t s) {
  KCMG_PAT(np, dim, { pack_part<T, NP, DIM, 0>(nat, nbr, C, V, s); });
}

template <typename TI>
void launch_pattern_pack_inverse(int np, int dim, const double* inv, int C, TI* D, cudaStream_t s) {
  KCMG_PAT(np, dim, { k_pat_pack_inverse<TI, NP, DIM><<<152 * 8, 256, 0, s>>>(inv, C, (C + 31) / 32, D); });
}

template <typename T>
void launch_pattern_spmv(int np, int dim, const int* n, const T* V, const T* x, T* y, const T* b, double* partial,
                         const EpiArgs& e, int conditional, cudaStream_t s) {
  const PatGrid g = pat_grid(n, dim);
  const int grid = pattern_blocks(np, dim, g.C);
  const bool resid = b != nullptr, norm = e.kind != EPI_NONE;
  KCMG_PAT(np, dim, {
    if (resid && norm) k_pat_spmv<T, NP, DIM, true, true><<<grid, kPatThreads, 0, s>>>(V, g, x, y, b, partial, e, conditional);
    else if (resid) k_pat_spmv<T, NP, DIM, true, false><<<grid, kPatThreads, 0, s>>>(V, g, x, y, b, partial, e, conditional);
    else k_pat_spmv<T, NP, DIM, false, false><<<grid, kPatThreads, 0, s>>>(V, g, x, y, b, partial, e, conditional);
  });
}

template <typename T, typename TI, typename TR, typename TZ>
void launch_pattern_sweep(int np, int dim, const int* n, const T* V, const TI* D, const TR* r, T* r_lo, const T* zold,
                          TZ* znew, double omega, int first, cudaStream_t s) {
  const PatGrid g = pat_grid(n, dim);
  const int grid = pattern_blocks(np, dim, g.C);
  KCMG_PAT(np, dim, {
    if constexpr (std::is_same<TZ, T>::value)
      if (first) k_pat_sweep<T, TI, TR, TZ, NP, DIM, true><<<grid, kPatThreads, 0, s>>>(V, D, g, r, r_lo, zold, znew, omega);
    if constexpr (std::is_same<TR, T>::value)
      if (!first) k_pat_sweep<T, TI, TR, TZ, NP, DIM, false><<<grid, kPatThreads, 0, s>>>(V, D, g, r, r_lo, zold, znew, omega);
  });
}

}  // namespace kcmg
