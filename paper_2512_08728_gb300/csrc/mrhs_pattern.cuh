// Batched operator application and block-Jacobi sweeps of the finest level for operators whose
// blocks have a tensor basis's zero pattern (tensor_pattern.cuh): the nonzero entries only, for
// every right-hand side.
//
// A lane owns one right-hand side of a cell; with up to 16 (8) right-hand sides a warp takes two
// (four) cells, so that few columns do not leave lanes idle.  A cell's entries are stored one
// after another in the order of use and read two (FP64) or four (FP32) at a time, the same
// address for all lanes of a cell; a row of the iterate is one access of the cell's lanes.  The
// FP64 kernels are bound by the FP64 FMA rate: 160 and 220 FMAs a cell and column (operator,
// sweep; np = 10, 3-D) where the dense kernels do 700; the FP32 sweep by HBM and L2.
// Measured (GB300): one level-0 cycle of 13 minimisations at 32^3 x 32 columns, FP64, 133 -> 61 ms;
// five FP32/BF16 sweeps at 48^3 x 32 as a whole call 1232 -> 788 us (staging copies and conversion
// passes gone as well), 666 us with four columns a lane (k_mpat_sweep4).
// Results are those of the dense kernels (k_mspmm64, k_msweep64, k_msweep_simt) bit for bit: a
// row sees its entries in the same order, and poison_rows() keeps what an infinity or NaN does to
// the dense kernels' zero products.
#pragma once
#include "pattern_device.cuh"

namespace kcmg {

constexpr int kMpatThreads = 128;

// entries of a cell: the pattern's (slot 0 padded to an even count), rounded up to a multiple of 4
template <int NP, int DIM> struct MPattern {
  using TP = TensorPattern<NP, DIM>;
  using Part = typename TP::template Part<1, 0>;
  static constexpr int N = Part::tab.n;
  static constexpr int STRIDE = (N + 3) / 4 * 4;
};

struct MLane { int cell, col; bool act; };
template <int RP>
static __device__ __forceinline__ MLane mpat_lane(int C, int R) {
  const int lane = threadIdx.x & 31, warp = blockIdx.x * (kMpatThreads / 32) + (threadIdx.x >> 5);
  MLane m;
  m.cell = warp * (32 / RP) + lane / RP;
  m.col = lane % RP;
  m.act = m.cell < C && m.col < R;
  return m;
}

template <typename T> static __device__ __forceinline__ void nmadd(T a, T x, T& acc) { acc = fma(-a, x, acc); }

// One slot's products for one column: acc[i] +- A[i][j] x[j]; the entries B..B+N of the cell
template <typename Part, bool NEG, typename T, typename ACC, int NP, int E>
static __device__ __forceinline__ void mpat_entry(const T* __restrict__ Vc, typename PairLoad<T>::type& d,
                                                  const T (&xv)[NP], ACC (&acc)[NP], int first) {
  constexpr int I = Part::tab.i[E], J = Part::tab.j[E];
  if ((E & 1) == 0 || E == first) d = PairLoad<T>::get(Vc + (E & ~1));
  if constexpr (I >= 0) {
    const T v = (E & 1) ? d.y : d.x;
    if constexpr (NEG) nmadd(v, xv[J], acc[I]);
    else madd(v, xv[J], acc[I]);
  }
}
template <typename Part, bool NEG, int B, typename T, typename ACC, int NP, int... E>
static __device__ __forceinline__ void mpat_entries(std::integer_sequence<int, E...>, const T* __restrict__ Vc,
                                                    typename PairLoad<T>::type& d, const T (&xv)[NP],
                                                    ACC (&acc)[NP], int first) {
  (mpat_entry<Part, NEG, T, ACC, NP, B + E>(Vc, d, xv, acc, first), ...);
}

// rows of a cell whose zero entries meet an infinity or NaN in column x (row stride R)
template <typename T, int NP, int DIM, int FROM>
static __device__ __noinline__ unsigned mpat_poison(const T* x, PatGrid g, int K, int c0, int c1, int c2, int R) {
  const auto m = TensorPattern<NP, DIM>::make_modes();
  unsigned rows = 0;
  for (int s = FROM; s < 2 * DIM + 1; ++s) {
    const int J = pat_neighbour<DIM>(g, K, c0, c1, c2, s);
    if (J < 0) continue;
    unsigned bad = 0;
    for (int j = 0; j < NP; ++j)
      if (mag_bits(x[((size_t)J * NP + j) * R]) >= Nonfinite<T>::FROM) bad |= 1u << j;
    for (int i = 0; i < NP && bad; ++i)
      for (int j = 0; j < NP; ++j)
        if ((bad >> j & 1u) && !TensorPattern<NP, DIM>::nz(m, s, i, j)) rows |= 1u << i;
  }
  return rows;
}

// acc[i] +- (A x) of the lane's cell and column over slots FROM..
template <typename T, int NP, int DIM, int FROM, bool NEG, typename ACC>
static __device__ __forceinline__ void mpat_apply(const T* __restrict__ V, const PatGrid& g, int K, int R,
                                                  const T* __restrict__ x /* + column */, ACC (&acc)[NP]) {
  using MP = MPattern<NP, DIM>;
  using Part = typename MP::Part;
  const T* Vc = V + (size_t)K * MP::STRIDE;
  const int q0 = (unsigned)K / (unsigned)g.n0, c0 = K - q0 * g.n0;
  const int c2 = DIM == 3 ? (unsigned)q0 / (unsigned)g.n1 : 0, c1 = DIM == 3 ? q0 - c2 * g.n1 : q0;
  typename PairLoad<T>::type d{};
  int mag = 0;
  auto slot = [&](auto sc) {
    constexpr int s = decltype(sc)::value;
    if constexpr (s >= FROM && s < MP::TP::S) {
      const int J = pat_neighbour<DIM>(g, K, c0, c1, c2, s);
      if (J >= 0) {
        T xv[NP];
        const T* xp = x + (size_t)J * NP * R;
#pragma unroll
        for (int j = 0; j < NP; ++j) xv[j] = __ldg(xp + (size_t)j * R);
#pragma unroll
        for (int j = 0; j < NP; ++j) mag = max(mag, mag_bits(xv[j]));
        constexpr int B = Part::tab.begin[s], N = Part::tab.begin[s + 1] - B;
        mpat_entries<Part, NEG, B>(std::make_integer_sequence<int, N>{}, Vc, d, xv, acc, B);
      }
    }
  };
  slot(std::integral_constant<int, 0>{});
  slot(std::integral_constant<int, 1>{});
  slot(std::integral_constant<int, 2>{});
  slot(std::integral_constant<int, 3>{});
  slot(std::integral_constant<int, 4>{});
  slot(std::integral_constant<int, 5>{});
  slot(std::integral_constant<int, 6>{});
  if (mag >= Nonfinite<T>::FROM) {
    const unsigned rows = mpat_poison<T, NP, DIM, FROM>(x, g, K, c0, c1, c2, R);
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if ((rows >> i) & 1u) poison(acc[i]);
  }
}

// y = A x (MODE 0), y = b - A x in double-double, rounded once (MODE 2)
template <int NP, int DIM, int RP, int MODE>
__global__ void __launch_bounds__(kMpatThreads)
k_mpat_spmm(const double* __restrict__ V, PatGrid g, int R, const double* __restrict__ x, double* __restrict__ y,
            const double* __restrict__ b) {
  const MLane m = mpat_lane<RP>(g.C, R);
  if (!m.act) return;
  using ACC = typename std::conditional<MODE == 2, DD, double>::type;
  ACC acc[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) acc[i] = ACC{};
  mpat_apply<double, NP, DIM, 0, false>(V, g, m.cell, R, x + m.col, acc);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const size_t o = ((size_t)m.cell * NP + i) * R + m.col;
    if constexpr (MODE == 0) y[o] = acc[i];
    else {
      double s, t;
      two_sum(__ldg(b + o), -acc[i].hi, s, t);
      y[o] = s + (t - acc[i].lo);
    }
  }
}

// One damped block-Jacobi sweep.  FP64 (T = double): t = r - A_off zo summed from r, as
// k_msweep64.  FP32: the coupling summed from zero, then r added, as k_msweep_simt; the first
// sweep reads the residual as TR and leaves the FP32 copy in r_lo, the last writes TZ.
template <typename T, typename TI, typename TR, typename TZ, int NP, int DIM, int RP, bool FIRST>
__global__ void __launch_bounds__(kMpatThreads)
k_mpat_sweep(const T* __restrict__ V, const TI* __restrict__ D, PatGrid g, int R, const TR* __restrict__ r,
             T* __restrict__ r_lo, const T* __restrict__ zo, TZ* __restrict__ zn, T om) {
  const MLane m = mpat_lane<RP>(g.C, R);
  if (!m.act) return;
  const size_t o0 = (size_t)m.cell * NP * R + m.col;
  T t[NP];
  if constexpr (FIRST) {
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = (T)__ldg(r + o0 + (size_t)i * R);
    if constexpr (!std::is_same<T, TR>::value) {
#pragma unroll
      for (int i = 0; i < NP; ++i) r_lo[o0 + (size_t)i * R] = t[i];
    }
  } else if constexpr (std::is_same<T, double>::value) {
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = __ldg(r + o0 + (size_t)i * R);
    mpat_apply<T, NP, DIM, 1, true>(V, g, m.cell, R, zo + m.col, t);
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = T(0);
    mpat_apply<T, NP, DIM, 1, true>(V, g, m.cell, R, zo + m.col, t);
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] += __ldg(r + o0 + (size_t)i * R);
  }
  const TI* Dc = D + (size_t)m.cell * NP * NP;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    T e = T(0);
    if constexpr (NP % 2 == 0) {
#pragma unroll
      for (int j = 0; j < NP; j += 2) {
        const auto d = PairLoad<TI>::get(Dc + i * NP + j);
        e = fma((T)d.x, t[j], e);
        e = fma((T)d.y, t[j + 1], e);
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) e = fma((T)Dc[i * NP + j], t[j], e);
    }
    const size_t o = o0 + (size_t)i * R;
    zn[o] = (TZ)(FIRST ? om * e : fma(T(1) - om, __ldg(zo + o), om * e));
  }
}

// The FP32 sweep for column counts that are a multiple of four (16 to 32): a lane owns four
// columns, so 32 columns are eight lanes and a warp takes four cells, and the entries and
// inverses of a block's cells are staged in shared memory, the inverses as FP32.  With a column a
// lane (above) the sweep is bound by L1: 200 load instructions a cell, 110 of them one address for
// the whole warp.  Here a row of the iterate is one 16-byte load a lane and an entry pair one
// conflict-free shared-memory read for four cells: about 100 L1 accesses a cell.
template <int NP, int DIM, int LPC> struct MSweep4 {
  static constexpr int CELLS = kMpatThreads / LPC;            // cells of a block
  static constexpr int VS = MPattern<NP, DIM>::STRIDE;        // floats of a cell's entries
  static constexpr int DR = (NP + 3) / 4 * 4;                 // floats of an inverse row
  static constexpr int BYTES = CELLS * (VS + NP * DR) * 4;
};

template <typename Part, int E>
static __device__ __forceinline__ void m4_entry(const float* Vc, const float4& x, float4 (&t)[Part::ROWS]) {
  constexpr int I = Part::tab.i[E];
  if constexpr (I >= 0) {
    const float v = Vc[E];
    t[I].x = fmaf(-v, x.x, t[I].x);
    t[I].y = fmaf(-v, x.y, t[I].y);
    t[I].z = fmaf(-v, x.z, t[I].z);
    t[I].w = fmaf(-v, x.w, t[I].w);
  }
}
template <typename Part, int B, int NP, int... E>
static __device__ __forceinline__ void m4_entries(std::integer_sequence<int, E...>, const float* Vc,
                                                  const float4 (&x)[NP], float4 (&t)[Part::ROWS]) {
  (m4_entry<Part, B + E>(Vc, x[Part::tab.j[B + E]], t), ...);
}
static __device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
static __device__ __forceinline__ float4 ld4(const double* p) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  return make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
}
static __device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
static __device__ __forceinline__ void st4(double* p, const float4& v) {
  *reinterpret_cast<double2*>(p) = make_double2(v.x, v.y);
  *reinterpret_cast<double2*>(p + 2) = make_double2(v.z, v.w);
}

template <typename TI, typename TR, typename TZ, int NP, int DIM, int LPC, bool FIRST>
__global__ void __launch_bounds__(kMpatThreads)
k_mpat_sweep4(const float* __restrict__ V, const TI* __restrict__ D, PatGrid g, int R, const TR* __restrict__ r,
              float* __restrict__ r_lo, const float* __restrict__ zo, TZ* __restrict__ zn, float om) {
  using MP = MPattern<NP, DIM>;
  using Part = typename MP::Part;
  using Sh = MSweep4<NP, DIM, LPC>;
  extern __shared__ __align__(16) float smem_m4[];
  float* Vs = smem_m4;
  float* Ds = smem_m4 + Sh::CELLS * Sh::VS;
  const int K0 = blockIdx.x * Sh::CELLS, nk = min(Sh::CELLS, g.C - K0);
  if (!FIRST) {
    const float4* src = reinterpret_cast<const float4*>(V + (size_t)K0 * Sh::VS);
    for (int q = threadIdx.x; q < nk * (Sh::VS / 4); q += kMpatThreads) reinterpret_cast<float4*>(Vs)[q] = __ldg(src + q);
  }
  for (int q = threadIdx.x; q < nk * NP * NP; q += kMpatThreads) {
    const int c = q / (NP * NP), e = q - c * NP * NP;
    Ds[(c * NP + e / NP) * Sh::DR + e % NP] = (float)D[(size_t)K0 * NP * NP + q];
  }
  __syncthreads();
  const int c = threadIdx.x / LPC, K = K0 + c, col = (threadIdx.x % LPC) * 4;
  if (c >= nk || col >= R) return;
  const size_t o0 = (size_t)K * NP * R + col;
  float4 t[NP];
  if constexpr (FIRST) {
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = ld4(r + o0 + (size_t)i * R);
    if constexpr (!std::is_same<float, TR>::value) {
#pragma unroll
      for (int i = 0; i < NP; ++i) st4(r_lo + o0 + (size_t)i * R, t[i]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) t[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* Vc = Vs + c * Sh::VS;
    const int q0 = (unsigned)K / (unsigned)g.n0, c0 = K - q0 * g.n0;
    const int c2 = DIM == 3 ? (unsigned)q0 / (unsigned)g.n1 : 0, c1 = DIM == 3 ? q0 - c2 * g.n1 : q0;
    int mag = 0;
    auto slot = [&](auto sc) {
      constexpr int s = decltype(sc)::value;
      if constexpr (s < MP::TP::S) {
        const int J = pat_neighbour<DIM>(g, K, c0, c1, c2, s);
        if (J >= 0) {
          float4 x[NP];
#pragma unroll
          for (int j = 0; j < NP; ++j) x[j] = ld4(zo + (size_t)J * NP * R + col + (size_t)j * R);
#pragma unroll
          for (int j = 0; j < NP; ++j)
            mag = max(max(mag, max(mag_bits(x[j].x), mag_bits(x[j].y))), max(mag_bits(x[j].z), mag_bits(x[j].w)));
          constexpr int B = Part::tab.begin[s], N = Part::tab.begin[s + 1] - B;
          m4_entries<Part, B>(std::make_integer_sequence<int, N>{}, Vc, x, t);
        }
      }
    };
    slot(std::integral_constant<int, 1>{});
    slot(std::integral_constant<int, 2>{});
    slot(std::integral_constant<int, 3>{});
    slot(std::integral_constant<int, 4>{});
    slot(std::integral_constant<int, 5>{});
    slot(std::integral_constant<int, 6>{});
    if (mag >= Nonfinite<float>::FROM) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const unsigned rows = mpat_poison<float, NP, DIM, 1>(zo + col + k, g, K, c0, c1, c2, R);
#pragma unroll
        for (int i = 0; i < NP; ++i)
          if ((rows >> i) & 1u) poison(k == 0 ? t[i].x : k == 1 ? t[i].y : k == 2 ? t[i].z : t[i].w);
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const float4 b = ld4(r + o0 + (size_t)i * R);
      t[i].x += b.x;
      t[i].y += b.y;
      t[i].z += b.z;
      t[i].w += b.w;
    }
  }
  const float* Dc = Ds + c * NP * Sh::DR;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const float d = Dc[i * Sh::DR + j];
      e.x = fmaf(d, t[j].x, e.x);
      e.y = fmaf(d, t[j].y, e.y);
      e.z = fmaf(d, t[j].z, e.z);
      e.w = fmaf(d, t[j].w, e.w);
    }
    const size_t o = o0 + (size_t)i * R;
    if constexpr (FIRST) {
      e.x *= om;
      e.y *= om;
      e.z *= om;
      e.w *= om;
    } else {
      const float4 z = ld4(zo + o);
      e.x = fmaf(1.f - om, z.x, om * e.x);
      e.y = fmaf(1.f - om, z.y, om * e.y);
      e.z = fmaf(1.f - om, z.z, om * e.z);
      e.w = fmaf(1.f - om, z.w, om * e.w);
    }
    st4(zn + o, e);
  }
}

namespace {


template <int NP, int DIM, typename TAB, typename T>
__global__ void k_mpat_pack(const double* __restrict__ nat, const int* __restrict__ nbr, int C,
                            const __grid_constant__ TAB tab, T* __restrict__ V) {
  constexpr int S = 2 * DIM + 1, ST = MPattern<NP, DIM>::STRIDE;
  const size_t total = (size_t)C * ST;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(q % ST), K = (int)(q / ST);
    double v = 0.0;
    if (e < tab.n && tab.i[e] >= 0) {
      int s = 0;
      while (e >= tab.begin[s + 1]) ++s;
      if (s == 0 || nbr[(size_t)K * (S - 1) + s - 1] >= 0)
        v = nat[(((size_t)s * C + K) * NP + tab.i[e]) * NP + tab.j[e]];
    }
    V[q] = (T)v;
  }
}

template <typename F>
bool mpat_switch(int np, int dim, F&& f) {
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
// lanes per cell: the smallest of 8, 16, 32 that holds R columns (TWO: of 8 and 32; the FP32
// kernels are bound by memory, idle lanes cost them little)
template <bool TWO, typename F>
void rp_switch(int R, F&& f) {
  if (R <= 8) f(std::integral_constant<int, 8>{});
  else if (!TWO && R <= 16) f(std::integral_constant<int, 16>{});
  else f(std::integral_constant<int, 32>{});
}

int mpat_grid(int C, int RP) {
  const int cells = (32 / RP) * (kMpatThreads / 32);
  return (C + cells - 1) / cells;
}
PatGrid mpat_dims(const int* n, int dim) {
  PatGrid g;
  g.n0 = n[0];
  g.n1 = n[1];
  g.n2 = dim == 3 ? n[2] : 1;
  g.C = g.n0 * g.n1 * g.n2;
  g.groups = (g.C + 31) / 32;
  return g;
}

}  // namespace


template <typename T>
void launch_mpattern_pack(int np, int dim, const double* nat, const int* nbr, int C, T* V, cudaStream_t s) {
  mpat_switch(np, dim, [&](auto NPc, auto DIMc) {
    constexpr int NP = decltype(NPc)::value, DIM = decltype(DIMc)::value;
    using Part = typename MPattern<NP, DIM>::Part;
    static constexpr auto tab = Part::make();
    k_mpat_pack<NP, DIM, typename Part::Tab, T><<<152 * 8, 256, 0, s>>>(nat, nbr, C, tab, V);
  });
}

template <typename T, typename TI, typename TR, typename TZ>
void launch_mpattern_sweep(int np, int dim, const int* n, int R, const T* V, const TI* D, const TR* r, T* r_lo,
                           const T* zo, TZ* zn, double omega, int first, cudaStream_t s) {
  const PatGrid g = mpat_dims(n, dim);
  if constexpr (std::is_same<T, float>::value) {
    // four columns a lane: rows on 16-byte boundaries and at least four lanes a cell (fewer columns
    // stage more cells than they keep busy); np = 20 would need 80 sums a lane
    if (R % 4 == 0 && R >= 16 && np <= 10) {
      mpat_switch(np, dim, [&](auto NPc, auto DIMc) {
        constexpr int NP = decltype(NPc)::value, DIM = decltype(DIMc)::value;
        auto go = [&](auto LPCc) {
          constexpr int LPC = decltype(LPCc)::value;
          using Sh = MSweep4<NP, DIM, LPC>;
          const int grid = (g.C + Sh::CELLS - 1) / Sh::CELLS;
          if constexpr (std::is_same<TZ, T>::value && !std::is_same<TR, T>::value)
            if (first) k_mpat_sweep4<TI, TR, TZ, NP, DIM, LPC, true><<<grid, kMpatThreads, Sh::BYTES, s>>>(V, D, g, R, r, r_lo, zo, zn, (T)omega);
          if constexpr (std::is_same<TR, T>::value)
            if (!first) k_mpat_sweep4<TI, TR, TZ, NP, DIM, LPC, false><<<grid, kMpatThreads, Sh::BYTES, s>>>(V, D, g, R, r, r_lo, zo, zn, (T)omega);
        };
        if constexpr (NP <= 10) {
          if (R > 16) go(std::integral_constant<int, 8>{});
          else go(std::integral_constant<int, 4>{});
        }
      });
      return;
    }
  }
  mpat_switch(np, dim, [&](auto NPc, auto DIMc) {
    rp_switch<std::is_same<T, float>::value>(R, [&](auto RPc) {
      constexpr int NP = decltype(NPc)::value, DIM = decltype(DIMc)::value, RP = decltype(RPc)::value;
      const int grid = mpat_grid(g.C, RP);
      // FP32: the first sweep reads FP64, the others FP32 residuals
      if constexpr (std::is_same<TZ, T>::value && (std::is_same<T, double>::value || !std::is_same<TR, T>::value))
        if (first) k_mpat_sweep<T, TI, TR, TZ, NP, DIM, RP, true><<<grid, kMpatThreads, 0, s>>>(V, D, g, R, r, r_lo, zo, zn, (T)omega);
      if constexpr (std::is_same<TR, T>::value)
        if (!first) k_mpat_sweep<T, TI, TR, TZ, NP, DIM, RP, false><<<grid, kMpatThreads, 0, s>>>(V, D, g, R, r, r_lo, zo, zn, (T)omega);
    });
  });
}

}  // namespace kcmg
