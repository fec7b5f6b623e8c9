// Device pieces of the pattern kernels: lane mapping, cell loads and the off-diagonal /
// whole-operator product over the pattern's entries.
#pragma once
#include "epilogue.cuh"
#include "tensor_pattern.cuh"

#include <type_traits>
#include <utility>

namespace kcmg {

constexpr int kPatThreads = 128;

struct PatGrid { int n0, n1, n2, C, groups; };

struct PatLane {
  int lane, part, slot, group, cell;   // slot: the group's place in the block
};

template <int PARTS>
static __device__ __forceinline__ PatLane pat_lane(const PatGrid& g) {
  PatLane L;
  const int warp = threadIdx.x >> 5;
  L.lane = threadIdx.x & 31;
  L.slot = warp / PARTS;
  L.part = warp % PARTS;
  L.group = blockIdx.x * (kPatThreads / 32 / PARTS) + L.slot;
  L.cell = L.group * 32 + L.lane;
  return L;
}

// f with the warp's part as a compile-time constant
template <int PARTS, typename F>
static __device__ __forceinline__ void pat_dispatch(int part, F&& f) {
  if constexpr (PARTS == 1) {
    f(std::integral_constant<int, 0>{});
  } else if constexpr (PARTS == 2) {
    if (part == 0) f(std::integral_constant<int, 0>{});
    else f(std::integral_constant<int, 1>{});
  } else {
    static_assert(PARTS == 4, "parts");
    if (part == 0) f(std::integral_constant<int, 0>{});
    else if (part == 1) f(std::integral_constant<int, 1>{});
    else if (part == 2) f(std::integral_constant<int, 2>{});
    else f(std::integral_constant<int, 3>{});
  }
}

template <typename T> struct PairLoad;
template <> struct PairLoad<double> {
  using type = double2;
  static __device__ __forceinline__ double2 get(const double* p) { return __ldg(reinterpret_cast<const double2*>(p)); }
};
template <> struct PairLoad<float> {
  using type = float2;
  static __device__ __forceinline__ float2 get(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
};
template <> struct PairLoad<__nv_bfloat16> {
  using type = float2;
  static __device__ __forceinline__ float2 get(const __nv_bfloat16* p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
  }
};

// the NP values of cell K: two at a time where a cell starts on that boundary (NP even; VEC: x
// itself does)
template <typename T, int NP, bool VEC = true>
static __device__ __forceinline__ void load_cell(const T* __restrict__ x, int K, T (&v)[NP]) {
  const T* p = x + (size_t)K * NP;
  if constexpr (VEC && NP % 2 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 2) {
      const auto a = PairLoad<T>::get(p + j);
      v[j] = a.x;
      v[j + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) v[j] = __ldg(p + j);
  }
}

// magnitude bits of the exponent word; >= Nonfinite<T>::FROM for an infinity or NaN
static __device__ __forceinline__ int mag_bits(double v) { return __double2hiint(v) & 0x7fffffff; }
static __device__ __forceinline__ int mag_bits(float v) { return __float_as_int(v) & 0x7fffffff; }
template <typename T> struct Nonfinite { static constexpr int FROM = sizeof(T) == 8 ? 0x7ff00000 : 0x7f800000; };

// error-free sum (Knuth) and a double-double accumulator
static __device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
struct DD { double hi, lo; };
static __device__ __forceinline__ void madd(double a, double x, double& acc) { acc = fma(a, x, acc); }
static __device__ __forceinline__ void madd(float a, float x, float& acc) { acc = fma(a, x, acc); }
static __device__ __forceinline__ void madd(double a, double x, DD& acc) {
  const double p = a * x, pe = fma(a, x, -p);
  double s, e;
  two_sum(acc.hi, p, s, e);
  acc.hi = s;
  acc.lo += e + pe;
}
static __device__ __forceinline__ void poison(double& a) { a = __longlong_as_double(0x7ff8000000000000ll); }
static __device__ __forceinline__ void poison(float& a) { a = __int_as_float(0x7fc00000); }
static __device__ __forceinline__ void poison(DD& a) { poison(a.hi); }

// neighbour of the cell at (c0, c1, c2) through slot s (the cell itself for slot 0), -1 outside
template <int DIM>
static __device__ __forceinline__ int pat_neighbour(const PatGrid& g, int K, int c0, int c1, int c2, int s) {
  switch (s) {
    case 0: return K;
    case 1: return c0 > 0 ? K - 1 : -1;
    case 2: return c0 < g.n0 - 1 ? K + 1 : -1;
    case 3: return c1 > 0 ? K - g.n0 : -1;
    case 4: return c1 < g.n1 - 1 ? K + g.n0 : -1;
    case 5: return c2 > 0 ? K - g.n0 * g.n1 : -1;
    default: return c2 < g.n2 - 1 ? K + g.n0 * g.n1 : -1;
  }
}

// rows of cell K whose zero entries meet an infinity or NaN in x (dense products would be NaN)
template <typename T, int NP, int DIM, int FROM>
static __device__ __noinline__ unsigned poison_rows(const T* x, PatGrid g, int K, int c0, int c1, int c2) {
  const auto m = TensorPattern<NP, DIM>::make_modes();
  unsigned rows = 0;
  for (int s = FROM; s < 2 * DIM + 1; ++s) {
    const int J = pat_neighbour<DIM>(g, K, c0, c1, c2, s);
    if (J < 0) continue;
    unsigned bad = 0;
    for (int j = 0; j < NP; ++j)
      if (mag_bits(x[(size_t)J * NP + j]) >= Nonfinite<T>::FROM) bad |= 1u << j;
    if (!bad) continue;
    for (int i = 0; i < NP; ++i)
      for (int j = 0; j < NP; ++j)
        if ((bad >> j & 1u) && !TensorPattern<NP, DIM>::nz(m, s, i, j)) rows |= 1u << i;
  }
  return rows;
}

// The products of one slot: entry E of the part multiplies column tab.j[E] of the neighbour into
// row tab.i[E]; entries come two to a stored pair.
template <typename T, typename Part, int PARTS, int Q, int E, int FIRST, typename ACC, int NP, int ROWS>
static __device__ __forceinline__ void pat_entry(const T* __restrict__ Vp, typename PairLoad<T>::type& d,
                                                 const T (&xv)[NP], ACC (&acc)[ROWS]) {
  constexpr int I = Part::tab.i[E], J = Part::tab.j[E];
  if constexpr ((E & 1) == 0 || E == FIRST) d = PairLoad<T>::get(Vp + (E >> 1) * 64);
  if constexpr (I >= 0) madd((E & 1) ? d.y : d.x, xv[J], acc[(I - Q) / PARTS]);
}
template <typename T, typename Part, int PARTS, int Q, int BEGIN, int FIRST, typename ACC, int NP, int ROWS, int... E>
static __device__ __forceinline__ void pat_entries(std::integer_sequence<int, E...>, const T* __restrict__ Vp,
                                                   typename PairLoad<T>::type& d, const T (&xv)[NP],
                                                   ACC (&acc)[ROWS]) {
  (pat_entry<T, Part, PARTS, Q, BEGIN + E, FIRST>(Vp, d, xv, acc), ...);
}

// acc[k] += (A x) of row Q + k PARTS of the lane's cell, over slots FROM..2 DIM.  V: the stored
// entries; lanes past the last cell apply zeros to the last cell's values.
template <typename T, int NP, int DIM, int PARTS, int Q, int FROM, bool VEC = true, typename ACC, int ROWS>
static __device__ __forceinline__ void pat_apply(const T* __restrict__ V, const PatGrid& g, const PatLane& L,
                                                 const T* __restrict__ x, ACC (&acc)[ROWS]) {
  using TP = TensorPattern<NP, DIM>;
  using Part = typename TP::template Part<PARTS, Q>;
  const T* Vp = V + ((size_t)L.group * PARTS + Q) * (TP::PAIRS * 64) + 2 * L.lane;
  const int K = min(L.cell, g.C - 1);
  const int q0 = (unsigned)K / (unsigned)g.n0, c0 = K - q0 * g.n0;
  const int c2 = DIM == 3 ? (unsigned)q0 / (unsigned)g.n1 : 0, c1 = DIM == 3 ? q0 - c2 * g.n1 : q0;
  typename PairLoad<T>::type d{};
  int mag = 0;
  auto slot = [&](auto sc) {
    constexpr int s = decltype(sc)::value;
    if constexpr (s >= FROM && s < TP::S) {
      const int J = pat_neighbour<DIM>(g, K, c0, c1, c2, s);
      T xv[NP];
      if (J >= 0) {
        load_cell<T, NP, VEC>(x, J, xv);
      } else {
#pragma unroll
        for (int j = 0; j < NP; ++j) xv[j] = T(0);
      }
#pragma unroll
      for (int j = 0; j < NP; ++j) mag = max(mag, mag_bits(xv[j]));
      constexpr int B = Part::tab.begin[s], N = Part::tab.begin[s + 1] - B;
      pat_entries<T, Part, PARTS, Q, B, Part::tab.begin[FROM]>(std::make_integer_sequence<int, N>{}, Vp, d, xv, acc);
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
    const unsigned rows = poison_rows<T, NP, DIM, FROM>(x, g, K, c0, c1, c2);
#pragma unroll
    for (int k = 0; k < ROWS; ++k)
      if ((rows >> (Q + k * PARTS)) & 1u) poison(acc[k]);
  }
}

}  // namespace kcmg
