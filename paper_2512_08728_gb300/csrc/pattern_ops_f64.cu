// FP64 pattern kernels and the setup of the pattern storage (pattern_ops.cuh).
#include "pattern_ops.cuh"

namespace kcmg {

int pattern_blocks(int np, int dim, int C) {
  int blocks = 0;
  KCMG_PAT(np, dim, {
    constexpr int GPB = kPatThreads / 32 / TensorPattern<NP, DIM>::PARTS;
    blocks = ((C + 31) / 32 + GPB - 1) / GPB;
  });
  return blocks;
}

size_t pattern_values(int np, int dim, int C) {
  size_t per = 0;
  KCMG_PAT(np, dim, { per = (size_t)TensorPattern<NP, DIM>::PARTS * TensorPattern<NP, DIM>::PAIRS * 64; });
  return (size_t)((C + 31) / 32) * per;
}

size_t pattern_coupling_values(int np, int dim, int C) {
  size_t per = 0;
  KCMG_PAT(np, dim, {
    constexpr auto m = TensorPattern<NP, DIM>::make_modes();
    for (int s = 1; s < TensorPattern<NP, DIM>::S; ++s)
      for (int e = 0; e < NP * NP; ++e) per += TensorPattern<NP, DIM>::nz(m, s, e / NP, e % NP);
  });
  return (size_t)C * per;
}

size_t pattern_inverse_values(int np, int dim, int C) {
  size_t per = 0;
  KCMG_PAT(np, dim, { per = (size_t)TensorPattern<NP, DIM>::PARTS * TensorPattern<NP, DIM>::INV_PAIRS * 64; });
  return (size_t)((C + 31) / 32) * per;
}

void launch_pattern_check(int np, int dim, const double* nat, const int* nbr, int C, int* outside, cudaStream_t s) {
  KCMG_PAT(np, dim, {
    constexpr auto zeros = TensorPattern<NP, DIM>::make_zeros();
    k_pat_check<NP, DIM><<<152 * 8, 256, 0, s>>>(nat, nbr, C, zeros, outside);
  });
}

void launch_pattern_residual_dd(int np, int dim, const int* n, const double* V, const double* x, double* r,
                                const double* b, double* partial, const EpiArgs& e, int conditional,
                                cudaStream_t s) {
  const PatGrid g = pat_grid(n, dim);
  KCMG_PAT(np, dim, {
    k_pat_residual_dd<NP, DIM><<<pattern_blocks(np, dim, g.C), kPatThreads, 0, s>>>(V, g, x, r, b, partial, e, conditional);
  });
}

void launch_pattern_residual_scratch(int np, int dim, const int* n, const double* V, const double* x, const double* b,
                                     double* r, double* scratch, int count_at, double* norm, cudaStream_t s) {
  const PatGrid g = pat_grid(n, dim);
  KCMG_PAT(np, dim, {
    const int grid = pattern_blocks(np, dim, g.C);
    if (((uintptr_t)x & 15) == 0)
      k_pat_residual_scratch<NP, DIM, true><<<grid, kPatThreads, 0, s>>>(V, g, x, b, r, scratch, count_at, norm);
    else   // a caller's vector that does not start on the vector loads' boundary
      k_pat_residual_scratch<NP, DIM, false><<<grid, kPatThreads, 0, s>>>(V, g, x, b, r, scratch, count_at, norm);
  });
}

cudaError_t pattern_residual_load(int np, int dim) {
  cudaError_t e = cudaErrorInvalidValue;
  cudaFuncAttributes fa;
  KCMG_PAT(np, dim, {
    e = cudaFuncGetAttributes(&fa, (const void*)k_pat_residual_scratch<NP, DIM, true>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, (const void*)k_pat_residual_scratch<NP, DIM, false>);
  });
  return e;
}

template void launch_pattern_pack<double>(int, int, const double*, const int*, int, double*, cudaStream_t);
template void launch_pattern_pack_inverse<double>(int, int, const double*, int, double*, cudaStream_t);
template void launch_pattern_spmv<double>(int, int, const int*, const double*, const double*, double*, const double*,
                                          double*, const EpiArgs&, int, cudaStream_t);
template void launch_pattern_sweep<double, double, double, double>(int, int, const int*, const double*, const double*,
                                                                   const double*, double*, const double*, double*,
                                                                   double, int, cudaStream_t);

}  // namespace kcmg
