// FP64 batched pattern kernels (mrhs_pattern.cuh).
#include "mrhs_pattern.cuh"

namespace kcmg {

size_t mpattern_values(int np, int dim, int C) {
  size_t per = 0;
  mpat_switch(np, dim, [&](auto NPc, auto DIMc) { per = MPattern<decltype(NPc)::value, decltype(DIMc)::value>::STRIDE; });
  return (size_t)C * per;
}

void launch_mpattern_spmm(int np, int dim, const int* n, int R, const double* V, const double* x, double* y,
                          const double* b, int mode, cudaStream_t s) {
  const PatGrid g = mpat_dims(n, dim);
  mpat_switch(np, dim, [&](auto NPc, auto DIMc) {
    rp_switch<false>(R, [&](auto RPc) {
      constexpr int NP = decltype(NPc)::value, DIM = decltype(DIMc)::value, RP = decltype(RPc)::value;
      const int grid = mpat_grid(g.C, RP);
      if (mode == 0) k_mpat_spmm<NP, DIM, RP, 0><<<grid, kMpatThreads, 0, s>>>(V, g, R, x, y, b);
      else k_mpat_spmm<NP, DIM, RP, 2><<<grid, kMpatThreads, 0, s>>>(V, g, R, x, y, b);
    });
  });
}

template void launch_mpattern_pack<double>(int, int, const double*, const int*, int, double*, cudaStream_t);
template void launch_mpattern_sweep<double, double, double, double>(int, int, const int*, int, const double*,
                                                                    const double*, const double*, double*,
                                                                    const double*, double*, double, int, cudaStream_t);

}  // namespace kcmg
