// FP32 pattern kernels (pattern_ops.cuh): sweeps of the mixed forms, the inner solve of the
// iterative refinement.
#include "pattern_ops.cuh"

namespace kcmg {

template void launch_pattern_pack<float>(int, int, const double*, const int*, int, float*, cudaStream_t);
template void launch_pattern_pack_inverse<float>(int, int, const double*, int, float*, cudaStream_t);
template void launch_pattern_pack_inverse<__nv_bfloat16>(int, int, const double*, int, __nv_bfloat16*, cudaStream_t);
template void launch_pattern_spmv<float>(int, int, const int*, const float*, const float*, float*, const float*,
                                         double*, const EpiArgs&, int, cudaStream_t);
#define KCMG_SWEEP_INST(TI, TR, TZ)                                                                                 \
  template void launch_pattern_sweep<float, TI, TR, TZ>(int, int, const int*, const float*, const TI*, const TR*,   \
                                                        float*, const float*, TZ*, double, int, cudaStream_t);
KCMG_SWEEP_INST(float, float, float)
KCMG_SWEEP_INST(float, double, float)
KCMG_SWEEP_INST(float, float, double)
KCMG_SWEEP_INST(__nv_bfloat16, float, float)
KCMG_SWEEP_INST(__nv_bfloat16, double, float)
KCMG_SWEEP_INST(__nv_bfloat16, float, double)

}  // namespace kcmg
