// FP32 batched pattern sweeps (mrhs_pattern.cuh).
#include "mrhs_pattern.cuh"

namespace kcmg {

template void launch_mpattern_pack<float>(int, int, const double*, const int*, int, float*, cudaStream_t);
#define KCMG_MSWEEP(TI, TR, TZ)                                                                                   \
  template void launch_mpattern_sweep<float, TI, TR, TZ>(int, int, const int*, int, const float*, const TI*,      \
                                                         const TR*, float*, const float*, TZ*, double, int,       \
                                                         cudaStream_t);
KCMG_MSWEEP(float, double, float)
KCMG_MSWEEP(float, float, float)
KCMG_MSWEEP(float, float, double)
KCMG_MSWEEP(__nv_bfloat16, double, float)
KCMG_MSWEEP(__nv_bfloat16, float, float)
KCMG_MSWEEP(__nv_bfloat16, float, double)

}  // namespace kcmg
