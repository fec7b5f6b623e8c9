// Several columns' whole solves in one persistent kernel, FP32 sweeps with BF16 inverses under FP64 minimisation.
#define CC_TV double
#define CC_T float
#define CC_TI __nv_bfloat16
#define CC_GROUP
#include "coarse_cycle_inst.cuh"
