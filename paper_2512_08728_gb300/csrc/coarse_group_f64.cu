// Several columns' whole solves in one persistent kernel, FP64 form.
#define CC_TV double
#define CC_T double
#define CC_TI double
#define CC_GROUP
#include "coarse_cycle_inst.cuh"
