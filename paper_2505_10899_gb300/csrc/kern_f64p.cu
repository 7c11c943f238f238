// FP64 step kernels without the short forms of lbm_math.cuh (reverse mode).
#define LBM_T double
#define LBM_PLAIN true
#include "kern_impl.cuh"
