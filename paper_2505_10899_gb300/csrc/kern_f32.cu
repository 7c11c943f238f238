// FP32 instantiation of the device kernels.
#define LBM_T float
#define LBM_PLAIN false
#include "kern_impl.cuh"
