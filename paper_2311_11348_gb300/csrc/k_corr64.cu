// FP64 instantiation of the correction kernels.
#define CORR_T double
#define CORR_NS corr64
#define CORR_LANES 1  // small order-4 groups: k_usolve_lanes
#include "k_corr_impl.cuh"
