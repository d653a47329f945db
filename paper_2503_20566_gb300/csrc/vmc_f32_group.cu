// Kernels with several chains per CTA for scalar type float.
#include "vmc_group.cuh"

GCF_INSTANTIATE_GROUP(float, false)
