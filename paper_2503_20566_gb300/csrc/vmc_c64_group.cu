// Kernels with several chains per CTA for scalar type cfloat.
#include "vmc_group.cuh"

GCF_INSTANTIATE_GROUP(cfloat, false)
