// Kernels with several chains per CTA for scalar type cdouble.
#include "vmc_group.cuh"

GCF_INSTANTIATE_GROUP(cdouble, false)
