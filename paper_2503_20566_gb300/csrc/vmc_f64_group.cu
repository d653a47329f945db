// Kernels with several chains per CTA for scalar type double.
#include "vmc_group.cuh"

GCF_INSTANTIATE_GROUP(double, false)
