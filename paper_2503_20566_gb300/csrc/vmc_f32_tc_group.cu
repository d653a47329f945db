// Kernels with several chains per CTA for scalar type float whose environment GEMMs may run on tcgen05 (BF16 form).
#include "vmc_group.cuh"

GCF_INSTANTIATE_GROUP(float, true)
