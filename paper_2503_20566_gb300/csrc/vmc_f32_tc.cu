// One-chain-per-CTA kernels for scalar type float whose environment GEMMs may run on tcgen05 (BF16 form).
#include "vmc_cta.cuh"

GCF_INSTANTIATE_CTA(float, true)
