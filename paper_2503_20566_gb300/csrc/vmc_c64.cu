// One-chain-per-CTA kernels for scalar type cfloat.
#include "vmc_cta.cuh"

GCF_INSTANTIATE_CTA(cfloat, false)
