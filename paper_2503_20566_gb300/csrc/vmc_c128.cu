// One-chain-per-CTA kernels for scalar type cdouble.
#include "vmc_cta.cuh"

GCF_INSTANTIATE_CTA(cdouble, false)
