// One-chain-per-CTA kernels for scalar type double.
#include "vmc_cta.cuh"

GCF_INSTANTIATE_CTA(double, false)
