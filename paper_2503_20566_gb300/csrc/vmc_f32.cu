// One-chain-per-CTA kernels for scalar type float.
#include "vmc_cta.cuh"

GCF_INSTANTIATE_CTA(float, false)

namespace gcf {
size_t sharedv_bytes() { return sizeof_sharedv_aligned(); }
}  // namespace gcf
