// Launchers of the kernels with several chains per CTA (one translation unit per scalar type).
#pragma once

#include "vmc_cta.cuh"

namespace gcf {

// 256 threads: two chain groups per CTA; 512: four (one CTA per SM)
template <class T, bool TC>
cudaError_t launch_vmc_grouped(const KParams<T>& k, int grid, int block, size_t smem, cudaStream_t st) {
  auto* fn = block == 512 ? vmc_kernel_grouped4<T, TC> : vmc_kernel_grouped<T, TC>;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  fn<<<grid, block, smem, st>>>(k);
  return cudaGetLastError();
}
template <class T, bool TC>
int occupancy_vmc_grouped(int block, size_t smem) {
  return blocks_per_sm(block == 512 ? vmc_kernel_grouped4<T, TC> : vmc_kernel_grouped<T, TC>, block, smem);
}
template <class T, bool TC>
cudaError_t launch_vmc_multi4(const KParams<T>* ks, int n_ctx, const long long* start, long long total, T* arena,
                              long long ws_stride, int grid, long long group_bytes, unsigned long long* queue,
                              size_t smem, cudaStream_t st) {
  cudaError_t e = allow_smem(vmc_kernel_multi4<T, TC>, smem);
  if (e != cudaSuccess) return e;
  vmc_kernel_multi4<T, TC><<<grid, 512, smem, st>>>(ks, n_ctx, start, total, arena, ws_stride, group_bytes, queue);
  return cudaGetLastError();
}
template <class T, bool TC>
int occupancy_vmc_multi4(size_t smem) { return blocks_per_sm(vmc_kernel_multi4<T, TC>, 512, smem); }

}  // namespace gcf

#define GCF_INSTANTIATE_GROUP(T, TC) \
  namespace gcf { \
  template cudaError_t launch_vmc_grouped<T, TC>(const KParams<T>&, int, int, size_t, cudaStream_t); \
  template int occupancy_vmc_grouped<T, TC>(int, size_t); \
  template cudaError_t launch_vmc_multi4<T, TC>(const KParams<T>*, int, const long long*, long long, T*, long long, int, \
                                            long long, unsigned long long*, size_t, cudaStream_t); \
  template int occupancy_vmc_multi4<T, TC>(size_t); \
  }
