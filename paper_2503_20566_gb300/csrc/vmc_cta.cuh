// Launchers of the one-chain-per-CTA kernels (one translation unit per scalar type).
#pragma once

#include "launch.h"
#include "vmc_kernel.cuh"

namespace gcf {

// static + dynamic shared memory above 48 KB needs the opt-in attribute
template <class F>
cudaError_t allow_smem(F* fn, size_t smem) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
template <class F>
int blocks_per_sm(F* fn, int block, size_t smem) {
  if (allow_smem(fn, smem) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem) != cudaSuccess) return 0;
  return n;
}

template <class T, bool TC>
cudaError_t launch_vmc(const KParams<T>& k, int grid, int block, size_t smem, cudaStream_t st) {
  cudaError_t e = allow_smem(vmc_kernel<T, TC>, smem);
  if (e != cudaSuccess) return e;
  vmc_kernel<T, TC><<<grid, block, smem, st>>>(k);
  return cudaGetLastError();
}
template <class T, bool TC>
int occupancy_vmc(int block, size_t smem) {
  const int n = blocks_per_sm(vmc_kernel<T, TC>, block, smem);
  return n > 0 ? n : 1;
}
template <class T, bool TC>
cudaError_t launch_vmc_multi(const KParams<T>* ks, int n_ctx, const long long* start, long long total, T* arena,
                             long long ws_stride, int grid, unsigned long long* queue, size_t smem, cudaStream_t st) {
  cudaError_t e = allow_smem(vmc_kernel_multi<T, TC>, smem);
  if (e != cudaSuccess) return e;
  vmc_kernel_multi<T, TC><<<grid, 256, smem, st>>>(ks, n_ctx, start, total, arena, ws_stride, queue);
  return cudaGetLastError();
}
template <class T, bool TC>
int occupancy_vmc_multi(size_t smem) { return blocks_per_sm(vmc_kernel_multi<T, TC>, 256, smem); }

}  // namespace gcf

#define GCF_INSTANTIATE_CTA(T, TC) \
  namespace gcf { \
  template cudaError_t launch_vmc<T, TC>(const KParams<T>&, int, int, size_t, cudaStream_t); \
  template int occupancy_vmc<T, TC>(int, size_t); \
  template cudaError_t launch_vmc_multi<T, TC>(const KParams<T>*, int, const long long*, long long, T*, long long, int, \
                                           unsigned long long*, size_t, cudaStream_t); \
  template int occupancy_vmc_multi<T, TC>(size_t); \
  }
