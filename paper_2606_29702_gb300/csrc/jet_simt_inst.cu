// Instantiates the SIMT kernels for one closure class; compiled once per class
// with -DJET_CLASS_ID=<id> so the classes build in parallel.
#include "jet_simt.cuh"

#ifndef JET_CLASS_ID
#error "JET_CLASS_ID must be defined"
#endif

namespace jet {

using ThisCls = ClassById<JET_CLASS_ID>::type;

// Called when a plan, a batch or the no-alloc path sizes its tile.  The kernel
// may take all the shared memory the device gives a block, and the query runs
// with the whole SM's as the preferred carve-out: one left by an earlier launch
// with a smaller tile would halve the residency it reports.
template <>
cudaError_t simt_max_active_id<JET_CLASS_ID>(bool fp64, int ru, int threads, size_t smem, int* blocks) {
  const auto kernel = fp64 ? simt_entry<ThisCls, double>(ru) : simt_entry<ThisCls, float>(ru);
  *blocks = 0;
  cudaFuncAttributes fa;
  int dev = 0, most = 0;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  most -= (int)fa.sharedSizeBytes;
  if (smem > (size_t)most || threads > fa.maxThreadsPerBlock) return cudaSuccess;  // no CTA fits
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kernel, threads, smem);
  return e;
}

template <>
cudaError_t simt_launch_id<JET_CLASS_ID>(bool fp64, const SimtArgs& a, int grid, size_t smem, cudaStream_t s) {
  const auto kernel = fp64 ? simt_entry<ThisCls, double>(a.ru) : simt_entry<ThisCls, float>(a.ru);
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, a.carveout);
  if (e != cudaSuccess) return e;
  return launch_dependent(kernel, grid, a.threads, smem, s, a);
}

template <>
cudaError_t debug_activation_id<JET_CLASS_ID>(int kind, long long n, const double* z, const double* v, double* out,
                                              cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int grid = (int)((n + 255) / 256);
  if (grid > 4096) grid = 4096;
  debug_activation_kernel<ThisCls><<<grid, 256, 0, s>>>(kind, n, z, v, out);
  return cudaGetLastError();
}

}  // namespace jet
