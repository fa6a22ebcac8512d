// FP64 instantiations of the grid-resident kernels.
#include "bq_grid.cuh"

namespace bq {

const void* grid_func_f64(int np, int ns, bool adj, int form) { return grid_func_t<double>(np, ns, adj, form); }

cudaError_t launch_grid_f64(const GridArgs& a, int np, int ns, bool adj, int ctas, int form, int smem_bytes, cudaStream_t s) {
  return launch_grid_any(grid_func_f64(np, ns, adj, form), a, ctas, form, smem_bytes, s);
}

cudaError_t grid_max_ctas(int dtype, int np, int ns, bool adj, int form, int smem_bytes, int* out) {
  *out = 0;
  const void* f = dtype == 0 ? grid_func_f64(np, ns, adj, form) : grid_func_f32(np, ns, adj, form);
  if (!f || smem_bytes > BQ_GRID_SMEM_MAX) return cudaSuccess;
  int dev = 0, sms = 0, coop = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, BQ_GRID_SMEM_MAX);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, grid_threads(form), smem_bytes);
  if (e != cudaSuccess) return e;
  *out = coop ? per_sm * sms : 0;
  return cudaSuccess;
}

}  // namespace bq
