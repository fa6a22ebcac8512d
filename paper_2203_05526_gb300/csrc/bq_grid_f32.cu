// FP32 instantiations of the grid-resident kernels.
#include "bq_grid.cuh"

namespace bq {

const void* grid_func_f32(int np, int ns, bool adj, int form) { return grid_func_t<float>(np, ns, adj, form); }

cudaError_t launch_grid_f32(const GridArgs& a, int np, int ns, bool adj, int ctas, int form, int smem_bytes, cudaStream_t s) {
  return launch_grid_any(grid_func_f32(np, ns, adj, form), a, ctas, form, smem_bytes, s);
}

}  // namespace bq
