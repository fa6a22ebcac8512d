// FP32 instantiations of the resident single-mode kernel, general layout.
#include "bq_resident.cuh"

namespace bq {

cudaError_t launch_resident_f32_gen(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s) {
  return launch_resident_t<float, false>(a, variant, n_bins, smem_bytes, s);
}

}  // namespace bq
