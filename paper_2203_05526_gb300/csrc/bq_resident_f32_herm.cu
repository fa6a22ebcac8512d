// FP32 instantiations of the resident single-mode kernel, Hermitian layout.
#include "bq_resident.cuh"

namespace bq {

cudaError_t launch_resident_f32_herm(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s) {
  return launch_resident_t<float, true>(a, variant, n_bins, smem_bytes, s);
}

}  // namespace bq
