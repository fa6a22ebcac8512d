// FP32 instantiations of the resident single-mode kernel.
#include "bq_resident.cuh"

namespace bq {

cudaError_t launch_resident_f32(const ResArgs& a, int mode, int ns, int herm, int n_bins, int smem_bytes, cudaStream_t s) {
  return launch_resident_t<float>(a, mode, ns, herm, n_bins, smem_bytes, s);
}

}  // namespace bq
