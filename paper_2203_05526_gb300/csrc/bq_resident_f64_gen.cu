// FP64 instantiations of the resident single-mode kernel, general layout, and the Hermitian check of both types.
#include "bq_resident.cuh"

namespace bq {

cudaError_t launch_resident_f64_gen(const ResArgs& a, int variant, int n_bins, int smem_bytes, cudaStream_t s) {
  return launch_resident_t<double, false>(a, variant, n_bins, smem_bytes, s);
}

// One warp per system: exact comparison of every element with its mirror (a NaN compares
// unequal: such a system takes the general layout).
template <typename T>
__global__ void k_res_check(const ResGroup* __restrict__ groups, int n, const void* y, const void* comp, int comp_zero,
                            unsigned char* flags) {
  using C = typename C2T<T>::type;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n) return;
  const ResGroup g = groups[w];
  bool ok = true;
  for (int arr = 0; arr < (comp_zero ? 1 : 2); ++arr) {
    const C* v = reinterpret_cast<const C*>(arr == 0 ? y : comp) + g.blk_off;
    if (g.gy_off >= 0)
      for (int i = lane; i < g.M; i += 32) ok = ok && v[i].x == v[g.gy_off + i].x && v[i].y == -v[g.gy_off + i].y;
    const C* r = v + g.r_off;
    for (int i = lane; i < g.M * g.M; i += 32) {
      const int k = i / g.M, l = i - k * g.M;
      const C a = r[i], b = r[l * g.M + k];
      ok = ok && a.x == b.x && a.y == -b.y;
    }
  }
  ok = __all_sync(0xffffffffu, ok);
  if (lane == 0) flags[g.sys] = ok ? 1 : 0;
}

cudaError_t launch_res_check(const ResGroup* groups, int n, const void* y, const void* comp, int comp_zero, int dtype,
                             unsigned char* flags, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int threads = 128, blocks = (n * 32 + threads - 1) / threads;
  if (dtype == 0)
    k_res_check<double><<<blocks, threads, 0, s>>>(groups, n, y, comp, comp_zero, flags);
  else
    k_res_check<float><<<blocks, threads, 0, s>>>(groups, n, y, comp, comp_zero, flags);
  return cudaGetLastError();
}

}  // namespace bq
