// trr_attn_group_step.cu - the kernels of trr_decode_step with a KV head and its query
// group per warp (trr_row.cuh), one instance per head size and groups per head; the kernel of
// trr_attn_group.cu merges their split partials.
#include "trr_row.cuh"

namespace trr {

template <int D, int NG>
static cudaError_t launch(dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  return launch_pdl(row_kernel<D, NG, false, true, true>, grid, dim3(32 * kRowWarps), smem, s, k);
}

cudaError_t launch_attn_group_step(const Layout& l, dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  const int ng = l.d / l.G;
  if (l.d == 64) return ng == 1 ? launch<64, 1>(grid, smem, s, k) : launch<64, 2>(grid, smem, s, k);
  if (ng == 1) return launch<128, 1>(grid, smem, s, k);
  return ng == 2 ? launch<128, 2>(grid, smem, s, k) : launch<128, 4>(grid, smem, s, k);
}

cudaError_t configure_attn_group_step() {
  const void* ks[] = {reinterpret_cast<const void*>(row_kernel<64, 1, false, true, true>),
                      reinterpret_cast<const void*>(row_kernel<64, 2, false, true, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 1, false, true, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 2, false, true, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 4, false, true, true>)};
  for (const void* f : ks) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace trr
