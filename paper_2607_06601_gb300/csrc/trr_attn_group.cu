// trr_attn_group.cu - the kernels of trr_decode_attn with a KV head and its query group
// per warp (g >= 2 whose (head, group) columns fit one 8-wide mma tile; trr_row.cuh), one
// instance per head size and groups per head, and the kernel that merges their split partials.
#include "trr_row.cuh"

namespace trr {

template <int D, int NG>
static cudaError_t launch(dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  return launch_pdl(row_kernel<D, NG, false, false, true>, grid, dim3(32 * kRowWarps), smem, s, k);
}

cudaError_t launch_attn_group(const Layout& l, dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  const int ng = l.d / l.G;
  if (l.d == 64) return ng == 1 ? launch<64, 1>(grid, smem, s, k) : launch<64, 2>(grid, smem, s, k);
  if (ng == 1) return launch<128, 1>(grid, smem, s, k);
  return ng == 2 ? launch<128, 2>(grid, smem, s, k) : launch<128, 4>(grid, smem, s, k);
}

cudaError_t launch_attn_combine(int d, int ctas, cudaStream_t s, const CombineArgs& ca) {
  return d == 64 ? launch_pdl(attn_combine_kernel<64>, dim3(ctas), dim3(32 * kCombineWarps), 0, s, ca)
                 : launch_pdl(attn_combine_kernel<128>, dim3(ctas), dim3(32 * kCombineWarps), 0, s, ca);
}

cudaError_t configure_attn_group() {
  const void* ks[] = {reinterpret_cast<const void*>(row_kernel<64, 1, false, false, true>),
                      reinterpret_cast<const void*>(row_kernel<64, 2, false, false, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 1, false, false, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 2, false, false, true>),
                      reinterpret_cast<const void*>(row_kernel<128, 4, false, false, true>)};
  for (const void* f : ks) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace trr
