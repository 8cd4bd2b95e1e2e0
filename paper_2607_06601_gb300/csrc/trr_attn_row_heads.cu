// trr_attn_row_heads.cu - the kernels of caches with per-head modes (presence masks
// read with every page): one instance per head size and groups
// per head.
#include "trr_row.cuh"

namespace trr {

template <int D, int NG>
static cudaError_t launch(dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  return launch_pdl(row_kernel<D, NG, true, false, false>, grid, dim3(32 * kRowWarps), smem, s, k);
}

cudaError_t launch_attn_row_heads(const Layout& l, dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  const int ng = l.d / l.G;
  if (l.d == 64) return ng == 1 ? launch<64, 1>(grid, smem, s, k) : launch<64, 2>(grid, smem, s, k);
  if (ng == 1) return launch<128, 1>(grid, smem, s, k);
  return ng == 2 ? launch<128, 2>(grid, smem, s, k) : launch<128, 4>(grid, smem, s, k);
}

cudaError_t configure_attn_row_heads() {
  const void* ks[] = {reinterpret_cast<const void*>(row_kernel<64, 1, true, false, false>),
                      reinterpret_cast<const void*>(row_kernel<64, 2, true, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 1, true, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 2, true, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 4, true, false, false>)};
  for (const void* f : ks) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace trr
