// trr_attn_row.cu - the kernels of trr_decode_attn with one query head per warp
// (one mode per query): one instance per head size and groups
// per head.
#include "trr_row.cuh"

namespace trr {

template <int D, int NG>
static cudaError_t launch(dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  return launch_pdl(row_kernel<D, NG, false, false, false>, grid, dim3(32 * kRowWarps), smem, s, k);
}

cudaError_t launch_attn_row(const Layout& l, dim3 grid, size_t smem, cudaStream_t s, const AttnKernelArgs& k) {
  const int ng = l.d / l.G;
  if (l.d == 64) return ng == 1 ? launch<64, 1>(grid, smem, s, k) : launch<64, 2>(grid, smem, s, k);
  if (ng == 1) return launch<128, 1>(grid, smem, s, k);
  return ng == 2 ? launch<128, 2>(grid, smem, s, k) : launch<128, 4>(grid, smem, s, k);
}

cudaError_t configure_attn_row() {
  const void* ks[] = {reinterpret_cast<const void*>(row_kernel<64, 1, false, false, false>),
                      reinterpret_cast<const void*>(row_kernel<64, 2, false, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 1, false, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 2, false, false, false>),
                      reinterpret_cast<const void*>(row_kernel<128, 4, false, false, false>)};
  for (const void* f : ks) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemLimit);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace trr
