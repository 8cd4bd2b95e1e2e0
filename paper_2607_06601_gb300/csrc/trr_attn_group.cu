// trr_attn_group.cu - the kernels of trr_decode_attn with a KV head and its query group per warp
// (g >= 2 whose (head, group) columns fit one 8-wide mma tile), and the kernel that merges their
// split partials.
#include "trr_row.cuh"

namespace trr {

TRR_ROW_FAMILY(, kGroup, false, false)

cudaError_t launch_attn_combine(int d, int ctas, cudaStream_t s, const CombineArgs& ca) {
  return d == 64 ? launch_pdl(attn_combine_kernel<64>, dim3(ctas), dim3(32 * kCombineWarps), 0, s, ca)
                 : launch_pdl(attn_combine_kernel<128>, dim3(ctas), dim3(32 * kCombineWarps), 0, s, ca);
}

}  // namespace trr
