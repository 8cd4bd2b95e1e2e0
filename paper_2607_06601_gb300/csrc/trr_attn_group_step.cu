// trr_attn_group_step.cu - the kernels of trr_decode_step with a KV head and its query group per warp.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kGroup, true, false)
}  // namespace trr
