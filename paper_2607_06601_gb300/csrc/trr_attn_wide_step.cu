// trr_attn_wide_step.cu - the kernels of trr_decode_step with a KV head and 8 / (d/G) heads of its query
// group per warp, for groups wider than that.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kWide, true, false)
}  // namespace trr
