// trr_attn_row_step.cu - the kernels of trr_decode_step with one query head per warp.
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kRow, true, false)
}  // namespace trr
