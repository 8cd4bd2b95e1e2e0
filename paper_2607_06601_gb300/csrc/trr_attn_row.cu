// trr_attn_row.cu - the kernels of trr_decode_attn with one query head per warp (one mode per query).
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kRow, false, false)
}  // namespace trr
