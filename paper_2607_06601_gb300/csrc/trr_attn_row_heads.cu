// trr_attn_row_heads.cu - the kernels of trr_decode_attn with one query head per warp (a mode per head).
#include "trr_row.cuh"

namespace trr {
TRR_ROW_FAMILY(, kHeads, false, false)
}  // namespace trr
