// step_rows2_s16.cu -- instances of the two-rows-per-thread D3Q19 step for
// BF16 and FP16 storage (FP32 arithmetic).

#include "step_rows2.cuh"

namespace maclab {
MACLAB_ROWS2_DISPATCH(, __nv_bfloat16, kRowsPlain)
MACLAB_ROWS2_DISPATCH(, __half, kRowsPlain)
}  // namespace maclab
