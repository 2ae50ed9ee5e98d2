// step_rows2_s16_any.cu -- instances of the two-rows-per-thread D3Q19 step for
// BF16 and FP16 storage (FP32 arithmetic),
// padded rows and ragged row counts.

#include "step_rows2.cuh"

namespace maclab {
MACLAB_ROWS2_DISPATCH(, __nv_bfloat16, kRowsEven)
MACLAB_ROWS2_DISPATCH(, __nv_bfloat16, kRowsOdd)
MACLAB_ROWS2_DISPATCH(, __half, kRowsEven)
MACLAB_ROWS2_DISPATCH(, __half, kRowsOdd)
}  // namespace maclab
