// step_rows2_f32_any.cu -- instances of the two-rows-per-thread D3Q19 step for
// FP32 storage,
// padded rows and ragged row counts.

#include "step_rows2.cuh"

namespace maclab {
MACLAB_ROWS2_DISPATCH(, float, kRowsEven)
MACLAB_ROWS2_DISPATCH(, float, kRowsOdd)
}  // namespace maclab
