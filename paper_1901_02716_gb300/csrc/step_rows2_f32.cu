// step_rows2_f32.cu -- instances of the two-rows-per-thread D3Q19 step for
// FP32 storage.

#include "step_rows2.cuh"

namespace maclab {
MACLAB_ROWS2_DISPATCH(, float, kRowsPlain)
}  // namespace maclab
