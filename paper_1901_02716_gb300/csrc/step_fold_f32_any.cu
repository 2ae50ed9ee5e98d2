// step_fold_f32_any.cu -- instances of the folded D3Q19 step for
// FP32 storage,
// padded rows and ragged row counts.

#include "step_fold.cuh"

namespace maclab {
MACLAB_FOLD_DISPATCH(, float, kRowsEven)
MACLAB_FOLD_DISPATCH(, float, kRowsOdd)
}  // namespace maclab
