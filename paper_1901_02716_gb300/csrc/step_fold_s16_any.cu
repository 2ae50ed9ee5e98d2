// step_fold_s16_any.cu -- instances of the folded D3Q19 step for
// BF16 and FP16 storage (FP32 arithmetic),
// padded rows and ragged row counts.

#include "step_fold.cuh"

namespace maclab {
MACLAB_FOLD_DISPATCH(, __nv_bfloat16, kRowsEven)
MACLAB_FOLD_DISPATCH(, __nv_bfloat16, kRowsOdd)
MACLAB_FOLD_DISPATCH(, __half, kRowsEven)
MACLAB_FOLD_DISPATCH(, __half, kRowsOdd)
}  // namespace maclab
