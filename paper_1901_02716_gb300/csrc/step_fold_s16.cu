// step_fold_s16.cu -- instances of the folded D3Q19 step for
// BF16 and FP16 storage (FP32 arithmetic).

#include "step_fold.cuh"

namespace maclab {
MACLAB_FOLD_DISPATCH(, __nv_bfloat16, kRowsPlain)
MACLAB_FOLD_DISPATCH(, __half, kRowsPlain)
}  // namespace maclab
