// step_fold_f32.cu -- instances of the folded D3Q19 step for
// FP32 storage.

#include "step_fold.cuh"

namespace maclab {
MACLAB_FOLD_DISPATCH(, float, kRowsPlain)
}  // namespace maclab
