// step_rows2_nu.cu -- the two-rows-per-thread D3Q19 kernel in its viscosity-term
// mode (FP32 storage); a translation unit of its own so the build compiles it
// in parallel with the step instances.

#include "step_rows2.cuh"

namespace maclab {

template <int RM>
static cudaError_t nu_dispatch(int bxc, int tyt, const TiledArgs& ta, const void* in, void* out,
                               const CUtensorMap& tm_own, const CUtensorMap& tm_halo, cudaStream_t st, dim3 grid,
                               int* resident) {
  switch (bxc * 100 + tyt) {
    case 1604: return launch_rows2_shape<float, 16, 4, true, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
    case 3202: return launch_rows2_shape<float, 32, 2, true, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
    case 3204: return launch_rows2_shape<float, 32, 4, true, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
  }
  return cudaErrorInvalidValue;
}

cudaError_t rows2_nu_dispatch(int bxc, int tyt, const TiledArgs& ta, const void* in, const void* out,
                              const CUtensorMap& tm_own, const CUtensorMap& tm_halo, cudaStream_t st, dim3 grid,
                              int* resident) {
  void* o = const_cast<void*>(out);  // read only in this mode
  if (ta.ny % ta.ty == 0)
    return nu_dispatch<kRowsPlain>(bxc, tyt, ta, in, o, tm_own, tm_halo, st, grid, resident);
  return nu_dispatch<kRowsEven>(bxc, tyt, ta, in, o, tm_own, tm_halo, st, grid, resident);
}

}  // namespace maclab
