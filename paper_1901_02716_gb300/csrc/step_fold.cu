// step_fold.cu -- host side of the D3Q19 step without halo-row threads
// (step_fold.cuh): block shapes, chunking of the march axis, instances.

#include "step_fold.cuh"

namespace maclab {

MACLAB_FOLD_DISPATCH(extern, float, kRowsPlain)
MACLAB_FOLD_DISPATCH(extern, float, kRowsEven)
MACLAB_FOLD_DISPATCH(extern, float, kRowsOdd)
MACLAB_FOLD_DISPATCH(extern, __nv_bfloat16, kRowsPlain)
MACLAB_FOLD_DISPATCH(extern, __nv_bfloat16, kRowsEven)
MACLAB_FOLD_DISPATCH(extern, __nv_bfloat16, kRowsOdd)
MACLAB_FOLD_DISPATCH(extern, __half, kRowsPlain)
MACLAB_FOLD_DISPATCH(extern, __half, kRowsEven)
MACLAB_FOLD_DISPATCH(extern, __half, kRowsOdd)

namespace {

// Instantiated (BXC, TY) in order of preference for each width (the first whose
// TY divides ny is the default): FP32 all of them, 16-bit storage (32, 8),
// (32, 4), (64, 4) and (128, 4).
constexpr FoldShape kFoldShapes[] = {{16, 8}, {32, 8}, {32, 4}, {64, 4}, {64, 8}, {128, 4}};

bool fold_shape_built(const FoldShape& s, int precision) {
  if (precision == MACLAB_F32) return true;
  if (precision == MACLAB_BF16_STORE || precision == MACLAB_F16_STORE)
    return (s.bxc == 32 && (s.ty == 8 || s.ty == 4)) || ((s.bxc == 64 || s.bxc == 128) && s.ty == 4);
  return false;
}

// ragged: where no TY divides ny, the first that does not exceed it (the last
// tile recomputes at most TY - 1 rows; the tiled kernel, which otherwise serves
// these, forms two halo rows for every tile: 15 steps of a 256 x 327 x 377
// cavity in BF16 storage take 6.0 ms on it and 3.5 ms here).
bool fold_shape(const Geometry& g, int precision, int ty_req, FoldShape* out, bool ragged) {
  if (g.d != 3 || g.lattice != kD3Q19 || !g.ilv || precision == MACLAB_F64) return false;
  const int bx = g.nx / 4;
  int bxc = 0;
  for (int c : {16, 32, 64, 128})
    if (bx <= c) { bxc = c; break; }
  if (!bxc) return false;
  for (const bool divides : {true, false}) {
    if (!divides && !ragged) break;
    for (const FoldShape& s : kFoldShapes) {
      if (s.bxc != bxc || (ty_req > 0 && s.ty != ty_req) || !fold_shape_built(s, precision)) continue;
      if (divides ? g.ny % s.ty != 0 : g.ny < s.ty) continue;
      *out = s;
      return true;
    }
  }
  return false;
}

}  // namespace

static int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 148;
  }
  return sms;
}

// Chunks of the march axis: an explicit tz gives ceil(nplanes / tz).  By
// default the chunks are as long as possible (every chunk re-reads and
// half-processes a plane at each end) while the grid still fills two waves of
// resident blocks: 32 planes, halved down to 8 until it does; then the block
// count is rounded up to whole waves and chunks are kept to at least 4 planes.
int fold_chunks(int nplanes, int ytiles, int tz_req, int per_sm) {
  if (tz_req > 0) return (nplanes + tz_req - 1) / tz_req;
  const long slots = (long)sm_count() * (per_sm < 1 ? 1 : per_sm);
  int tz = 32;
  while (tz > 8 && (long)((nplanes + tz - 1) / tz) * ytiles < 2 * slots) tz /= 2;
  const long blocks = (long)((nplanes + tz - 1) / tz) * ytiles;
  const long waves = (blocks + slots - 1) / slots;
  int nzc = (int)((waves * slots) / ytiles);
  const int max_chunks = nplanes / 4 > 0 ? nplanes / 4 : 1;
  if (nzc > max_chunks) nzc = max_chunks;
  if (nzc < 1) nzc = 1;
  return nzc;
}


bool fold_supported(const Geometry& g, int precision, int ty, bool ragged) {
  FoldShape s;
  return fold_shape(g, precision, ty, &s, ragged);
}

int fold_threads(const Geometry& g, int precision, int ty) {
  FoldShape s;
  return fold_shape(g, precision, ty, &s, true) ? s.bxc * s.ty : 0;
}

cudaError_t launch_fold(const StepLaunch& sl, cudaStream_t stream, int ty, int tz) {
  const Geometry& g = sl.g;
  FoldShape s;
  if (!fold_shape(g, sl.precision, ty, &s, true)) return cudaErrorInvalidValue;
  TiledArgs ta{};
  ta.nx = g.nx;
  ta.ny = g.ny;
  ta.nplanes = g.nz;
  ta.n = g.n;
  ta.plane_stride = (int64_t)g.nx * g.ny;
  ta.ty = s.ty;
  const int ytiles = (g.ny + s.ty - 1) / s.ty;
  const RowMode rows = (g.pad & 1) ? kRowsOdd : (g.pad || g.ny % s.ty != 0) ? kRowsEven : kRowsPlain;
  auto dispatch = [&](const void* in, void* out, dim3 grid, int* resident) {
    auto typed = [&](auto zero) {
      using S = decltype(zero);
      switch (rows) {
        case kRowsPlain: return fold_dispatch<S, kRowsPlain>(s, ta, in, out, stream, grid, resident);
        case kRowsEven: return fold_dispatch<S, kRowsEven>(s, ta, in, out, stream, grid, resident);
        default: return fold_dispatch<S, kRowsOdd>(s, ta, in, out, stream, grid, resident);
      }
    };
    switch (sl.precision) {
      case MACLAB_F32: return typed(float{});
      case MACLAB_BF16_STORE: return typed(__nv_bfloat16{});
      case MACLAB_F16_STORE: return typed(__half{});
    }
    return cudaErrorInvalidValue;
  };
  int resident = 0;
  cudaError_t e = dispatch(nullptr, nullptr, dim3(), &resident);
  if (e != cudaSuccess) return e;
  ta.nzc = fold_chunks(ta.nplanes, ytiles, tz, resident);
  ta.px = (g.periodic & 1u) ? 1 : 0;
  ta.py = (g.periodic & 2u) ? 1 : 0;
  ta.pz = (g.periodic & 4u) ? 1 : 0;
  ta.wall_mode = g.wall_mode;
  ta.mask = g.mask;
  for (int i = 0; i < 3; ++i) ta.force[i] = sl.force[i];
  ta.set_overlap_pad(sl.overlap, g.pad);
  return dispatch(sl.in, sl.out, dim3(ta.nzc, ytiles), nullptr);
}

}  // namespace maclab
