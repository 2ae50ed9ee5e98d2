// step_fold.cu -- host side of the D3Q19 step without halo-row threads
// (step_fold.cuh): block shapes, chunking of the march axis, instances.

#include <algorithm>

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

// Chunks of the march axis: an explicit tz gives ceil(nplanes / tz).  By default
// the count whose slowest SM ends first.  A chunk of p planes takes a block p +
// `start` plane times (its launch, first copies and two halo planes are worth
// `start`), a plane time grows with the warps that share a scheduler beyond
// `free` by `share` each, and blocks beyond what the device holds at once run in
// further waves.  (Fitted to cavities of 32^3 to 200 x 200 x 64; before, chunks
// had at least four planes: 32^3 6.9 -> 3.8 us a step, 64^3 7.1 -> 5.2, 72^3
// 9.5 -> 8.1, 192 x 192 x 64 28.9 -> 25.7.)
int fold_chunks(int nplanes, int ytiles, int tz_req, int per_sm, int threads, const ChunkCost& c) {
  if (tz_req > 0) return (nplanes + tz_req - 1) / tz_req;
  const int sms = sm_count(), resident = per_sm < 1 ? 1 : per_sm;
  int best = 1;
  double least = 1e300;
  for (int p = nplanes; p >= 1; --p) {
    const int nzc = (nplanes + p - 1) / p;
    if ((nplanes + nzc - 1) / nzc != p) continue;  // the same count with shorter chunks
    const int64_t blocks = (int64_t)nzc * ytiles;
    const int64_t waves = (blocks + (int64_t)resident * sms - 1) / ((int64_t)resident * sms);
    const int64_t per = std::min<int64_t>(resident, (blocks + sms - 1) / sms);
    const double warps = (double)((per * threads + 127) / 128);  // of the fullest scheduler
    const double cost = waves * (p + c.start) * (1.0 + (warps > c.free ? c.share * (warps - c.free) : 0.0));
    if (cost < least) {
      least = cost;
      best = nzc;
    }
  }
  return best;
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
  const int wall_pad = (g.periodic & 1u) ? 0 : g.pad;  // what moves the right wall
  const RowMode rows = (wall_pad & 1) ? kRowsOdd : (wall_pad || g.ny % s.ty != 0) ? kRowsEven : kRowsPlain;
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
  ta.nzc = fold_chunks(ta.nplanes, ytiles, tz, resident, s.bxc * s.ty, ChunkCost{1.3, 2.0, 0.3});
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
