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

// Chunks of the march axis: an explicit tz gives ceil(nplanes / tz).  By default as
// many as fill whole waves of resident blocks, for the number of waves that ends
// first: a chunk of p planes takes a block p + 1.2 plane times (its launch, first
// copies and two halo planes).  One wave in most cases; more where the tiles of a
// plane do not divide the resident blocks well (160^3: 7 chunks in one wave, 48.6 us
// a step; 15 in two, 49.5), where 64 more are looked at, so that a launch costs the
// host the same on any length.  Of 56 shapes from 16 x 16 x 600 to 512 x 128 x 256,
// FP32 and BF16, every one is within 1.3 % of the best count; both rules before it
// (at least four planes; a cost that grew with the warps of an SM) left some 5 to 15 %
// behind: 160 x 40 x 100 folded 12.7 -> 11.3, 64 x 64 x 64 two rows 5.5 -> 5.25, 32 x
// 64 x 256 11.1 -> 9.6.
//
// images: every step is followed by the kernel that renews the periodic images
// (launch_wrap_columns).  Its blocks find no place beside a last wave that takes up
// all there is, and the next step's then come late: 67^3 10.2 us a step with a
// seventh of the places left free, 13.1 without; 255 x 30 x 30 9.6 and 17.9.  A last
// wave that leaves less counts 2.4 plane times more, which long steps do not mind.
int fold_chunks(int nplanes, int ytiles, int tz_req, int per_sm, bool images) {
  if (tz_req > 0) return (nplanes + tz_req - 1) / tz_req;
  const int64_t all = (int64_t)sm_count() * (per_sm < 1 ? 1 : per_sm), left = images ? all / 7 : 0;
  int best = 1;
  int64_t least = INT64_MAX;
  for (const int64_t slots : {all, all - left}) {
    const int64_t first = (ytiles + slots - 1) / slots;  // waves of one chunk
    for (int64_t w = first; w <= first + 64; ++w) {
      const int chunks = (int)std::min<int64_t>(nplanes, w * slots / ytiles);
      const bool full = w * slots - (int64_t)chunks * ytiles + (all - slots) < left;
      const int64_t cost = w * (5 * (int64_t)((nplanes + chunks - 1) / chunks) + 6) + (full ? 12 : 0);
      if (cost < least) {
        least = cost;
        best = chunks;
      }
      if (chunks == nplanes) break;
    }
    if (!images) break;
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
  ta.nzc = fold_chunks(ta.nplanes, ytiles, tz, resident, wrap_columns(g));
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
