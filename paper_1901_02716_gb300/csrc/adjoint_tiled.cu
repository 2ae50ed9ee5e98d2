// adjoint_tiled.cu -- host side of the tiled reverse steps (adjoint_tiled.cuh, adjoint_rows.cuh):
// block shapes, instantiations and the launch.

#include "adjoint_rows.cuh"

namespace maclab {

namespace {

struct AdjShape {
  int bxc, ry, ty;  // threads along x, rows with halo, rows
  bool rows;        // adjoint_rows.cuh
};

// Tiled reverse steps built (us a step, periodic):
//  * adj_step_rows for natural rows in FP32 and interleaved rows in FP64, of 3
//    to 128 nodes in 3D and to 512 in 2D.  FP32 97x96x95: 32.5 (reference kernels
//    62.8), 33x40x50 9.9 (16.6), 255x256 6.1 (12.4); FP64 96^3: 328
//    (adj_step_tiled 479), 256^2 19.3 (32.1).
//  * adj_step_tiled for interleaved FP32 rows, whose threads keep twice the bytes
//    in flight: 96^3 19.1 (adj_step_rows 27.3), 128^3 38.8 (72.5); up to 512
//    nodes in 3D, 1024 in 2D.
// The rest takes the reference kernels, natural FP64 rows because they are
// faster there (97x64x64: 160, adj_step_rows 190).
// Blocks of adj_step_rows: FP32 8 rows with the halo, 53x61x47 12.1 (10 rows, one
// block an SM: 16.4) and 127x80x80 23.9 (6 rows: 32.7); FP64 is bound by its
// arithmetic, not by the blocks an SM holds: 32^3 34 (10 rows: 45), but with 64
// columns its registers spill (96^3: 356 with 64 x 8 threads).
bool adj_shape(const Geometry& g, int precision, AdjShape* s) {
  if (precision == MACLAB_BF16_STORE || precision == MACLAB_F16_STORE || g.nx < 3) return false;
  const bool f64 = precision == MACLAB_F64;
  if (f64 == (g.ilv != 0)) {  // FP32 natural, FP64 interleaved: AdjRows::NAT
    const int pairs = (g.nx + 1) / 2;
    if (g.d == 2) *s = pairs <= 64 ? AdjShape{64, 1, 1, true} : AdjShape{256, 1, 1, true};
    else if (pairs <= 32) *s = AdjShape{32, 8, 6, true};
    else if (f64) *s = pairs <= 48 ? AdjShape{48, 6, 4, true} : AdjShape{64, 6, 4, true};
    else *s = AdjShape{64, 8, 6, true};
    return pairs <= s->bxc;
  }
  if (f64) return false;
  const int bx = g.nx / 4;
  int bxc = 0;
  for (int c : {16, 32, 64, 128, 256})
    if (bx <= c) { bxc = c; break; }
  if (!bxc) return false;
  if (g.d == 2) {
    *s = AdjShape{bxc, 1, 1, false};
    return true;
  }
  int ty = 0;
  switch (bxc) {
    case 16: ty = 8; break;
    case 32: ty = 4; break;
    case 64: ty = 4; break;
    case 128: ty = 2; break;
    default: return false;
  }
  *s = AdjShape{bxc, ty + 2, ty, false};
  return true;
}

int sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
  }
  return n;
}

AdjArgs adj_args(const Geometry& g, int ty, const double* force, int overlap) {
  AdjArgs A{};
  A.overlap = overlap;
  A.nx = g.nx;
  A.ny = g.d == 3 ? g.ny : 1;
  A.nplanes = g.d == 3 ? g.nz : g.ny;
  A.n = g.n;
  A.plane_stride = (int64_t)g.nx * A.ny;
  A.ty = ty;
  A.px = (g.periodic & 1u) ? 1 : 0;
  A.py = g.d == 3 ? ((g.periodic & 2u) ? 1 : 0) : 0;
  A.pz = g.d == 3 ? ((g.periodic & 4u) ? 1 : 0) : ((g.periodic & 2u) ? 1 : 0);
  A.wall_mode = g.wall_mode;
  A.mask = g.mask;
  for (int i = 0; i < 3; ++i) A.force[i] = force[i];
  return A;
}

// Blocks along the march axis.
int adj_chunks(int nplanes, int ytiles, int resident) {
  // about 8 planes per block, rounded up to whole waves of resident blocks
  int nzc = (nplanes + 7) / 8;
  const long slots = (long)resident * sms();
  const long blocks = (long)nzc * ytiles;
  const long waves = (blocks + slots - 1) / slots;
  nzc = (int)((waves * slots) / ytiles);
  if (nzc > nplanes / 2) nzc = nplanes / 2 > 0 ? nplanes / 2 : 1;
  if (nzc < 1) nzc = 1;
  return nzc;
}

template <int LAT, typename S>
cudaError_t tiled_dispatch(const AdjShape& s, const AdjArgs& A, const void* sn, const void* sn1,
                           const void* lam1, void* lam0, double* gf, cudaStream_t st, int ytiles,
                           int* resident) {
#define MACLAB_ADJ_ROWS(BXC, RY)         \
  if (s.rows && s.bxc == BXC && s.ry == RY) \
    return launch_adj_rows<LAT, S, BXC, RY>(A, sn, sn1, lam1, lam0, gf, st, ytiles, resident);
#define MACLAB_ADJ_TILED(BXC, RY) \
  if (!s.rows && s.bxc == BXC)    \
    return launch_adj_tiled<LAT, S, BXC, RY>(A, sn, sn1, lam1, lam0, gf, st, ytiles, resident);
  constexpr bool f64 = sizeof(S) == 8;
  if constexpr (LAT == kD2Q9) {
    MACLAB_ADJ_ROWS(64, 1)
    MACLAB_ADJ_ROWS(256, 1)
    if constexpr (!f64) {
      MACLAB_ADJ_TILED(16, 1)
      MACLAB_ADJ_TILED(32, 1)
      MACLAB_ADJ_TILED(64, 1)
      MACLAB_ADJ_TILED(128, 1)
      MACLAB_ADJ_TILED(256, 1)
    }
  } else {
    MACLAB_ADJ_ROWS(32, 8)
    if constexpr (f64) {
      MACLAB_ADJ_ROWS(48, 6)
      MACLAB_ADJ_ROWS(64, 6)
    } else {
      MACLAB_ADJ_ROWS(64, 8)
      MACLAB_ADJ_TILED(16, 10)
      MACLAB_ADJ_TILED(32, 6)
      MACLAB_ADJ_TILED(64, 6)
      MACLAB_ADJ_TILED(128, 4)
    }
  }
#undef MACLAB_ADJ_ROWS
#undef MACLAB_ADJ_TILED
  return cudaErrorInvalidValue;
}

template <int LAT, typename S>
cudaError_t tiled_adjoint_t(const Geometry& g, const AdjShape& s, const void* sn, const void* sn1,
                            const void* lam1, void* lam0, const double* force, double* gf,
                            int overlap, cudaStream_t st) {
  AdjArgs A = adj_args(g, s.ty, force, overlap);
  const int ytiles = g.d == 3 ? (A.ny + s.ty - 1) / s.ty : 1;
  int resident = 0;
  cudaError_t e = tiled_dispatch<LAT, S>(s, A, sn, sn1, lam1, lam0, gf, st, ytiles, &resident);
  if (e != cudaSuccess) return e;
  A.nzc = adj_chunks(A.nplanes, ytiles, resident);
  return tiled_dispatch<LAT, S>(s, A, sn, sn1, lam1, lam0, gf, st, ytiles, nullptr);
}

}  // namespace

bool tiled_adjoint_supported(const Geometry& g, int precision) {
  AdjShape s;
  return adj_shape(g, precision, &s);
}

cudaError_t launch_tiled_adjoint(const Geometry& g, int precision, const void* state_n,
                                 const void* state_np1, const void* lam_np1, void* lam_n,
                                 const double force_lat[3], double* grad_force, int overlap, cudaStream_t st) {
  AdjShape s;
  if (!adj_shape(g, precision, &s)) return cudaErrorInvalidValue;
  if (g.lattice == kD2Q9) {
    if (precision == MACLAB_F64)
      return tiled_adjoint_t<kD2Q9, double>(g, s, state_n, state_np1, lam_np1, lam_n, force_lat, grad_force, overlap, st);
    return tiled_adjoint_t<kD2Q9, float>(g, s, state_n, state_np1, lam_np1, lam_n, force_lat, grad_force, overlap, st);
  }
  if (precision == MACLAB_F64)
    return tiled_adjoint_t<kD3Q19, double>(g, s, state_n, state_np1, lam_np1, lam_n, force_lat, grad_force, overlap, st);
  return tiled_adjoint_t<kD3Q19, float>(g, s, state_n, state_np1, lam_np1, lam_n, force_lat, grad_force, overlap, st);
}

// adj_nu_rows where it beats the per-node kernel (us, per node and by rows): 29^3 8.3
// and 7.4; then its blocks, one an SM, march too few planes each (33^3 8.3 and 9.3,
// 111 x 24 x 24 8.7 and 10.1, 49^3 10.3 and 12.4), until the nodes count (53^3 12.4 and
// 12.3, 63^3 14.5 and 13.2, 127 x 80 x 80 35 and 22).
bool rows_nu_supported(const Geometry& g, int precision) {
  AdjShape s;
  if (g.n > 26000 && g.n < 148000) return false;
  return precision == MACLAB_F32 && g.d == 3 && adj_shape(g, precision, &s) && s.rows;
}

cudaError_t launch_rows_nu(const Geometry& g, const void* state_n, const void* state_np1, const void* lam_np1,
                           const double force_lat[3], double* acc, int overlap, cudaStream_t st) {
  AdjShape s;
  if (!rows_nu_supported(g, MACLAB_F32) || !adj_shape(g, MACLAB_F32, &s)) return cudaErrorInvalidValue;
  AdjArgs A = adj_args(g, s.ty, force_lat, overlap);
  const int ytiles = (A.ny + s.ty - 1) / s.ty;
  auto launch = [&](int* resident) {
    return s.bxc == 32 ? launch_nu_rows<32, 8>(A, state_n, state_np1, lam_np1, acc, st, ytiles, resident)
                       : launch_nu_rows<64, 8>(A, state_n, state_np1, lam_np1, acc, st, ytiles, resident);
  };
  int resident = 0;
  const cudaError_t e = launch(&resident);
  if (e != cudaSuccess) return e;
  A.nzc = adj_chunks(A.nplanes, ytiles, resident);
  return launch(nullptr);
}

}  // namespace maclab
