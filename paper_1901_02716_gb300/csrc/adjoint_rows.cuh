// adjoint_rows.cuh -- reverse step on natural rows (nx not a multiple of 4) in
// FP32 and on interleaved rows in FP64.  The arithmetic of adjoint.cu, the
// staging of adjoint_tiled.cuh with one node pair (x, x + H), H = (nx + 1) / 2,
// a thread.  In an odd row the last pair's second lane stands for the image of
// node 0: its record is that node's, it is neither stored nor counted, and the
// seam copy takes node nx - 1 from the pair before.
//
// Factored by planes as the step is (d3q19.cuh): a destination reads the nine
// records around it in each plane once, not 19 over three planes; from them
// come the sums of the plane's own directions and, with g = b +- L_z, those of
// the directions to the plane above and below, carried along the march (integer
// weights 36 w, divided out at the end).  That is half the arithmetic and half
// the shared-memory reads of the direct sum, and two staged planes instead of
// four.  Bound by latency and by the halo rows and planes, whose records are
// formed again by every block (FP32 97x96x95: 32.5 us for 33 MB of states and
// adjoints read three times and written once; the reference kernels took 62.8),
// in FP64 by the arithmetic pipe (96^3: 328 us, the direct sums 478).
#pragma once
#include "adjoint_tiled.cuh"

namespace maclab {

// Weighted sums (x 36) of g over the neighbours in one plane along the march
// axis: t all five (three in 2D), s and d sum and difference along x and y.
template <typename P>
struct AdjBelow {
  P t, sx, dx, sy, dy;
};
// Moments of a destination before the plane above it: G0, G1 and G2 of its own
// plane and the plane below, whose t, dx, dy also enter the components along
// the march axis.
template <typename P>
struct AdjPend {
  P g0, x, y, xx, yy, xy, t, dx, dy;
};

template <int LAT, typename S, int BXC, int RY>
struct AdjRows {
  using C = typename Store<S>::C;
  using P = typename Pair<C>::P;
  static constexpr bool NAT = sizeof(S) == 4;     // natural rows (FP64: interleaved)
  static constexpr int D = Lattice<LAT>::D;
  static constexpr int K = D + 1;                 // record components: L_r, L_m
  static constexpr int G = AdjUnit<P>::G;         // components per unit
  static constexpr int NU = (K + G - 1) / G;      // units per pair record
  static constexpr int W = BXC + 2;               // columns, with the two seam copies
  static constexpr int SEAM_L = BXC, SEAM_R = BXC + 1;
  static constexpr int STAGES = 2;
  static constexpr int STAGE = RY * NU * W;   // units per stage
  static constexpr int THREADS = BXC * RY;
  static constexpr int MIN_BLOCKS = sizeof(S) == 8 || THREADS > 256 ? 1 : 2;
  static constexpr bool PREFETCH = sizeof(C) == 4;  // registers for a plane in flight (FP64 has none to spare)
  __host__ __device__ static constexpr size_t smem_bytes() { return (size_t)16 * STAGES * STAGE; }
  __device__ __forceinline__ static constexpr int unit(int k, int rr, int u, int col) {
    return ((k * RY + rr) * NU + u) * W + col;
  }
};

template <int LAT, typename S, int BXC, int RY>
__global__ void __launch_bounds__(BXC * RY, (AdjRows<LAT, S, BXC, RY>::MIN_BLOCKS))
    adj_step_rows(AdjArgs A, const S* __restrict__ in_state, const S* __restrict__ out_state,
                   const typename Store<S>::C* __restrict__ lam1, typename Store<S>::C* __restrict__ lam0,
                   double* __restrict__ grad_force) {
  using T = AdjRows<LAT, S, BXC, RY>;
  using C = typename T::C;
  using O = Pair<C>;
  using P = typename O::P;
  using U = AdjUnit<P>;
  using L = Lattice<LAT>;
  using F = Frame<LAT>;
  constexpr bool NAT = T::NAT;
  constexpr int D = T::D, K = T::K, G = T::G, NU = T::NU;
  extern __shared__ __align__(16) uint4 units[];
  pdl_wait();  // the previous kernel's writes are visible from here on
  pdl_launch_next();
  const int tx = threadIdx.x, r = threadIdx.y;
  const int H = (A.nx + 1) >> 1;
  const int bxr = H;
  const bool active = tx < bxr;

  int row = 0, row_mem = 0;
  bool row_exists = true, interior = true;
  if (D == 3) {
    row = blockIdx.y * A.ty + r - 1;
    interior = r >= 1 && r <= RY - 2 && row < A.ny;
    row_mem = row;
    if (row < 0 || row >= A.ny) {
      if (A.py) row_mem = (row + A.ny) % A.ny;
      else row_exists = false;
    }
  }
  interior = interior && active;
  const bool stages_own = active && row_exists;
  const int64_t row_off = (int64_t)row_mem * A.nx + (NAT ? tx : 2 * tx);  // storage index of lane x in a plane
  const bool two = !NAT || tx + H < A.nx;  // lane y of the last pair of an odd row is the image of node 0
  const int hi = two ? H : -tx;            // from lane x to lane y (natural rows)

  const int z0 = (int)(((int64_t)blockIdx.x * A.nplanes) / A.nzc);
  const int z1 = (int)(((int64_t)(blockIdx.x + 1) * A.nplanes) / A.nzc);
  auto plane_exists = [&](int p) { return (p >= 0 && p < A.nplanes) || A.pz; };
  auto plane_mem = [&](int p) { return p < 0 ? p + A.nplanes : (p >= A.nplanes ? p - A.nplanes : p); };

  // wall lanes as bits 0 and 1; box walls off the march axis are fixed per thread
  uint32_t box_bits = 0;
  if (A.wall_mode == kWallBox) {
    if (!A.px) box_bits |= (tx == 0 ? 1u : 0u) | (tx == A.nx - 1 - H || !two ? 2u : 0u);
    if (D == 3 && !A.py && (row_mem == 0 || row_mem == A.ny - 1)) box_bits = 3u;
  }

  P force[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) force[i] = O::splat(C(A.force[i]));
  NuAcc<C> gf[3];  // sums of lam' over the fluid nodes

  auto ld = [&](const C* p) {
    P v;
    if constexpr (NAT) v.x = p[0], v.y = p[hi];
    else v = *reinterpret_cast<const P*>(p);
    return v;
  };
  // post-step state and lam' of this thread's pair in one plane
  struct Raw {
    P st[K], lm[K];
    uint32_t wall;
    bool have;
  };
  auto load_raw = [&](int p, Raw& R) {
    R.have = stages_own && plane_exists(p);
    R.wall = 0;
    if (R.have) {
      const int pm = plane_mem(p);
      const int64_t off = (int64_t)pm * A.plane_stride + row_off;
#pragma unroll
      for (int f = 0; f < K; ++f) {
        R.st[f] = ld(out_state + f * A.n + off);
        R.lm[f] = ld(lam1 + f * A.n + off);
      }
      if (A.wall_mode == kWallMask) {
        R.wall = (A.mask[off] ? 1u : 0u) | (A.mask[off + (NAT ? hi : 1)] ? 2u : 0u);
      } else if (A.wall_mode == kWallBox) {
        R.wall = (!A.pz && (pm == 0 || pm == A.nplanes - 1)) ? 3u : box_bits;
      }
    }
  };

  uint32_t wq = 0;  // wall bits of the last staged planes, newest in bits 0..3
  // records of plane p into stage p & 3 (zeros where the row or plane is absent)
  auto stage = [&](int p, const Raw& R) {
    wq = (wq << 2) | R.wall;
    if (!active) return;
    const int k = p & (T::STAGES - 1);
    P rec[NU * G];
#pragma unroll
    for (int c = 0; c < NU * G; ++c) rec[c] = O::splat(C(0));
    if (R.have) {
      const bool counted = interior && p >= z0 && p < z1 && grad_force;
      const P inv = O::rcp(O::add(O::splat(C(1)), R.st[0]));
      P lr = R.lm[0];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const P um = adj_sub<C>(R.st[1 + i], force[i]);  // m' / rho'
        lr = adj_sub<C>(lr, O::mul(O::mul(R.lm[1 + i], um), inv));
        rec[1 + i] = O::mul(R.lm[1 + i], inv);
      }
      rec[0] = lr;
      const bool w0 = R.wall & 1u, w1 = R.wall & 2u;
#pragma unroll
      for (int c = 0; c < K; ++c) {  // walls carry no (L_r, L_m)
        if (w0) rec[c].x = C(0);
        if (w1) rec[c].y = C(0);
      }
      if (counted) {
#pragma unroll
        for (int i = 0; i < D; ++i) {
          gf[i].add(w0 ? C(0) : R.lm[1 + i].x);
          gf[i].add(w1 || !two ? C(0) : R.lm[1 + i].y);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < NU; ++u) U::st(&units[T::unit(k, r, u, tx)], &rec[u * G]);
    // the left neighbours (nx - 1, H - 1) of the first pair
    if (tx == bxr - 1 || tx == A.nx - 1 - H)
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        C* const seam = reinterpret_cast<C*>(&units[T::unit(k, r, u, T::SEAM_L)]);
#pragma unroll
        for (int c = 0; c < G; ++c) {
          if (tx == A.nx - 1 - H) seam[2 * c] = rec[u * G + c].y;
          if (tx == bxr - 1) seam[2 * c + 1] = rec[u * G + c].x;
        }
      }
    if (tx == 0)  // swapped first pair: right neighbours of the last one
#pragma unroll
      for (int u = 0; u < NU; ++u) U::st_swapped(&units[T::unit(k, r, u, T::SEAM_R)], &rec[u * G]);
  };

  const int col_l = tx == 0 ? T::SEAM_L : tx - 1;
  const int col_r = tx == bxr - 1 ? T::SEAM_R : tx + 1;
  constexpr int iy = D == 3 ? 1 : 0, iz = D - 1;  // components along y (3D) and the march axis
  // The rounded weights are those of the reference kernels: 1 / 36 scales all
  // (axes: twice that), and a rest weight rounded by itself differs from wc / 36
  // by a little more.  In sum lam grows by 1.5e-8 a step, as there; dL/dnu keeps
  // the offset against the forward steps' rounding that it had with them.
  constexpr C rest = C((double)(C(D == 3 ? 12 : 16) / C(36)) / (double)C(1.0 / 36.0) - (D == 3 ? 12.0 : 16.0));
  constexpr int wc = D == 3 ? 12 : 16, wa = D == 3 ? 2 : 4;  // 36 w: rest, axes (diagonals 1)

  AdjPend<P> pend{};    // of plane p - 1: its own plane's sums and those from below
  AdjBelow<P> below{};  // what plane p - 1 sends to plane p
  Raw R;
  load_raw(z0 - 1, R);
  stage(z0 - 1, R);
  load_raw(z0, R);
  for (int p = z0 - 1; p <= z1; ++p) {
    const int q = p - 1;  // the plane this one completes
    const int64_t off = (int64_t)q * A.plane_stride + row_off;
    __syncthreads();  // plane p is staged, the reads of plane p - 1 are done
    if (p < z1) {
      if constexpr (!T::PREFETCH) load_raw(p + 1, R);
      stage(p + 1, R);
      if constexpr (T::PREFETCH)
        if (p + 1 < z1) load_raw(p + 2, R);
    } else {
      wq <<= 2;
    }
    if (!interior) continue;
    const uint32_t wd = (wq >> 4) & 3u;  // wall lanes of plane q
    P st[K], res[K];
    if (q >= z0)
#pragma unroll
      for (int f = 0; f < K; ++f) st[f] = ld(in_state + f * A.n + off);
    // the record at (cx, cy) from this pair
    auto rec = [&](int cx, int cy, P* v) {
      const int col = cx == 0 ? tx : cx == 1 ? col_r : col_l;
#pragma unroll
      for (int u = 0; u < NU; ++u) U::ld(&units[T::unit(p & (T::STAGES - 1), r + cy, u, col)], &v[u * G]);
    };
    // g at the neighbours in the plane's axes, and what c_z = +-1 adds to it
    AdjBelow<P> up, dn;
    P vc[NU * G], ve[NU * G], vw[NU * G];
    rec(0, 0, vc);
    rec(1, 0, ve);
    rec(-1, 0, vw);
    const P ge = O::add(ve[0], ve[1]), gw = adj_sub<C>(vw[0], vw[1]);
    const P se = O::add(ge, gw), de = adj_sub<C>(ge, gw);
    {
      const P zs = O::add(ve[1 + iz], vw[1 + iz]), zd = adj_sub<C>(ve[1 + iz], vw[1 + iz]);
      up.sx = O::add(se, zs);
      dn.sx = adj_sub<C>(se, zs);
      up.dx = O::add(de, zd);
      dn.dx = adj_sub<C>(de, zd);
      up.t = O::fma(O::add(vc[0], vc[1 + iz]), O::splat(C(wa)), up.sx);
      dn.t = O::fma(adj_sub<C>(vc[0], vc[1 + iz]), O::splat(C(wa)), dn.sx);
    }
    AdjPend<P> own{};
    own.x = O::mul(de, O::splat(C(wa)));
    own.xx = O::mul(se, O::splat(C(wa)));
    own.g0 = O::fma(vc[0], O::splat(C(wc)), O::fma(vc[0], O::splat(rest), own.xx));
    if constexpr (D == 3) {
      P vn[NU * G], vs[NU * G];
      rec(0, 1, vn);
      rec(0, -1, vs);
      const P gn = O::add(vn[0], vn[1 + iy]), gs = adj_sub<C>(vs[0], vs[1 + iy]);
      const P sn = O::add(gn, gs), dnn = adj_sub<C>(gn, gs);
      const P zs = O::add(vn[1 + iz], vs[1 + iz]), zd = adj_sub<C>(vn[1 + iz], vs[1 + iz]);
      up.sy = O::add(sn, zs);
      dn.sy = adj_sub<C>(sn, zs);
      up.dy = O::add(dnn, zd);
      dn.dy = adj_sub<C>(dnn, zd);
      up.t = O::add(up.t, up.sy);
      dn.t = O::add(dn.t, dn.sy);
      // diagonals of the plane: north (east, west), south
      P v[NU * G];
      rec(1, 1, v);
      const P gne = O::add(v[0], O::add(v[1], v[1 + iy]));
      rec(-1, 1, v);
      const P gnw = O::add(v[0], adj_sub<C>(v[1 + iy], v[1]));
      rec(1, -1, v);
      const P gse = O::add(v[0], adj_sub<C>(v[1], v[1 + iy]));
      rec(-1, -1, v);
      const P gsw = adj_sub<C>(v[0], O::add(v[1], v[1 + iy]));
      const P north = O::add(gne, gnw), south = O::add(gse, gsw);
      const P nd = adj_sub<C>(gne, gnw), sd = adj_sub<C>(gse, gsw);
      const P all = O::add(north, south);
      own.y = O::fma(dnn, O::splat(C(wa)), adj_sub<C>(north, south));
      own.yy = O::fma(sn, O::splat(C(wa)), all);
      own.xy = adj_sub<C>(nd, sd);
      own.x = O::add(own.x, O::add(nd, sd));
      own.g0 = O::add(own.g0, own.yy);
      own.xx = O::add(own.xx, all);
    }
    if (q >= z0) {
      const AdjPend<P>& h = pend;
      const P G0 = O::add(h.g0, up.t);
      P G1[3], G2[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        G1[i] = O::splat(C(0));
#pragma unroll
        for (int j = 0; j < 3; ++j) G2[i][j] = O::splat(C(0));
      }
      G1[0] = O::add(h.x, up.dx);
      G2[0][0] = O::add(h.xx, up.sx);
      if constexpr (D == 3) {
        G1[iy] = O::add(h.y, up.dy);
        G2[iy][iy] = O::add(h.yy, up.sy);
        G2[0][iy] = h.xy;
        G2[iy][iz] = adj_sub<C>(up.dy, h.dy);
      }
      G1[iz] = adj_sub<C>(up.t, h.t);
      G2[iz][iz] = O::add(up.t, h.t);
      G2[0][iz] = adj_sub<C>(up.dx, h.dx);
      // equilibrium Jacobian at the destination (its own state)
      const P rho = O::add(O::splat(C(1)), st[0]);
      P u[3], G2u[3];
      P uu = O::splat(C(0)), uG1 = O::splat(C(0)), uG2u = O::splat(C(0));
#pragma unroll
      for (int i = 0; i < D; ++i) {
        u[i] = st[1 + i];
        uu = O::fma(u[i], u[i], uu);
        uG1 = O::fma(u[i], G1[i], uG1);
      }
#pragma unroll
      for (int i = 0; i < D; ++i) {
        G2u[i] = O::splat(C(0));
#pragma unroll
        for (int j = 0; j < D; ++j) G2u[i] = O::fma(i <= j ? G2[i][j] : G2[j][i], u[j], G2u[i]);
        uG2u = O::fma(u[i], G2u[i], uG2u);
      }
      // sums carry the factor 36 of the integer weights
      const P k36 = O::splat(C(1.0 / 36.0));
      P lr = O::fma(O::fma(uu, O::splat(C(-1.5)), O::splat(C(1))), G0,
                    O::fma(uG1, O::splat(C(3)), O::mul(uG2u, O::splat(C(4.5)))));
      res[0] = O::mul(lr, k36);
      const P rk = O::mul(rho, k36);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        P t = O::fma(G2u[i], O::splat(C(9)), O::mul(G1[i], O::splat(C(3))));
        t = adj_sub<C>(t, O::mul(O::mul(u[i], G0), O::splat(C(3))));
        res[1 + i] = O::mul(rk, t);
      }
    }
    // plane p: its own sums and what plane p - 1 sent up
    const AdjBelow<P>& b = below;
    pend.g0 = O::add(own.g0, b.t);
    pend.x = O::add(own.x, b.dx);
    pend.xx = O::add(own.xx, b.sx);
    pend.t = b.t;
    pend.dx = b.dx;
    if constexpr (D == 3) {
      pend.y = O::add(own.y, b.dy);
      pend.yy = O::add(own.yy, b.sy);
      pend.xy = own.xy;
      pend.dy = b.dy;
    }
    below = dn;
    if (q >= z0) {
      if (wd) {  // a wall node's output is its input: pass lam' through
#pragma unroll
        for (int f = 0; f < K; ++f) {
          const P l1 = ld(lam1 + f * A.n + off);
          if (wd & 1u) res[f].x += l1.x;
          if (wd & 2u) res[f].y += l1.y;
        }
      }
#pragma unroll
      for (int f = 0; f < K; ++f) {
        C* const o = lam0 + f * A.n + off;
        if constexpr (NAT) {
          o[0] = res[f].x;
          if (two) o[H] = res[f].y;
        } else {
          *reinterpret_cast<P*>(o) = res[f];
        }
      }
    }
  }

  if (grad_force) {
    // block sum of the force gradient: warp shuffles, then one value per warp
    __shared__ double red[3][32];
    const int lane = (threadIdx.y * blockDim.x + threadIdx.x) & 31;
    const int warp = (threadIdx.y * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (blockDim.x * blockDim.y + 31) >> 5;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double v = gf[i].value();
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
      if (lane == 0) red[i][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0)
      for (int i = 0; i < D; ++i) {
        double s = 0.0;
        for (int w = 0; w < nwarps; ++w) s += red[i][w];
        atomicAdd(grad_force + i, s);
      }
  }
}

// The viscosity term of adjoint.cu (its definition and sums) on natural FP32
// rows of D3Q19, given the state after the step (m' / rho' = u' - F there), with
// the same staging of the state alone.  Of a source (drho, u) with
// e = 3/2 rho u.u, r = rho c.u and h = 9/2 rho (c.u)^2, direction c carries
//   w (drho + e - h)         to sum c w rho (1 - 9/2 (c.u)^2 + 3/2 u.u) and
//   w (3 r + 2 (h - e))      to sum dF;
// h is shared by c and -c, so by the planes above and below.  97x96x95: 34.0 us,
// the per-node kernel of adjoint.cu (19 gathers of four values) 47.2; 127x80x80
// 24.6 and 43.1, 25^3 7.2 and 8.2.  Bound by latency, one block an SM.
template <int BXC, int RY>
__global__ void __launch_bounds__(BXC * RY, (AdjRows<kD3Q19, float, BXC, RY>::MIN_BLOCKS))
    adj_nu_rows(AdjArgs A, const float* __restrict__ state, const float* __restrict__ next,
                const float* __restrict__ lam, double* __restrict__ acc) {
  using T = AdjRows<kD3Q19, float, BXC, RY>;
  using O = Pair<float>;
  using P = float2;
  using U = AdjUnit<P>;
  extern __shared__ __align__(16) uint4 units[];
  pdl_wait();  // the previous kernel's writes are visible from here on
  pdl_launch_next();
  const int tx = threadIdx.x, r = threadIdx.y;
  const int H = (A.nx + 1) >> 1;
  const int row = blockIdx.y * A.ty + r - 1;
  const bool active = tx < H;
  const bool interior = active && r >= 1 && r <= RY - 2 && row < A.ny;
  const bool inside = row >= 0 && row < A.ny;
  const int row_mem = inside ? row : (row + A.ny) % A.ny;
  const bool stages_own = active && (inside || A.py);
  const int64_t row_off = (int64_t)row_mem * A.nx + tx;
  const bool two = tx + H < A.nx;  // lane y of the last pair of an odd row is the image of node 0
  const int hi = two ? H : -tx;
  const int z0 = (int)(((int64_t)blockIdx.x * A.nplanes) / A.nzc);
  const int z1 = (int)(((int64_t)(blockIdx.x + 1) * A.nplanes) / A.nzc);
  auto ld = [&](const float* p) { return make_float2(p[0], p[hi]); };

  struct Raw {
    P st[4];
  };
  auto load_raw = [&](int p, Raw& R) {
    const bool have = stages_own && ((p >= 0 && p < A.nplanes) || A.pz);
    const int pm = p < 0 ? p + A.nplanes : (p >= A.nplanes ? p - A.nplanes : p);
#pragma unroll
    for (int f = 0; f < 4; ++f)
      R.st[f] = have ? ld(state + f * A.n + (int64_t)pm * A.plane_stride + row_off) : make_float2(0.f, 0.f);
  };
  auto stage = [&](int p, const Raw& R) {
    if (!active) return;
    const int k = p & (T::STAGES - 1);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      U::st(&units[T::unit(k, r, u, tx)], &R.st[2 * u]);
      // the left neighbours (nx - 1, H - 1) of the first pair
      float* const seam = reinterpret_cast<float*>(&units[T::unit(k, r, u, T::SEAM_L)]);
      if (tx == A.nx - 1 - H) seam[0] = R.st[2 * u].y, seam[2] = R.st[2 * u + 1].y;
      if (tx == H - 1) seam[1] = R.st[2 * u].x, seam[3] = R.st[2 * u + 1].x;
      if (tx == 0) U::st_swapped(&units[T::unit(k, r, u, T::SEAM_R)], &R.st[2 * u]);
    }
  };
  const int col_l = tx == 0 ? T::SEAM_L : tx - 1;
  const int col_r = tx == H - 1 ? T::SEAM_R : tx + 1;
  // a source and what its directions share
  struct Src {
    P a, e, rho, u[3];
  };
  auto src = [&](int cx, int cy, int p) {  // the source of direction (cx, cy)
    P v[4];
#pragma unroll
    for (int u = 0; u < 2; ++u)
      U::ld(&units[T::unit(p & (T::STAGES - 1), r - cy, u, cx == 0 ? tx : cx == 1 ? col_l : col_r)], &v[2 * u]);
    Src s;
    s.rho = O::add(O::splat(1.f), v[0]);
    const P uu = O::fma(v[1], v[1], O::fma(v[2], v[2], O::mul(v[3], v[3])));
    s.e = O::mul(O::mul(uu, O::splat(1.5f)), s.rho);
    s.a = O::add(v[0], s.e);
#pragma unroll
    for (int i = 0; i < 3; ++i) s.u[i] = v[1 + i];
    return s;
  };
  // weights of one: g to the momentum sums, the return value to sum dF
  auto dir = [&](const Src& s, P t, P& g) {
    const P rt = O::mul(s.rho, t), h = O::mul(O::mul(t, O::splat(4.5f)), rt);
    g = adj_sub<float>(s.a, h);
    const P d = adj_sub<float>(h, s.e);
    return O::fma(rt, O::splat(3.f), O::add(d, d));
  };
  struct Sums {
    P d, m[3];
  };
  Sums pend{}, below{};  // of plane p - 1: without the plane above; what plane p - 1 sends up
  NuAcc<float> total;
  Raw R;
  load_raw(z0 - 1, R);
  stage(z0 - 1, R);
  load_raw(z0, R);
  for (int p = z0 - 1; p <= z1; ++p) {
    const int q = p - 1;  // the plane this one completes
    __syncthreads();      // plane p is staged, the reads of plane p - 1 are done
    if (p < z1) {
      stage(p + 1, R);
      if (p + 1 < z1) load_raw(p + 2, R);
    }
    if (!interior) continue;
    P nx4[4], lm[4];
    if (q >= z0) {
      const int64_t off = (int64_t)q * A.plane_stride + row_off;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        nx4[f] = ld(next + f * A.n + off);
        lm[f] = ld(lam + f * A.n + off);
      }
    }
    Sums own, up, dn;  // destinations in this plane, above (c_z = 1), below (c_z = -1)
    P g;
    {
      const Src s = src(0, 0, p);
      own.d = O::mul(s.e, O::splat(-24.f));
      own.m[0] = own.m[1] = own.m[2] = O::splat(0.f);
      const P d = dir(s, s.u[2], g), r3 = O::mul(O::mul(s.rho, s.u[2]), O::splat(6.f));
      up.d = O::add(d, d);
      dn.d = adj_sub<float>(adj_sub<float>(up.d, r3), r3);
      up.m[2] = O::add(g, g);
      dn.m[2] = O::mul(g, O::splat(-2.f));
      up.m[0] = up.m[1] = dn.m[0] = dn.m[1] = O::splat(0.f);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = k >> 1, sg = 1 - 2 * (k & 1);  // the axis and its sign
      const Src s = src(i == 0 ? sg : 0, i == 1 ? sg : 0, p);
      const P t = O::mul(s.u[i], O::splat(float(sg)));
      P d = dir(s, t, g);
      own.d = O::fma(d, O::splat(2.f), own.d);
      own.m[i] = O::fma(g, O::splat(2.f * sg), own.m[i]);
      d = dir(s, O::add(t, s.u[2]), g);
      up.d = O::add(up.d, d);
      up.m[i] = O::fma(g, O::splat(float(sg)), up.m[i]);
      up.m[2] = O::add(up.m[2], g);
      d = dir(s, adj_sub<float>(t, s.u[2]), g);
      dn.d = O::add(dn.d, d);
      dn.m[i] = O::fma(g, O::splat(float(sg)), dn.m[i]);
      dn.m[2] = adj_sub<float>(dn.m[2], g);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int cx = 1 - 2 * (k & 1), cy = 1 - (k & 2);
      const Src s = src(cx, cy, p);
      const P t = O::fma(s.u[0], O::splat(float(cx)), O::mul(s.u[1], O::splat(float(cy))));
      own.d = O::add(own.d, dir(s, t, g));
      own.m[0] = O::fma(g, O::splat(float(cx)), own.m[0]);
      own.m[1] = O::fma(g, O::splat(float(cy)), own.m[1]);
    }
    if (q >= z0) {
      const P inv = O::rcp(O::add(O::splat(1.f), nx4[0]));
      const P dR = O::add(pend.d, dn.d);  // x 36, as all below
      P t = adj_sub<float>(O::splat(0.f), O::mul(lm[0], dR));
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const P f = O::splat(float(A.force[i]));
        const P unf = adj_sub<float>(nx4[1 + i], f);  // m' / rho'
        const P md = O::add(pend.m[i], dn.m[i]);
        const P du = O::mul(O::fma(unf, dR, md), inv);
        t = O::fma(lm[1 + i], O::fma(f, O::splat(-36.f), du), t);
      }
      bool w0 = false, w1 = !two;
      if (A.wall_mode == kWallMask) {
        const uint8_t* const mk = A.mask + (int64_t)q * A.plane_stride + row_off;
        w0 = mk[0];
        w1 = w1 || mk[hi];
      } else if (A.wall_mode == kWallBox) {
        const bool all = (!A.pz && (q == 0 || q == A.nplanes - 1)) || (!A.py && (row == 0 || row == A.ny - 1));
        w0 = all || (!A.px && tx == 0);
        w1 = w1 || all || (!A.px && tx == A.nx - 1 - H);
      }
      if (!w0) total.add(t.x);
      if (!w1) total.add(t.y);
    }
    pend.d = O::add(own.d, below.d);
#pragma unroll
    for (int i = 0; i < 3; ++i) pend.m[i] = O::add(own.m[i], below.m[i]);
    below = up;
  }
  // block sum: warp shuffles, one value per warp, one FP64 atomic per block
  double v = total.value();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __shared__ double red[32];
  const int id = threadIdx.y * blockDim.x + threadIdx.x;
  if ((id & 31) == 0) red[id >> 5] = v;
  __syncthreads();
  if (id == 0) {
    for (int w = 1; w < (int)(blockDim.x * blockDim.y) >> 5; ++w) v += red[w];
    atomicAdd(acc, v / 36.0);
  }
}

// Launch helper of both kernels (instantiated in adjoint_tiled.cu): the arguments
// after A go to the kernel.  Returns the number of blocks of this shape one SM
// holds through *resident.
template <typename T, int BXC, int RY, typename Kern, typename... Args>
cudaError_t launch_rows(Kern kern, const AdjArgs& A, cudaStream_t st, int ytiles, int* resident, Args... args) {
  constexpr size_t smem = T::smem_bytes();
  static int resident_dev[64] = {};  // per instantiation and device
  int dev = 0;
  cudaError_t e0 = cudaGetDevice(&dev);
  if (e0 != cudaSuccess) return e0;
  if (resident && (*resident = resident_dev[dev & 63])) return cudaSuccess;
  if (resident) {  // sizing query only
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    int nb = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, T::THREADS, smem);
    if (e == cudaSuccess) *resident = resident_dev[dev & 63] = nb < 1 ? 1 : nb;
    return e;
  }
  const int unit = RY % 4 == 0 ? 8 : RY % 2 == 0 ? 16 : 32;  // whole warps a block
  const int width = ((A.nx + 1) / 2 + unit - 1) / unit * unit;
  return launch_kernel(kern, dim3(A.nzc, ytiles), dim3(width, RY), smem, st, A.overlap, A, args...);
}

template <int LAT, typename S, int BXC, int RY>
cudaError_t launch_adj_rows(const AdjArgs& A, const void* in_state, const void* out_state, const void* lam1, void* lam0,
                            double* grad_force, cudaStream_t st, int ytiles, int* resident) {
  using T = AdjRows<LAT, S, BXC, RY>;
  using C = typename T::C;
  return launch_rows<T, BXC, RY>(adj_step_rows<LAT, S, BXC, RY>, A, st, ytiles, resident,
                                 static_cast<const S*>(in_state), static_cast<const S*>(out_state),
                                 static_cast<const C*>(lam1), static_cast<C*>(lam0), grad_force);
}

template <int BXC, int RY>
cudaError_t launch_nu_rows(const AdjArgs& A, const void* state, const void* next, const void* lam, double* acc,
                           cudaStream_t st, int ytiles, int* resident) {
  return launch_rows<AdjRows<kD3Q19, float, BXC, RY>, BXC, RY>(
      adj_nu_rows<BXC, RY>, A, st, ytiles, resident, static_cast<const float*>(state), static_cast<const float*>(next),
      static_cast<const float*>(lam), acc);
}

}  // namespace maclab
