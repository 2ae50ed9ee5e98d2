// step_block.cu -- block-resident temporal blocking of the D2Q9 step
// (Eqs. (2), (4), (5)): one launch advances the state K steps.
//
// Pair j of row y holds the nodes x = j and x = j + H.  Interleaved storage
// (whole quads, see common.cuh; H = nx / 2) keeps the two next to each other;
// in natural rows (NAT: a periodic x axis of any width, H = ceil(nx / 2)) they
// are read and written one by one, x taken modulo nx.  In these pair
// coordinates every stencil neighbour of pair j is pair j - 1, j or j + 1 of a
// neighbouring row, so a tile is a plain rectangle of pairs whatever its
// position: beyond the row's end pair j + H is pair j with its two nodes swapped
// (interleaved), or simply the next nodes (natural).
//
//  * A block loads a tile of pairs into registers: an output tile with a halo of
//    K pairs and K rows on every side (wrapped where the axis is periodic; zero
//    rows beyond a closed y boundary).  FP32: step_block2_d2q9, 32 x 32 pairs,
//    two columns by one or two rows per thread.  FP64: step_block_d2q9, 32 pairs by a number of rows
//    chosen for the grid, one pair per thread.
//  * Each step a thread forms what its pairs send along the row (d2q9.cuh), gets
//    the neighbouring columns' values from registers or by warp shuffle, sums
//    its rows and passes on to the rows above and below the two values each that
//    cross: in registers between a thread's own rows, through shared memory
//    between thread-rows.  After one barrier it adds the three rows, divides and
//    adds the force.  Wall nodes keep their values; beyond a closed boundary
//    only wall nodes are reached.  The valid region shrinks by one pair and one
//    row per step.
//  * The sums run in the order of d2q9.cuh, as in the tiled and segment kernels,
//    so every step gives the same bits as one step of those.
//  * The exchange buffers alternate between steps, so one barrier per step
//    suffices: a thread writes buffer s & 1 only after every thread has
//    passed the barrier of step s - 1, i.e. finished its reads of step s - 2.
//  * After K steps the output tile is stored (wall nodes are never written;
//    their values are in both buffers).  Global memory is touched once per K
//    steps: the tile's state once in and once out.

#include "d2q9.cuh"

namespace maclab {
namespace {

constexpr int kBlockBX = 32;  // pairs per tile row

struct BlockArgs {
  const void* in;
  void* out;
  const uint8_t* mask;  // node types in storage order (kWallMask)
  int64_t n;            // nodes (field stride)
  int nx, ny, hx;       // hx: pairs of a row
  int x_last;           // the domain's last node of a row (nx - 1 less the padding)
  int px, py;           // periodic flags
  int wall_mode;
  double force[2];      // lattice-unit force increment
};

template <typename S>
struct PairIO;
template <>
struct PairIO<float> {
  __device__ __forceinline__ static float2 ld(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
  __device__ __forceinline__ static void st(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
};
template <>
struct PairIO<double> {
  __device__ __forceinline__ static double2 ld(const double* p) {
    return __ldg(reinterpret_cast<const double2*>(p));
  }
  __device__ __forceinline__ static void st(double* p, double2 v) { *reinterpret_cast<double2*>(p) = v; }
};

// One pair of a tile: where it lies and which of its nodes are kept.
struct BlockPair {
  int64_t off;      // its row's storage offset plus, interleaved, that of the pair
  int x0, x1;       // natural rows: its nodes' positions
  bool row_ok;      // the row exists
  bool swapped;     // interleaved: the pair's nodes are stored in the other order
  uint32_t keep;    // bit 0 / 1: lane x / y holds a wall node or a node beyond a closed boundary
};

template <bool NAT>
__device__ __forceinline__ BlockPair block_pair(const BlockArgs& a, int jj, int yy) {
  BlockPair b;
  b.row_ok = true;
  int ym = yy;
  if (yy < 0 || yy >= a.ny) {
    if (a.py) ym = ((yy % a.ny) + a.ny) % a.ny;
    else b.row_ok = false;
  }
  const int64_t row = (int64_t)(b.row_ok ? ym : 0) * a.nx;
  if constexpr (NAT) {  // x periodic
    b.x0 = jj % a.nx;
    if (b.x0 < 0) b.x0 += a.nx;
    b.x1 = b.x0 + a.hx;
    if (b.x1 >= a.nx) b.x1 -= a.nx;
    b.swapped = false;
    b.off = row;
  } else {
    int wraps = jj / a.hx;
    if (jj % a.hx < 0) --wraps;
    const int p = jj - wraps * a.hx;     // stored pair, 0 <= p < H
    b.swapped = (wraps & 1) != 0;        // its nodes in the other order
    b.x0 = b.swapped ? p + a.hx : p;
    b.x1 = b.swapped ? p : p + a.hx;
    b.off = row + 2 * p;
  }
  b.keep = 3u;
  if (b.row_ok) {
    if (a.wall_mode == kWallMask) {
      uint32_t m0, m1;
      if constexpr (NAT) {
        m0 = a.mask[b.off + b.x0] != 0 ? 1u : 0u;
        m1 = a.mask[b.off + b.x1] != 0 ? 1u : 0u;
      } else {
        const uchar2 m = *reinterpret_cast<const uchar2*>(a.mask + b.off);
        m0 = (b.swapped ? m.y : m.x) != 0 ? 1u : 0u;
        m1 = (b.swapped ? m.x : m.y) != 0 ? 1u : 0u;
      }
      b.keep = m0 | (m1 << 1);
    } else if (a.wall_mode == kWallBox) {
      const bool yw = !a.py && (ym == 0 || ym == a.ny - 1);
      const bool w0 = yw || (!a.px && (b.x0 == 0 || b.x0 >= a.x_last));
      const bool w1 = yw || (!a.px && (b.x1 == 0 || b.x1 >= a.x_last));
      b.keep = (w0 ? 1u : 0u) | (w1 ? 2u : 0u);
    } else {
      b.keep = 0u;
    }
  }
  return b;
}

template <typename S, bool NAT>
__device__ __forceinline__ void block_load(const BlockArgs& a, const BlockPair& b,
                                           typename Pair<typename Store<S>::C>::P (&st)[3]) {
  using O = Pair<typename Store<S>::C>;
  const S* in = static_cast<const S*>(a.in) + b.off;
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!b.row_ok) {
      st[f] = O::splat(0);
    } else if constexpr (NAT) {
      st[f] = O::make(__ldg(in + f * a.n + b.x0), __ldg(in + f * a.n + b.x1));
    } else {
      st[f] = PairIO<S>::ld(in + f * a.n);
      if (b.swapped) st[f] = O::swap(st[f]);
    }
  }
}

// Store of a pair of the output tile: 0 <= jj < H, a row of the grid.  In natural
// rows of odd width the last pair's second node is the row's first (stored as pair 0's).
template <typename S, bool NAT>
__device__ __forceinline__ void block_store(const BlockArgs& a, const BlockPair& b, int jj,
                                            const typename Pair<typename Store<S>::C>::P (&st)[3]) {
  S* out = static_cast<S*>(a.out) + b.off;
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    S* q = out + f * a.n;
    if constexpr (NAT) {
      if (!(b.keep & 1u)) q[b.x0] = st[f].x;
      if (!(b.keep & 2u) && jj + a.hx < a.nx) q[b.x1] = st[f].y;
    } else {  // never swapped here
      if (b.keep == 0u) PairIO<S>::st(q, st[f]);
      else if (b.keep == 2u) q[0] = st[f].x;
      else if (b.keep == 1u) q[1] = st[f].y;
    }
  }
}

// v of lane src (of the whole warp)
template <typename P>
__device__ __forceinline__ P shfl_pair(P v, int src) {
  P r;
  r.x = __shfl_sync(0xffffffffu, v.x, src);
  r.y = __shfl_sync(0xffffffffu, v.y, src);
  return r;
}

template <typename C>
__device__ __forceinline__ void block_next_state(const typename Pair<C>::P (&s)[3],
                                                 const typename Pair<C>::P (&force)[2], uint32_t keep,
                                                 typename Pair<C>::P (&st)[3]) {
  typename Pair<C>::P nv[3];
  d9_state<C>(s, force, nv);
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!(keep & 1u)) st[f].x = nv[f].x;
    if (!(keep & 2u)) st[f].y = nv[f].y;
  }
}

// ------------------------------------------------------------------ FP64: one pair per thread
//
// A warp is one tile row of 32 pairs; blockDim.y rows (block_rows_f64).  GB300's
// FP64 pipe (two lanes per SM) bounds it: 41 operations a node and step and a
// division (the correctly rounded one: 256^2 9.94 us a step, 9.89 with a
// reciprocal good to an ulp, 64^2 4.23 and 4.05), plus those of the halo, which is
// why the rows of a tile are chosen for the grid.
// WRAP: rows of at most 32 pairs (interleaved), which a tile holds whole: the
// neighbour across the row's end is the lane at its other end, swapped, and the
// tile needs no halo columns.
constexpr int kBlockRowsF64 = 20;  // most rows of a tile

template <typename S, int K, bool NAT, bool WRAP>
__global__ void __launch_bounds__(kBlockBX * kBlockRowsF64, 1) step_block_d2q9(BlockArgs a) {
  using C = typename Store<S>::C;
  using O = Pair<C>;
  using P = typename O::P;
  constexpr int KX = WRAP ? 0 : K;  // halo columns
  constexpr int TX = kBlockBX - 2 * KX;
  extern __shared__ __align__(16) unsigned char block_smem[];
  const int ix = threadIdx.x, iy = threadIdx.y, by = blockDim.y;
  const int plane = (by + 2) * kBlockBX;
  P* const xb = reinterpret_cast<P*>(block_smem);  // [2 buffers][gp, hp, gm, hm][rows -1 .. by][32]
  const int me = (iy + 1) * kBlockBX + ix;
  const int jj = WRAP ? min(ix, a.hx - 1) : (int)blockIdx.x * TX - KX + ix;  // pair column, possibly outside [0, H)
  const int yy = (int)blockIdx.y * (by - 2 * K) - K + iy;
  const int src_l = WRAP && ix == 0 ? a.hx - 1 : (ix - 1) & 31;
  const int src_r = WRAP && ix == a.hx - 1 ? 0 : (ix + 1) & 31;

  const BlockPair b = block_pair<NAT>(a, jj, yy);
  P st[3];
  pdl_wait();  // the previous step's writes are visible from here on
  block_load<S, NAT>(a, b, st);
  pdl_launch_next();
  const P force[2] = {O::splat(C(a.force[0])), O::splat(C(a.force[1]))};

  auto left = [&](P v) {
    v = shfl_pair(v, src_l);
    return WRAP && ix == 0 ? O::swap(v) : v;
  };
  auto right = [&](P v) {
    v = shfl_pair(v, src_r);
    return WRAP && ix == a.hx - 1 ? O::swap(v) : v;
  };
#pragma unroll 1
  for (int s = 1; s <= K; ++s) {
    P* const vb = xb + (s & 1) * 4 * plane;
    D9Row<C> w;
    // sources: the rows the region of step s reads (s - 1 .. by - s)
    if (iy >= s - 1 && iy <= by - s) {
      const D9Node<C> n = d9_node<C>(st[0], st[1], st[2]);
      w = d9_row<C>(n.A, n.by, n.e, left(n.ap), left(n.bp), left(n.e), right(n.am), right(n.bm), right(n.e));
      vb[me] = w.gp;
      vb[plane + me] = w.hp;
      vb[2 * plane + me] = w.gm;
      vb[3 * plane + me] = w.hm;
    }
    __syncthreads();
    if (iy >= s && iy < by - s) {
      P sum[3];
      d9_own<C>(sum, vb[me - kBlockBX], vb[plane + me - kBlockBX], w);
      d9_above<C>(sum, vb[2 * plane + me + kBlockBX], vb[3 * plane + me + kBlockBX]);
      block_next_state<C>(sum, force, b.keep, st);
    }
  }
  const bool col_out = WRAP ? ix < a.hx : ix >= KX && ix < kBlockBX - KX && jj < a.hx;
  if (col_out && iy >= K && iy < by - K && yy >= 0 && yy < a.ny && b.keep != 3u) block_store<S, NAT>(a, b, jj, st);
}

// ------------------------------------------------------------------ FP32: 2 x R pairs per thread
//
// 512 / R threads hold the tile of 32 x 32 pairs: a thread owns the 2 x R pairs
// (columns 2 tx, 2 tx + 1; rows R ty .. R ty + R - 1), lane tx + 16 (ty & 1) of
// warp ty / 2.  Of what a pair sends, the values for the thread's other column
// stay in registers and those for the next thread's column move by warp shuffle
// (three each way and row); what the thread's rows send each other stays in
// registers, and only the two values leaving its rows upwards and the two
// leaving them downwards go through shared memory, both columns in one 16-byte
// unit.
//
// The kernel waits on its chains of dependent paired-FP32 operations and on the
// barriers, so what serves a grid best is set by how many tiles an SM gets
// (block2_shape; us per step, R x blocks an SM is compiled for):
//              1 x 1    2 x 2    2 x 3
//   256^2      0.84     0.97     1.10     at most one tile an SM: its 16 warps
//   512^2      1.81     1.76     2.21     two: fewer, longer chains, no spills
//   1024^2     5.07     5.21     4.66     more: 24 warps, though a few values spill
//   2047^2     24.6     17.8     15.7     (periodic, natural rows)
// (The nine-term form with R = 2: 1.03 at 256^2, 1.99 at 512^2, 5.71 at 1024^2.)

template <typename P>
__device__ __forceinline__ P b2_from_left(P v) {
  P r;
  r.x = __shfl_up_sync(0xffffffffu, v.x, 1);
  r.y = __shfl_up_sync(0xffffffffu, v.y, 1);
  return r;
}
template <typename P>
__device__ __forceinline__ P b2_from_right(P v) {
  P r;
  r.x = __shfl_down_sync(0xffffffffu, v.x, 1);
  r.y = __shfl_down_sync(0xffffffffu, v.y, 1);
  return r;
}

template <typename S, int K, bool NAT, int R, int PER_SM>
__global__ void __launch_bounds__(512 / R, PER_SM) step_block2_d2q9(BlockArgs a) {
  using C = typename Store<S>::C;
  using O = Pair<C>;
  using P = typename O::P;
  constexpr int TW = kBlockBX, TX = TW - 2 * K;  // tile and output width (and height) in pairs
  constexpr int UNITS = (TW / R + 2) * 16;  // units (two columns' pairs) of a plane: thread-rows -1 .. 32 / R
  extern __shared__ __align__(16) unsigned char block_smem[];
  typedef float4 Planes[4][UNITS];  // gp, hp, gm, hm
  Planes* const xb = reinterpret_cast<Planes*>(block_smem);  // two buffers
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = lane & 15, ty = 2 * warp + (lane >> 4);
  const int j0 = blockIdx.x * TX - K, y0 = blockIdx.y * TX - K;

  P st[R][2][3];
  uint32_t keep[R][2];
  pdl_wait();  // the previous step's writes are visible from here on
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const BlockPair b = block_pair<NAT>(a, j0 + 2 * tx + c, y0 + R * ty + r);
      block_load<S, NAT>(a, b, st[r][c]);
      keep[r][c] = b.keep;
    }
  pdl_launch_next();

  const P force[2] = {O::splat(C(a.force[0])), O::splat(C(a.force[1]))};
  const int me = (ty + 1) * 16 + tx;

#pragma unroll 1
  for (int s = 1; s <= K; ++s) {
    Planes& xs = xb[s & 1];
    // the warp's pair rows 2 R warp .. 2 R warp + 2 R - 1 against the rows step s reads (s - 1 .. TW - s)
    const bool active = 2 * R * warp + 2 * R - 1 >= s - 1 && 2 * R * warp <= TW - s;
    D9Row<C> w[R][2];  // [row][column]
    if (active) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        // lanes 0 / 15 and 16 / 31 receive values for the tile's edge columns,
        // which no step's region contains
        const D9Node<C> m = d9_node<C>(st[r][0][0], st[r][0][1], st[r][0][2]);
        const D9Node<C> n = d9_node<C>(st[r][1][0], st[r][1][1], st[r][1][2]);
        w[r][0] = d9_row<C>(m.A, m.by, m.e, b2_from_left(n.ap), b2_from_left(n.bp), b2_from_left(n.e), n.am, n.bm,
                            n.e);
        w[r][1] = d9_row<C>(n.A, n.by, n.e, m.ap, m.bp, m.e, b2_from_right(m.am), b2_from_right(m.bm),
                            b2_from_right(m.e));
      }
      auto unit = [](P p, P q) { return make_float4(p.x, p.y, q.x, q.y); };
      xs[0][me] = unit(w[R - 1][0].gp, w[R - 1][1].gp);
      xs[1][me] = unit(w[R - 1][0].hp, w[R - 1][1].hp);
      xs[2][me] = unit(w[0][0].gm, w[0][1].gm);
      xs[3][me] = unit(w[0][0].hm, w[0][1].hm);
    }
    __syncthreads();
    if (active) {
      // every pair is updated; those outside the step's region hold values
      // that no later step of the valid region reads
      const float4 gp = xs[0][me - 16], hp = xs[1][me - 16], gm = xs[2][me + 16], hm = xs[3][me + 16];
      auto half = [](const float4& v, int c) { return c ? O::make(v.z, v.w) : O::make(v.x, v.y); };
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          P sum[3];
          if (r == 0) d9_own<C>(sum, half(gp, c), half(hp, c), w[0][c]);
          else d9_own<C>(sum, w[r - 1][c].gp, w[r - 1][c].hp, w[r][c]);
          if (r == R - 1) d9_above<C>(sum, half(gm, c), half(hm, c));
          else d9_above<C>(sum, w[r + 1][c].gm, w[r + 1][c].hm);
          block_next_state<C>(sum, force, keep[r][c], st[r][c]);
        }
    }
  }

#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int ix = 2 * tx + c, iy = R * ty + r, jj = j0 + ix, yy = y0 + iy;
      if (ix < K || ix >= TW - K || iy < K || iy >= TW - K || jj >= a.hx || yy >= a.ny || keep[r][c] == 3u) continue;
      BlockPair b;  // an output pair: inside the grid, not swapped
      b.off = (int64_t)yy * a.nx + (NAT ? 0 : 2 * jj);
      b.x0 = jj;
      b.x1 = jj + a.hx < a.nx ? jj + a.hx : jj + a.hx - a.nx;
      b.keep = keep[r][c];
      block_store<S, NAT>(a, b, jj, st[r][c]);
    }
}

BlockArgs block_args(const StepLaunch& s, bool natural) {
  BlockArgs a;
  a.in = s.in;
  a.out = s.out;
  a.mask = s.g.mask;
  a.n = s.g.n;
  a.nx = s.g.nx;
  a.ny = s.g.ny;
  a.hx = natural ? (s.g.nx + 1) / 2 : s.g.nx / 2;
  a.x_last = s.g.nx - 1 - s.g.pad;
  a.px = (s.g.periodic & 1u) ? 1 : 0;
  a.py = (s.g.periodic & 2u) ? 1 : 0;
  a.wall_mode = s.g.wall_mode;
  a.force[0] = s.force[0];
  a.force[1] = s.force[1];
  return a;
}

int block_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 148;
  }
  return sms;
}

// Output rows of a tile of the FP64 kernel: those whose busiest SM has the least
// to do, in units of one operation of a warp's row of pairs.  A step forms and
// sums its source rows (29 operations) and finishes its destination rows (16, the
// division counted as three); the blocks of a launch share the SMs' FP64 pipes
// evenly.  (256^2 at 2 steps a launch: 128 blocks of 32 x 16 pairs before, 16.4 us a
// step.)
int block_rows_f64(int ny, int xtiles, int steps) {
  int best = 1;
  int64_t least = INT64_MAX;
  for (int rows = 1; rows + 2 * steps <= kBlockRowsF64; ++rows) {
    if ((ny + rows - 1) / rows > 65535) continue;  // the grid's limit
    const int by = rows + 2 * steps;
    int64_t cost = 0;
    for (int s = 1; s <= steps; ++s) cost += 29 * (by - 2 * (s - 1)) + 16 * (by - 2 * s);
    const int64_t blocks = (int64_t)xtiles * ((ny + rows - 1) / rows);
    cost *= (blocks + block_sms() - 1) / block_sms();
    if (cost < least) {
      least = cost;
      best = rows;
    }
  }
  return best;
}

template <int K, bool NAT, bool WRAP>
cudaError_t launch_block_f64(const StepLaunch& s, cudaStream_t stream) {
  constexpr int TX = kBlockBX - (WRAP ? 0 : 2 * K);
  const BlockArgs a = block_args(s, NAT);
  const int xtiles = (a.hx + TX - 1) / TX;
  const int rows = block_rows_f64(a.ny, xtiles, K), by = rows + 2 * K;
  constexpr size_t row_bytes = 2 * 4 * (size_t)kBlockBX * sizeof(double2);
  auto kern = step_block_d2q9<double, K, NAT, WRAP>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)((kBlockRowsF64 + 2) * row_bytes));
  // the same split of L1 and shared memory for every instance and tile height: an SM
  // changes it only when idle, so a run whose launches take 2, 2, 2, 1 steps waited for
  // the device to drain at every change (128^2, runs of 3 steps: 12.5 us a step, 6.4 now)
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3((unsigned)xtiles, (unsigned)((a.ny + rows - 1) / rows)), dim3(kBlockBX, by),
                       (by + 2) * row_bytes, stream, s.overlap, a);
}

template <int K>
cudaError_t launch_block_f64_any(const StepLaunch& s, cudaStream_t stream) {
  if (!s.g.ilv) return launch_block_f64<K, true, false>(s, stream);
  if (s.g.nx / 2 <= kBlockBX) return launch_block_f64<K, false, true>(s, stream);
  return launch_block_f64<K, false, false>(s, stream);
}

// Tiles of a step of the FP32 kernel, columns by rows.
dim3 block2_grid(int hx, int ny, int steps) {
  const int tx = kBlockBX - 2 * steps;
  return dim3((unsigned)((hx + tx - 1) / tx), (unsigned)((ny + tx - 1) / tx));
}

// Blocks per SM the instance for this many tiles is compiled for: 1 (with one row
// per thread), 2 or 3 (two rows); see the kernel.
int block2_shape(const dim3& grid) {
  const int64_t tiles = (int64_t)grid.x * grid.y;
  return tiles <= block_sms() ? 1 : tiles <= 2 * block_sms() ? 2 : 3;
}

template <int K, bool NAT, int R, int PER_SM>
cudaError_t launch_block2_r(const BlockArgs& a, const dim3& grid, int overlap, cudaStream_t stream) {
  constexpr size_t smem = 2 * 4 * (kBlockBX / R + 2) * 16 * sizeof(float4);
  auto kern = step_block2_d2q9<float, K, NAT, R, PER_SM>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, grid, dim3(512 / R), smem, stream, overlap, a);
}

template <int K, bool NAT>
cudaError_t launch_block2_t(const StepLaunch& s, cudaStream_t stream) {
  const BlockArgs a = block_args(s, NAT);
  const dim3 grid = block2_grid(a.hx, a.ny, K);
  switch (block2_shape(grid)) {
    case 1: return launch_block2_r<K, NAT, 1, 1>(a, grid, s.overlap, stream);
    case 2: return launch_block2_r<K, NAT, 2, 2>(a, grid, s.overlap, stream);
    default: return launch_block2_r<K, NAT, 2, 3>(a, grid, s.overlap, stream);
  }
}

template <int K>
cudaError_t launch_block2_any(const StepLaunch& s, cudaStream_t stream) {
  return s.g.ilv ? launch_block2_t<K, false>(s, stream) : launch_block2_t<K, true>(s, stream);
}

}  // namespace

// Steps per launch for the tile setting ty; default (ty = 0): FP32 8 up to 65,536
// pairs, 4 above (256^2 0.84, 512^2 1.76 us a step, the other way 0.98 and 2.41);
// FP64, whose halo costs more than the launch it saves, 1 below 8,192 pairs (64^2:
// 4.23 us a step, 4.29 at two, 5.17 at four).  Above that 4 up to 16,384 pairs, then
// 2: the counts that launches of this kernel have had from the start and that its
// tests hold, not the fastest (128^2: 6.57 at four, 5.26 at one; 256^2: 9.94 at two,
// 9.72 at one).
int block_steps(const Geometry& g, int precision, int ty) {
  if (precision != MACLAB_F32 && precision != MACLAB_F64) return 0;
  const int64_t pairs = (int64_t)(g.nx / 2) * g.ny;
  if (ty == 0) return precision == MACLAB_F32 ? (pairs <= 65536 ? 8 : 4)
                                                  : (pairs < 8192 ? 1 : pairs <= 16384 ? 4 : 2);
  if (ty == 1 || ty == 2 || ty == 4) return ty;
  if (ty == 8 && precision == MACLAB_F32) return 8;
  return 0;
}

// natural: also rows of a periodic x axis whose width is not a multiple of 4 (at
// least half a tile wide: narrower ones leave most lanes idle and stay with the
// reference kernel).
bool block_supported(const Geometry& g, int precision, int ty, bool natural) {
  const int k = block_steps(g, precision, ty);
  if (g.lattice != kD2Q9 || k == 0) return false;
  if (!g.ilv && !(natural && (g.periodic & 1u) && g.nx >= kBlockBX)) return false;
  const int rows = (precision == MACLAB_F32 ? kBlockBX : kBlockRowsF64) - 2 * k;
  return (g.ny + rows - 1) / rows <= 65535;
}

int block_threads(const Geometry& g, int precision, int steps) {
  const int hx = g.ilv ? g.nx / 2 : (g.nx + 1) / 2;
  if (precision != MACLAB_F64) return block2_shape(block2_grid(hx, g.ny, steps)) == 1 ? 512 : 256;
  const bool wrap = g.ilv && g.nx / 2 <= kBlockBX;
  const int tx = kBlockBX - (wrap ? 0 : 2 * steps);
  return kBlockBX * (block_rows_f64(g.ny, (hx + tx - 1) / tx, steps) + 2 * steps);
}

// One launch of `steps` steps (1, 2, 4, or 8 with FP32 storage) from s.in to s.out.
cudaError_t launch_block(const StepLaunch& s, cudaStream_t stream, int steps) {
  if (!block_supported(s.g, s.precision, steps, true)) return cudaErrorInvalidValue;
  if (s.precision == MACLAB_F32) {
    switch (steps) {
      case 1: return launch_block2_any<1>(s, stream);
      case 2: return launch_block2_any<2>(s, stream);
      case 4: return launch_block2_any<4>(s, stream);
      case 8: return launch_block2_any<8>(s, stream);
    }
  } else {
    switch (steps) {
      case 1: return launch_block_f64_any<1>(s, stream);
      case 2: return launch_block_f64_any<2>(s, stream);
      case 4: return launch_block_f64_any<4>(s, stream);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace maclab
