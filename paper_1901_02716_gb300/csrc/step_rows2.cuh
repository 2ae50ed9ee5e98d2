// step_rows2.cuh -- D3Q19 MacLAB step with two rows per thread (Eqs. (2),
// (4), (5); the same update as step_naive, summed in another order).
//
// Layout and march as in step_tiled.cuh: storage rows interleaved in halves
// (a thread's 16-byte quad is the node pairs a = (2t, 2t + H), b = (2t + 1,
// 2t + 1 + H)), a block marches z over a chunk of planes keeping the sums of
// the destination planes p - 1, p, p + 1 in registers.  What differs:
//
//  * Each thread owns the quads of two adjacent rows (r0 = 2 tr, r1 = r0 + 1)
//    of a tile of TY = 2 TYT rows, and the update is factored by rows and planes
//    (d3q19.cuh): what a node sends along x moves to the neighbouring lanes by
//    shuffles (five values each way and row), what the thread's rows send each
//    other stays in registers, and only the four values leaving the row pair
//    upwards and the four leaving it downwards go through shared memory, one
//    16-byte unit per column and value, at the sender's own column.
//  * Between planes a thread keeps four sums of the plane about to be completed
//    and three of what the last plane sent on.
//  * The halo rows next to the tile are loaded by the first and last
//    thread-rows, which publish what they send into the tile in the units a
//    neighbouring thread-row would have filled: every thread then gathers the
//    same way, with no branch on its position.
//  * Measured at 128^3 (FP32 cavity): 14.3 us a step, 7.1 M warp instructions,
//    213 registers, where forming the nineteen terms took 15.2 us, 7.8 M and 253.
//    With the whole update replaced by a copy of the staged quads it takes 7.8
//    us: neither memory nor issue (42 %) bounds it but the plane's chain of
//    dependent operations, at two 128-thread blocks per SM; a lone block takes
//    1.0 us a plane, two together 1.45.  A fifth warp for the halo rows leaves
//    168 registers per thread (three warps on one scheduler) and spills: 19.5 us.
//  * Box x-walls: the lanes holding x = 0 or x = nx - 1 store the wall node's
//    unchanged values in place of the computed ones, with selects, so every
//    lane stores whole quads.  The values come from the staged plane: when a
//    plane is taken from its stage slot, these lanes copy their wall node's
//    four values of both rows into a small per-thread shared-memory slot
//    (two, by plane parity), which the store of that plane reads a plane
//    later.  (A global load at the store exposed its latency, and registers
//    held across a plane's update do not fit.)
//
// Requires: D3Q19, FP32 arithmetic (FP32, BF16 or FP16 storage), nx % 4 == 0,
// nx / 4 <= BXC, ny >= TY, TYT >= 2.  Where TY does not divide ny, the last tile
// is moved up to end at the last row; the rows it shares with the tile before
// are stored by that one only.
//
// Viscosity-term mode (NU, FP32 storage): the same march and exchanges gather
// the moments of g_a = w_a (drho + rho (3/2 u.u - 9/2 (c.u)^2)) (the
// equilibrium less its derivative along u and its constant: Eq. (2) with no
// linear part and the quadratic part negated) instead of Eq. (2) itself, and
// the store becomes a sum: with R and u' of the stored state after the step,
// drho' along u is dR = R - G0, and each fluid node adds
//   lam_rho (-dR / 36) + sum_i lam_u_i (Md_i / (36 + R) + (u'_i - F_i) dR / (36 + R) - F_i),
// Md = the first moments of g, into the accumulator (the term of
// maclab_adjoint_nu_term, per node as in adj_nu_term).

#pragma once
#include "d3q19.cuh"
#include "step_fold.cuh"

namespace maclab {

// ------------------------------------------------------------------ layout

template <typename S, int BXC, int TYT>
struct Rows2Layout {
  static constexpr int TY = 2 * TYT;
  static constexpr int RS = TY + 2;       // staged rows: lower halo, TY own, upper halo
  static constexpr int NSLOT = TYT + 1;   // receiving rows per sign (see step_rows2)
  static constexpr int VAL_UNITS = NSLOT * BXC;
  static constexpr int SIGN_UNITS = 4 * VAL_UNITS;  // G, H, T of c_z = +1 and -1
  static constexpr int BUF_UNITS = 2 * SIGN_UNITS;
  static constexpr size_t y_bytes = (size_t)2 * BUF_UNITS * 16;  // two buffers of 16-byte units
  // a stage slot: the TY own rows [4 fields][TY][row], then the halo rows
  // below and above, [4 fields][row] each, as the tile copies lay them out
  // (BXC quads a row); offsets are multiples of 128 bytes
  static constexpr size_t QB = (size_t)BXC * Quad<S>::BYTES;  // the widest row
  static constexpr size_t slot_bytes = 4 * RS * QB;
  static constexpr size_t halo_lo = 4 * TY * QB;
  static constexpr size_t halo_hi = halo_lo + 4 * QB;
  static constexpr size_t stage_bytes = (size_t)kStages * slot_bytes;
  static constexpr size_t mbar_off = stage_bytes;        // one mbarrier per slot
  static constexpr size_t y_off = stage_bytes + 16;
  // box x-wall values of the two planes in flight, [plane parity][TYT][side]
  // [2 rows x 4 fields] floats, each slot written and read by its own thread
  static constexpr size_t wall_off = y_off + y_bytes;
  static constexpr size_t wall_bytes = (size_t)2 * TYT * 2 * 8 * sizeof(float);
  // + 128: the base is rounded up to a 128-byte boundary at run time
  static constexpr size_t smem = 128 + wall_off + wall_bytes;
  static constexpr int THREADS = BXC * TYT;
  // at least eight warps per SM where shared memory allows
  static constexpr int SMEM_BLOCKS = (int)((220 * 1024) / smem) < 1 ? 1 : (int)((220 * 1024) / smem);
  static constexpr int WANT = 256 / THREADS < 1 ? 1 : 256 / THREADS;
  static constexpr int MIN_BLOCKS = WANT < SMEM_BLOCKS ? WANT : SMEM_BLOCKS;
};

// ------------------------------------------------------------------ kernel

// Running float-float sum of one thread (viscosity-term mode): Knuth's two-sum
// keeps the rounding error of every FP32 addition.
struct Rows2Sum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
    hi = s;
  }
};

// Whether value k (G, H, T of c_z = +1, T of c_z = -1) crosses rows in this mode.
template <int MODE>
__host__ __device__ constexpr bool rows2_sends(int k) {
  return k < 2 ? MODE == kMid : k == 2 ? MODE != kLast : MODE != kFirst;
}

// NU: viscosity-term mode (see the top of this file); `out` is then the state
// after the step, read only.
// Tile copies: tm_own maps the state as [4 fields][nz][ny][nx] with a box of the
// tile's TY own rows of every field; tm_halo the same tensor with a box of one
// row of every field.
// RM: the rows it serves (RowMode).
template <typename S, int BXC, int TYT, bool NU = false, int RM = kRowsPlain>
__global__ void __launch_bounds__(BXC * TYT, Rows2Layout<S, BXC, TYT>::MIN_BLOCKS)
    step_rows2(TiledArgs ta, const S* __restrict__ in, S* __restrict__ out,
               const __grid_constant__ CUtensorMap tm_own, const __grid_constant__ CUtensorMap tm_halo) {
  using Lay = Rows2Layout<S, BXC, TYT>;
  using C = float;
  using O = Pair<C>;
  using P = typename O::P;
  constexpr int TY = Lay::TY;
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  // stage slots at a 128-byte boundary (tile copies land on it), then the
  // mbarriers, then the y exchange
  unsigned char* const smem_raw = smem_dyn + ((128u - (smem_u32(smem_dyn) & 127u)) & 127u);
  const int tx = threadIdx.x, tr = threadIdx.y;
  // issues the tile copies: a thread of a middle thread-row, which forms no
  // halo row, where there is one
  const bool leader = tx == 0 && tr == (TYT > 2 ? 1 : 0);
  const uint32_t mbar0 = smem_u32(smem_raw + Lay::mbar_off);
  if (leader) {
    mbar_init(mbar0, 1);
    mbar_init(mbar0 + 8, 1);
    mbar_init_fence();
  }
  __syncthreads();
  pdl_wait();  // the previous step's writes are visible from here on
  pdl_launch_next();

  const int bxr = ta.nx >> 2;  // threads per row actually used
  const bool active = tx < bxr;
  float4* const Y = reinterpret_cast<float4*>(smem_raw + Lay::y_off);

  const bool seam_r = tx == bxr - 1;  // right neighbour across the seam: its lanes swapped
  const bool seam_l = tx == 0;        // left neighbour across the seam
  // shuffle sources and lane swaps of the x exchange (width BXC)
  const int src_l = tx == 0 ? bxr - 1 : tx - 1;
  const int src_r = tx == bxr - 1 ? 0 : tx + 1;

  // rows: own rows 2 tr, 2 tr + 1 of the tile; the first thread-row also
  // forms the equilibria of the row below the tile, the last one those of the
  // row above (staged with the tile)
  const int first_row = blockIdx.y * TY;  // rows before it are the previous tile's
  const int tile_row0 = RM == kRowsPlain ? first_row : min(first_row, ta.ny - TY);
  const int row0 = tile_row0 + 2 * tr;
  const int halo = tr == 0 ? 1 : (tr == TYT - 1 ? -1 : 0);
  // whether some thread of the warp has a halo row: its shuffles take the whole
  // warp.  (Beyond a closed y boundary the values are of no row; the row next to
  // it is a wall row and keeps its values.)
  const bool warp_halo = BXC >= 32 ? halo != 0 : true;
  bool row_wall[2];  // not stored: a wall row, or the previous tile's
  row_wall[0] = (!ta.py && row0 == 0) || (RM != kRowsPlain && row0 < first_row);
  row_wall[1] = (!ta.py && row0 + 1 == ta.ny - 1) || (RM != kRowsPlain && row0 + 1 < first_row);
  const int64_t row_off = (int64_t)row0 * ta.nx + 4 * tx;
  const bool x_lo_wall = ta.wall_mode == kWallBox && !ta.px && tx == 0;
  const bool x_hi_wall = ta.wall_mode == kWallBox && !ta.px && tx == (RM == kRowsPlain ? bxr - 1 : hi_wall_quad(ta.nx, ta.pad()));
  const bool box_x = ta.wall_mode == kWallBox && !ta.px;
  const bool per_node_store = ta.wall_mode == kWallMask || (x_lo_wall && x_hi_wall);
  // box x-walls: the lanes holding x = 0 or nx - 1 keep the wall node's values
  // of a staged plane (walls never change) in their own shared-memory slot
  // until the plane is stored, a plane later, instead of registers or a
  // global load at the store
  const bool keep_walls = !NU && box_x && (x_lo_wall || x_hi_wall) && !per_node_store;
  float* const WV = reinterpret_cast<float*>(smem_raw + Lay::wall_off);
  auto wall_slot = [&](int parity) { return ((parity * TYT + tr) * 2 + (x_hi_wall ? 1 : 0)) * 8; };

  // field f of this thread's quad in row j of plane 0: out + f * n + row_off + j * nx
  S* const op0 = out + row_off;
  const uint8_t* mrow = ta.wall_mode == kWallMask ? ta.mask + row_off : nullptr;
  P force[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) force[i] = O::splat(C(ta.force[i]));
  const int z0 = (int)(((int64_t)blockIdx.x * ta.nplanes) / ta.nzc);
  const int z1 = (int)(((int64_t)(blockIdx.x + 1) * ta.nplanes) / ta.nzc);
  const int64_t ps = ta.plane_stride;
  const int64_t nx64 = ta.nx;
  auto plane_exists = [&](int p) { return (p >= 0 && p < ta.nplanes) || ta.pz; };
  auto plane_mem = [&](int p) { return p < 0 ? p + ta.nplanes : (p >= ta.nplanes ? p - ta.nplanes : p); };
  const bool zwall = !ta.pz;

  // stage slots (Lay): own row j of this thread at row 2 tr + j of the own
  // block, the halo row below or above in its block; the tile copies write rows
  // of BXC quads (what lies beyond the end of a row is filled with zeros), so
  // every offset in a slot is a constant
  constexpr int QW = Quad<S>::BYTES;
  static_assert(kStages == 2, "two stage slots, two mbarriers");
  constexpr uint32_t rowB = (uint32_t)Lay::QB;
  constexpr uint32_t fieldB = (uint32_t)TY * rowB;  // own block: [4 fields][TY rows]
  const uint32_t own_off = (uint32_t)(2 * tr) * rowB + (uint32_t)tx * QW;
  const uint32_t halo_off = (uint32_t)(halo == 1 ? Lay::halo_lo : Lay::halo_hi) + (uint32_t)tx * QW;
  const uint32_t stage_sh = smem_u32(smem_raw);
  const int np = z1 - z0 + 2;  // planes z0 - 1 .. z1
  // halo rows of the tile (wrapped on a periodic y axis; none beyond a closed one)
  int lo_row = tile_row0 - 1, hi_row = tile_row0 + TY;
  bool lo_ok = true, hi_ok = true;
  if (lo_row < 0) {
    if (ta.py) lo_row += ta.ny;
    else lo_ok = false;
  }
  if (hi_row >= ta.ny) {
    if (ta.py) hi_row -= ta.ny;
    else hi_ok = false;
  }
  const uint32_t tile_bytes = 4 * fieldB + (lo_ok ? 4 * rowB : 0u) + (hi_ok ? 4 * rowB : 0u);
  // debug builds: a quad copy or load of 4 values at element offset e (from
  // `in` or `out`) and a stage byte offset b must lie in bounds
  const int64_t n4 = 4 * ta.n;
  const int64_t in_off = row_off;
  // plane z0 - 1 + i into slot i & 1: one thread copies the tile's own rows
  // and its halo rows of the four fields; a plane that does not exist (beyond
  // a closed march axis) completes the slot's phase with no bytes
  auto fetch = [&](int i) {
    if (!leader || i >= np) return;
    const int p = z0 - 1 + i;
    const uint32_t s = (uint32_t)(i & 1);
    const uint32_t bar = mbar0 + 8 * s;
    const uint32_t dst = stage_sh + s * (uint32_t)Lay::slot_bytes;
    if (plane_exists(p)) {
      const int pm = plane_mem(p);
      proxy_async_fence();  // the block's reads of this slot (before its last barrier) come first
      mbar_arrive_expect_tx(bar, tile_bytes);
      tma_load_4d(dst, &tm_own, 0, tile_row0, pm, 0, bar);
      if (lo_ok) tma_load_4d(dst + (uint32_t)Lay::halo_lo, &tm_halo, 0, lo_row, pm, 0, bar);
      if (hi_ok) tma_load_4d(dst + (uint32_t)Lay::halo_hi, &tm_halo, 0, hi_row, pm, 0, bar);
    } else {
      mbar_arrive(bar);
    }
  };
  const unsigned char* slot_base = smem_raw;
  int slot_parity = 0;
  auto take = [&](int i) {  // wait for plane z0 - 1 + i
    const uint32_t s = (uint32_t)(i & 1);
    if (!mbar_wait(mbar0 + 8 * s, (uint32_t)(i >> 1) & 1u) && ta.status) atomicOr(ta.status, 1u);
    slot_base = smem_raw + (size_t)s * Lay::slot_bytes;
    slot_parity = i & 1;
  };
  // a quad of the plane taken, at byte `off` of its field 0 and fields `stride` apart
  auto quad = [&](P(&v)[4][2], uint32_t off, uint32_t stride) {
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int64_t b = (int64_t)(slot_base - smem_raw) + off + f * stride;
      if (bounds_ok(ta.bounds, b, (int64_t)Lay::stage_bytes - QW + 1)) {
        Quad<S>::lds(reinterpret_cast<const S*>(smem_raw + b), v[f][0], v[f][1]);
      } else {
        v[f][0] = v[f][1] = O::splat(C(0));
      }
    }
  };

  // ---------------------------------------------------------------- one plane
  // a value of the lane holding the node pair at x - 1 / x + 1
  auto from_left = [&](P v) {
    v = fold_shfl<BXC>(v, src_l);
    return seam_l ? O::swap(v) : v;
  };
  auto from_right = [&](P v) {
    v = fold_shfl<BXC>(v, src_r);
    return seam_r ? O::swap(v) : v;
  };
  // Sums of plane p - 1 (cur: R, M_x, M_y, M_z) and what plane p - 1 sent on to
  // plane p (next: R = M_z, M_x, M_y), of [row][pair].
  P cur[2][2][4] = {}, next[2][2][3] = {};
  int ybuf = 0;
  auto unit = [&](float4* ybase, int sign, int val, int slot) {
    float4* const u = ybase + sign * Lay::SIGN_UNITS + val * Lay::VAL_UNITS + slot * BXC + tx;
    return bounds_ok(ta.bounds, u - Y, 2 * Lay::BUF_UNITS) ? u : nullptr;
  };
  auto publish = [&](float4* ybase, int sign, int val, int slot, P a, P b) {
    if (float4* const u = unit(ybase, sign, val, slot)) *u = make_float4(a.x, a.y, b.x, b.y);
  };
  auto receive = [&](float4* ybase, int sign, int val, int slot, P(&v)[2]) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (const float4* const u = unit(ybase, sign, val, slot)) t = *u;
    v[0] = O::make(t.x, t.y);
    v[1] = O::make(t.z, t.w);
  };

  // Source plane p: completes cur (plane p - 1), which stays for the store, and
  // leaves plane p's own sums in `own` and what it sends on in `next`.
  auto update = [&](auto mode, P(&own)[2][2][4]) {
    constexpr int MODE = decltype(mode)::value;
    constexpr bool kUp = MODE != kLast, kDown = MODE != kFirst, kOwn = MODE == kMid;
    float4* const ybase = Y + ybuf * Lay::BUF_UNITS;
    ybuf ^= 1;
    P down[2][2] = {};  // R of what goes to plane p - 1 (its M_z: the negative)
    P link[4][2] = {};  // what the lower row gets from the upper one
    // the row below (SIGN 1) or above (-1) adds (g, h, t of c_z = +1, t of c_z = -1)
    auto add_row = [&](auto signc, int j, int q, P g, P h, P tp, P tm) {
      constexpr int SIGN = decltype(signc)::value;
      auto signed_add = [](P x, P y) { return SIGN > 0 ? O::add(x, y) : O::sub(x, y); };
      if constexpr (kOwn) {
        own[j][q][0] = O::add(own[j][q][0], g);
        own[j][q][1] = O::add(own[j][q][1], h);
        own[j][q][2] = signed_add(own[j][q][2], g);
      }
      if constexpr (kDown) {
        down[j][q] = O::add(down[j][q], tm);
        cur[j][q][2] = signed_add(cur[j][q][2], tm);
      }
      if constexpr (kUp) {
        next[j][q][0] = O::add(next[j][q][0], tp);
        next[j][q][2] = SIGN > 0 ? tp : O::sub(next[j][q][2], tp);
      }
    };
    using Below = std::integral_constant<int, 1>;
    using Above = std::integral_constant<int, -1>;
    P up0[4][2] = {};   // what the upper row gets from the lower one
    static_for<0, 2>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      P st[4][2];
      quad(st, own_off + j * rowB, fieldB);
      if (keep_walls) {
        const int w = wall_slot(slot_parity) + 4 * j;
#pragma unroll
        for (int f = 0; f < 4; ++f)
          if (bounds_ok(ta.bounds, w + f, (int64_t)(Lay::wall_bytes / sizeof(float))))
            WV[w + f] = x_lo_wall ? st[f][0].x : (RM == kRowsOdd ? st[f][0].y : st[f][1].y);
      }
      const D3Node<C> a = d3_node<C, NU>(st[0][0], st[1][0], st[2][0], st[3][0]);
      const D3Node<C> b = d3_node<C, NU>(st[0][1], st[1][1], st[2][1], st[3][1]);
      D3Node<C> l, r;  // the neighbouring lanes' pair b and pair a
      l.ap = from_left(b.ap);
      l.bp = from_left(b.bp);
      l.dp = from_left(b.dp);
      l.e = from_left(b.e);
      l.f = from_left(b.f);
      r.am = from_right(a.am);
      r.bm = from_right(a.bm);
      r.dm = from_right(a.dm);
      r.e = from_right(a.e);
      r.f = from_right(a.f);
      P send[2][4][2];  // [below, above] of the values for the row above / below
      static_for<0, 2>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const D3Node<C>& n = q == 0 ? a : b;
        const D3Row<C> w = q == 0 ? d3_row<C, NU>(a, l, b) : d3_row<C, NU>(b, a, r);
        if constexpr (kDown) {
          down[j][q] = w.km;
          cur[j][q][1] = O::add(cur[j][q][1], w.xm);
        }
        if constexpr (kOwn) {
          own[j][q][0] = O::fma(n.A, O::splat(C(12)), O::fma(w.sA, O::splat(C(2)), next[j][q][0]));
          own[j][q][1] = O::fma(w.dA, O::splat(C(2)), next[j][q][1]);
          own[j][q][2] = next[j][q][2];
          own[j][q][3] = next[j][q][0];
        }
        if constexpr (kUp) {
          next[j][q][0] = w.kp;
          next[j][q][1] = w.xp;
        }
        send[0][0][q] = w.gp;
        send[0][1][q] = w.hp;
        send[0][2][q] = n.tpp;
        send[0][3][q] = n.tpm;
        send[1][0][q] = w.gm;
        send[1][1][q] = w.hm;
        send[1][2][q] = n.tmp;
        send[1][3][q] = n.tmm;
      });
      static_for<0, 4>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        if constexpr (rows2_sends<MODE>(k)) {
          if constexpr (j == 0) {
            publish(ybase, 1, k, tr, send[1][k][0], send[1][k][1]);  // to the thread-row below
            up0[k][0] = send[0][k][0];
            up0[k][1] = send[0][k][1];
          } else {
            publish(ybase, 0, k, tr + 1, send[0][k][0], send[0][k][1]);  // to the thread-row above
            link[k][0] = send[1][k][0];
            link[k][1] = send[1][k][1];
          }
        }
      });
      if constexpr (j == 1) {
#pragma unroll
        for (int q = 0; q < 2; ++q) add_row(Below{}, 1, q, up0[0][q], up0[1][q], up0[2][q], up0[3][q]);
      }
    });
    // ---- halo row: what it sends into the tile.  The row above the tile is the
    // mirror image in y of the row below it: with u_y negated it sends upwards
    // what it sends downwards.
    if (warp_halo) {
      P st[4][2];
      quad(st, halo_off, rowB);
      if (halo == -1) {
        st[2][0] = O::sub(O::splat(C(0)), st[2][0]);
        st[2][1] = O::sub(O::splat(C(0)), st[2][1]);
      }
      const D3Node<C> a = d3_node<C, NU>(st[0][0], st[1][0], st[2][0], st[3][0]);
      const D3Node<C> b = d3_node<C, NU>(st[0][1], st[1][1], st[2][1], st[3][1]);
      const int sign = halo == 1 ? 0 : 1, slot = halo == 1 ? 0 : TYT;
      if constexpr (kOwn) {
        D3Node<C> l = a, r = b;
        l.ap = from_left(b.ap);
        l.bp = from_left(b.bp);
        l.e = from_left(b.e);
        r.am = from_right(a.am);
        r.bm = from_right(a.bm);
        r.e = from_right(a.e);
        const D3Row<C> wa = d3_row<C, NU>(a, l, b), wb = d3_row<C, NU>(b, a, r);
        if (halo != 0) {
          publish(ybase, sign, 0, slot, wa.gp, wb.gp);
          publish(ybase, sign, 1, slot, wa.hp, wb.hp);
        }
      }
      if (halo != 0) {
        if constexpr (kUp) publish(ybase, sign, 2, slot, a.tpp, b.tpp);
        if constexpr (kDown) publish(ybase, sign, 3, slot, a.tpm, b.tpm);
      }
    }
    __syncthreads();
    P v[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k][0] = v[k][1] = O::splat(C(0));
    static_for<0, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (rows2_sends<MODE>(k)) receive(ybase, 0, k, tr, v[k]);
    });
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      add_row(Below{}, 0, q, v[0][q], v[1][q], v[2][q], v[3][q]);
      add_row(Above{}, 0, q, link[0][q], link[1][q], link[2][q], link[3][q]);
    }
    static_for<0, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      if constexpr (rows2_sends<MODE>(k)) receive(ybase, 1, k, tr + 1, v[k]);
    });
#pragma unroll
    for (int q = 0; q < 2; ++q) add_row(Above{}, 1, q, v[0][q], v[1][q], v[2][q], v[3][q]);
    if constexpr (kDown) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          cur[j][q][0] = O::add(cur[j][q][0], down[j][q]);
          cur[j][q][3] = O::sub(cur[j][q][3], down[j][q]);
        }
    }
  };

  // ---------------------------------------------------------------- store
  Rows2Sum nus;  // viscosity-term mode: this thread's sum
  // viscosity-term mode: the stored state after the step and lam of the plane
  // q the next store sums, loaded early so their latency overlaps the update
  P nsn[2][4][2], nlm[2][4][2];
  auto nu_prefetch = [&](int q) {
    if constexpr (NU) {
      const bool zskip = zwall && (q == 0 || q == ta.nplanes - 1);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool skip = !active || row_wall[j] || zskip || q < 0 || q >= ta.nplanes;
        const int64_t off = (int64_t)q * ps + j * nx64;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const int64_t e = f * ta.n + in_off + off;
          if (!skip && bounds_ok(ta.bounds, e, n4 - 3)) {
            Quad<S>::ld(out + e, nsn[j][f][0], nsn[j][f][1]);
            Quad<float>::ld(ta.lam + e, nlm[j][f][0], nlm[j][f][1]);
          } else {
            nsn[j][f][0] = nsn[j][f][1] = nlm[j][f][0] = nlm[j][f][1] = O::splat(C(0));
          }
        }
      }
    }
  };
  auto store = [&](int q, P(&acc)[2][2][4]) {
    const bool zskip = zwall && (q == 0 || q == ta.nplanes - 1);
    if constexpr (NU) {
      // the viscosity term of the fluid nodes of the two rows: R and u' of the
      // stored state after the step and lam, loaded by nu_prefetch(q) before
      // the plane update that precedes this store
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (!active || row_wall[j] || zskip) continue;
        const int64_t off = (int64_t)q * ps + j * nx64;
        const P(&sn)[4][2] = nsn[j];
        const P(&lm)[4][2] = nlm[j];
        // fluid lanes: (pair a.x, a.y, b.x, b.y) = storage positions 4 tx .. 4 tx + 3
        bool fl[4] = {!x_lo_wall, true, true, !x_hi_wall};
        if (ta.wall_mode == kWallMask && bounds_ok(ta.bounds, in_off + off, ta.n - 3)) {
          const uchar4 mk = *reinterpret_cast<const uchar4*>(mrow + off);
          fl[0] = mk.x == 0; fl[1] = mk.y == 0; fl[2] = mk.z == 0; fl[3] = mk.w == 0;
        }
        float part = 0.f;
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
          const P R = O::mul(sn[0][qq], O::splat(C(36)));
          const P inv = O::rcp(O::add(O::splat(C(36)), R));
          const P dR = O::sub(R, acc[j][qq][0]);
          const P dRi = O::mul(dR, inv);
          P t = O::mul(lm[0][qq], O::mul(dR, O::splat(C(-1.0 / 36.0))));
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const P unf = O::sub(sn[1 + i][qq], force[i]);
            const P du = O::sub(O::fma(unf, dRi, O::mul(acc[j][qq][1 + i], inv)), force[i]);
            t = O::fma(lm[1 + i][qq], du, t);
          }
          part += (fl[2 * qq] ? t.x : 0.f) + (fl[2 * qq + 1] ? t.y : 0.f);
        }
        nus.add(part);
      }
      return;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool skip = !active || row_wall[j] || zskip;
      const int64_t off = (int64_t)q * ps + j * nx64;
      if (per_node_store) {
        S* const fp[4] = {op0, op0 + ta.n, op0 + 2 * ta.n, op0 + 3 * ta.n};
        store_plane<kD3Q19, S, RM>(fp, mrow, ta, off, x_lo_wall, x_hi_wall, skip, acc[j], force);
        continue;
      }
      if (skip) continue;
      // box x-walls: the values kept when plane q was staged (take index q - z0 + 1)
      float wv[4] = {0.f, 0.f, 0.f, 0.f};
      if (keep_walls) {
        const int w = wall_slot((q - z0 + 1) & 1) + 4 * j;
#pragma unroll
        for (int f = 0; f < 4; ++f)
          if (bounds_ok(ta.bounds, w + f, (int64_t)(Lay::wall_bytes / sizeof(float)))) wv[f] = WV[w + f];
      }
      P v[4][2];
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        const P inv = O::rcp(O::add(O::splat(C(36)), acc[j][qq][0]));
        v[0][qq] = O::mul(acc[j][qq][0], O::splat(C(1.0 / 36.0)));
#pragma unroll
        for (int i = 0; i < 3; ++i) v[1 + i][qq] = O::fma(acc[j][qq][1 + i], inv, force[i]);
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        v[f][0].x = x_lo_wall ? wv[f] : v[f][0].x;
        if constexpr (RM == kRowsOdd) v[f][0].y = x_hi_wall ? wv[f] : v[f][0].y;
        else v[f][1].y = x_hi_wall ? wv[f] : v[f][1].y;
        if (bounds_ok(ta.bounds, f * ta.n + in_off + off, n4 - 3)) Quad<S>::st(op0 + f * ta.n + off, v[f][0], v[f][1]);
      }
    }
  };

  P own[2][2][4] = {};

#pragma unroll
  for (int i = 0; i < kStages - 1; ++i) fetch(i);
  // first (halo) plane z0 - 1: only what it sends up the march axis
  fetch(kStages - 1);
  take(0);
  // (the barrier inside update, or this one, keeps slot 0's next copy behind
  // every thread's wait for its current one)
  if (plane_exists(z0 - 1)) update(std::integral_constant<int, kFirst>{}, own);
  else __syncthreads();

  // full planes: after plane p, plane p - 1 is complete.  The loop body is not
  // unrolled: one copy of the two-row update keeps the code within the
  // instruction cache.
#pragma unroll 1
  for (int p = z0; p < z1; ++p) {
    const int i = p - z0 + 1;
    fetch(i + kStages - 1);
    nu_prefetch(p - 1);
    take(i);
    update(std::integral_constant<int, kMid>{}, own);
    if (p - 1 >= z0) store(p - 1, cur);
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) cur[j][q][k] = own[j][q][k];
  }
  // last (halo) plane z1: only what it sends down, to plane z1 - 1
  {
    const int i = np - 1;
    fetch(i + kStages - 1);
    nu_prefetch(z1 - 1);
    take(i);
    if (plane_exists(z1)) update(std::integral_constant<int, kLast>{}, own);
    store(z1 - 1, cur);
  }
  if constexpr (NU) {
    // block sum: warp shuffles, one value per warp, one FP64 atomic per block
    double v = (double)nus.hi + (double)nus.lo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __shared__ double red[32];
    const int lid = tr * BXC + tx;
    if ((lid & 31) == 0) red[lid >> 5] = v;
    __syncthreads();
    if (lid == 0) {
      double sum = 0.0;
      for (int w = 0; w < (BXC * TYT) / 32; ++w) sum += red[w];
      atomicAdd(ta.nu_acc, sum);
    }
  }
}

// The viscosity-term mode, FP32 storage (instances in step_rows2_nu.cu): rows
// without padding, any ny of at least a tile.
cudaError_t rows2_nu_dispatch(int bxc, int tyt, const TiledArgs& ta, const void* in, const void* out,
                              const CUtensorMap& tm_own, const CUtensorMap& tm_halo, cudaStream_t st, dim3 grid,
                              int* resident);

// Launch one instance.  With resident_out set,
// only report the blocks of this shape one SM holds.
template <typename S, int BXC, int TYT, bool NU = false, int RM = kRowsPlain>
cudaError_t launch_rows2_shape(const TiledArgs& ta, const void* in, void* out, const CUtensorMap& tm_own,
                               const CUtensorMap& tm_halo, cudaStream_t stream, dim3 grid, int* resident_out) {
  auto kern = step_rows2<S, BXC, TYT, NU, RM>;
  constexpr size_t smem = Rows2Layout<S, BXC, TYT>::smem;
  static int resident_dev[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int& resident = resident_dev[dev & 63];
  if (!resident) {
    // set whatever the size: static shared memory counts against the 48 KB
    // default as well
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, BXC * TYT, smem);
    if (e != cudaSuccess) return e;
    resident = nb < 1 ? 1 : nb;
  }
  if (resident_out) {
    *resident_out = resident;
    return cudaSuccess;
  }
  return launch_kernel(kern, grid, dim3(BXC, TYT), smem, stream, ta.overlap(), ta, static_cast<const S*>(in),
                       static_cast<S*>(out), tm_own, tm_halo);
}

// Launch of the instance (bxc, tyt) for storage type S and row mode RM
// (instances in step_rows2_f32*.cu and step_rows2_s16*.cu, which compile in
// parallel).
template <typename S, int RM>
cudaError_t rows2_dispatch(int bxc, int tyt, const TiledArgs& ta, const void* in, void* out,
                           const CUtensorMap& tm_own, const CUtensorMap& tm_halo, cudaStream_t st, dim3 grid,
                           int* resident) {
  switch (bxc * 100 + tyt) {
    case 1604: return launch_rows2_shape<S, 16, 4, false, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
    case 3202:
      if constexpr (sizeof(S) == 4)
        return launch_rows2_shape<S, 32, 2, false, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
      break;
    case 3204: return launch_rows2_shape<S, 32, 4, false, RM>(ta, in, out, tm_own, tm_halo, st, grid, resident);
  }
  return cudaErrorInvalidValue;
}
#define MACLAB_ROWS2_DISPATCH(EXTERN, S, RM)                                                                    \
  EXTERN template cudaError_t rows2_dispatch<S, RM>(int, int, const TiledArgs&, const void*, void*,             \
                                                     const CUtensorMap&, const CUtensorMap&, cudaStream_t, dim3, \
                                                     int*);

}  // namespace maclab
