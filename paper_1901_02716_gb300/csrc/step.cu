// step.cu -- the MacLAB time step (Eqs. (2), (4), (5)) on the GPU.
//
// Stored state: drho = rho / rho0 - 1 and ut = u / e, structure of arrays in
// storage order (see mem_x in common.cuh).
// With rho = 1 + drho and P_a = 3 c_a.ut + 9/2 (c_a.ut)^2 - 3/2 ut.ut, the
// equilibrium of Eq. (2) is f_a^eq = w_a (1 + drho + (1 + drho) P_a).  The
// constant w_a sums to 1 over a and w_a c_a sums to 0, so Eqs. (4)-(5) become
//   drho'(x) = sum_a w_a T_a(x - c_a),   m'(x) = sum_a w_a c_a T_a(x - c_a),
//   ut'(x)   = m'(x) / (1 + drho'(x)) + force,   T_a = drho + (1 + drho) P_a,
// in which every term is small: this is what keeps FP32 (and 16-bit storage)
// accurate.  Wall nodes are never written: both ping-pong buffers hold their
// values.  Periodic axes wrap; on closed axes a fluid node's upstream
// neighbours always exist because the outer layers are walls (checked on the
// host at create time).
//
// Kernels here:
//  * step_naive: one thread per node, the Q upstream states read straight from
//    global memory.  Any size; the reference the faster kernel is tested on.
//  * step_tiled (step_tiled.cu): strips of 4 nodes per thread, a march along
//    the slowest axis, equilibria exchanged through shared memory.

#include "common.cuh"
#include "lattice.cuh"

namespace maclab {

template <typename C>
struct Force {
  C f[3];
};

template <int LAT>
__device__ __forceinline__ bool is_wall_node(const Geometry& g, int x, int y, int z, int64_t node) {
  if (g.wall_mode == kWallNone) return false;
  if (g.wall_mode == kWallMask) return g.mask[node] != 0;
  bool w = false;
  if (!(g.periodic & 1u)) w |= (x == 0) | (x >= g.nx - 1 - g.pad);
  if (!(g.periodic & 2u)) w |= (y == 0) | (y == g.ny - 1);
  if (Lattice<LAT>::D == 3 && !(g.periodic & 4u)) w |= (z == 0) | (z == g.nz - 1);
  return w;
}

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// ------------------------------------------------------------------ naive kernel

template <int LAT, typename S>
__global__ void __launch_bounds__(256) step_naive(Geometry g, const S* __restrict__ in,
                                                  S* __restrict__ out,
                                                  Force<typename Store<S>::C> force) {
  using C = typename Store<S>::C;
  using L = Lattice<LAT>;
  constexpr int D = L::D;
  const int64_t N = g.n;
  for (int64_t node = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; node < N;
       node += (int64_t)gridDim.x * blockDim.x) {
    const int x = log_x(g, (int)(node % g.nx));
    const int y = (int)((node / g.nx) % g.ny);
    const int z = (int)(node / ((int64_t)g.nx * g.ny));
    if (is_wall_node<LAT>(g, x, y, z, node)) continue;
    C dr = 0, m[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < L::Q; ++a) {
      const int xs = wrap(x - L::c(a, 0), g.nx);
      const int ys = wrap(y - L::c(a, 1), g.ny);
      const int zs = D == 3 ? wrap(z - L::c(a, 2), g.nz) : 0;
      const int64_t s = ((int64_t)zs * g.ny + ys) * g.nx + mem_x(g, xs);
      const C r = Store<S>::ld(in + s);
      C u[3] = {Store<S>::ld(in + N + s), Store<S>::ld(in + 2 * N + s),
                D == 3 ? Store<S>::ld(in + 3 * N + s) : C(0)};
      C cu = 0, uu = 0;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        cu += C(L::c(a, i)) * u[i];
        uu += u[i] * u[i];
      }
      const C P = C(3) * cu + C(4.5) * cu * cu - C(1.5) * uu;
      const C T = (r + (C(1) + r) * P) * (C(L::w36(a)) / C(36));
      dr += T;
#pragma unroll
      for (int i = 0; i < D; ++i)
        if (L::c(a, i) != 0) m[i] += C(L::c(a, i)) * T;
    }
    const C inv = C(1) / (C(1) + dr);
    Store<S>::st(out + node, dr);
#pragma unroll
    for (int i = 0; i < D; ++i) Store<S>::st(out + (1 + i) * N + node, m[i] * inv + force.f[i]);
  }
}

// ------------------------------------------------------------------ dispatch

template <int LAT, typename S>
static cudaError_t launch_naive_t(const StepLaunch& s, cudaStream_t stream) {
  using C = typename Store<S>::C;
  Force<C> f{{C(s.force[0]), C(s.force[1]), C(s.force[2])}};
  const int threads = 256;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t blocks = (s.g.n + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  step_naive<LAT, S><<<(unsigned)blocks, threads, 0, stream>>>(
      s.g, static_cast<const S*>(s.in), static_cast<S*>(s.out), f);
  return cudaGetLastError();
}

template <int LAT>
static cudaError_t launch_naive_lat(const StepLaunch& s, cudaStream_t stream) {
  switch (s.precision) {
    case MACLAB_F64: return launch_naive_t<LAT, double>(s, stream);
    case MACLAB_F32: return launch_naive_t<LAT, float>(s, stream);
    case MACLAB_BF16_STORE: return launch_naive_t<LAT, __nv_bfloat16>(s, stream);
    case MACLAB_F16_STORE: return launch_naive_t<LAT, __half>(s, stream);
    default: return cudaErrorInvalidValue;
  }
}

// Time steps per launch of the segment kernel for the tile setting ty (2 asks
// for two steps per launch: FP32 or FP64 storage and nx >= 8; otherwise 1).
// Default: two with FP32 storage, which halves the state's traffic and the
// launches (1024^2: 4.71 us a step, 5.58 with one); FP64 is bound by its
// arithmetic, which the second step's halo rows add to, and takes two only on
// small grids, where the launches count.
int segment_depth(const Geometry& g, int precision, int ty) {
  const bool two_ok = (precision == MACLAB_F32 || precision == MACLAB_F64) && g.nx >= 8;
  if (ty == 0) return two_ok && (precision == MACLAB_F32 || (int64_t)(g.nx / 4) * g.ny < 200000) ? 2 : 1;
  return (ty == 2 || ty == 3) && two_ok ? 2 : 1;  // 3: two steps, runs in one persistent launch
}

// Rows per work item: asked for, or as few as make one wave of resident warps.
// Every item repeats the sums of the halo rows at its ends, and a second wave
// that is nearly empty costs as much as a full one (FP32 cavities, us a step,
// with the fixed rows before -> one wave: 1024^2 5.6 -> 4.7, 2048^2 14.2 -> 12.0,
// 4096^2 53.9 -> 40.1, 8192^2 173 -> 165).
int segment_rows(const Geometry& g, int precision, int ty, int tz) {
  if (tz > 0) return tz;
  const int depth = segment_depth(g, precision, ty);
  return batch_fit_rows({g.nx / 4}, {g.ny}, depth, batch_warp_slots(precision, depth));
}

bool step_kernel_supported(const Geometry& g, int precision, int kernel) {
  if (kernel == MACLAB_KERNEL_REFERENCE) return true;
  if (kernel == MACLAB_KERNEL_TILED) return tiled_supported(g, precision, 0, 0);
  if (kernel == MACLAB_KERNEL_FOLDED) return fold_supported(g, precision, 0);
  if (kernel == MACLAB_KERNEL_SEGMENT) return g.lattice == kD2Q9 && g.ilv == 1;
  if (kernel == MACLAB_KERNEL_ROWS2) return rows2_supported(g, precision, 0);
  if (kernel == MACLAB_KERNEL_BLOCK) return block_supported(g, precision, 0);
  return false;
}

// D3Q19 with 16-bit storage: the folded kernel wherever its tiles are whole rows
// of the caller's width.  The two-rows kernel is faster there (BF16 128^3: 14.1 us
// a step, folded 17.0), but it sums in another order, and every step's rounding to
// 16 bits shows that in the state (BF16 128^3, 20 steps: 1.2e-3 of the largest
// value): such runs and their checkpoints keep the values they have.  Else, and
// with FP32 storage, the two-rows-per-thread kernel where it applies (rows of up to
// 128 nodes), else the folded one where it is built (at least a tile of rows).
// D2Q9 grids with nx % 4 == 0: the block kernel
// with FP32 storage below 524,288 node pairs (us a step, block and segment
// kernel: 256^2 0.84 and 2.1, 560^2 1.77 and 2.91, 800^2 3.05 and 3.81, 1000^2
// 4.08 and 4.26, 1200^2 5.76 and 5.63, 2048^2 15.3 and 12.0) and with FP64
// storage up to 131,072 (1.9x to 2.4x), else the segment kernel; else the tiled
// one, else the reference kernel.
int pick_step_kernel(const Geometry& g, int precision) {
  const bool s16 = precision == MACLAB_BF16_STORE || precision == MACLAB_F16_STORE;
  if (s16 && g.pad == 0 && fold_supported(g, precision, 0)) return MACLAB_KERNEL_FOLDED;
  if (rows2_supported(g, precision, 0, true)) return MACLAB_KERNEL_ROWS2;
  if (fold_supported(g, precision, 0, true)) return MACLAB_KERNEL_FOLDED;
  if ((block_grid(g, precision) || !g.ilv) && block_supported(g, precision, 0, true))
    return MACLAB_KERNEL_BLOCK;  // natural rows have no other fast kernel
  if (step_kernel_supported(g, precision, MACLAB_KERNEL_SEGMENT)) return MACLAB_KERNEL_SEGMENT;
  return step_kernel_supported(g, precision, MACLAB_KERNEL_TILED) ? MACLAB_KERNEL_TILED
                                                                 : MACLAB_KERNEL_REFERENCE;
}

// D2Q9, closed x axis (the block kernel takes periodic ones as they are): whether the
// kernel that would serve the padded rows is faster than the one-thread-per-node
// kernel on natural ones (us a step, natural and padded).  Narrow rows leave lanes of
// the block kernel's 32 pairs and of the segment kernel's 28 quads idle, and a
// tall domain pays for them:
//   block, FP64:   17 x 1000 11.0 and 9.5, 17 x 2000 12.3 and 13.7, 25 x 6000 37.2 and
//                  40.7, 29 x 8000 55.3 and 53.5
//   segment, FP32 and 16 bits: 17 x 15882 BF16 8.2 and 7.8, 17 x 17647 8.2 and 8.7,
//                  25 x 24000 12.3 and 10.1, 17 x 64705 FP32 18.5 and 20.9
//   segment, FP64: 65 x 4153 64 and 78, 161 x 1863 72 and 79, 257 x 1167 74 and 65;
//                  57 x 10526 143 and 140, 49 x 12244 143 and 164
static bool pad_pays_2d(const Geometry& g, int precision, int kernel) {
  const int64_t n = (int64_t)(g.nx - g.pad) * g.ny;
  if (kernel == MACLAB_KERNEL_BLOCK) return precision != MACLAB_F64 || g.nx >= 32 || n < 20000;
  if (precision != MACLAB_F64) return g.nx >= 28 || n < 270000;
  const int quads = g.nx / 4, segments = (quads + kBatchSegW2 - 1) / kBatchSegW2;
  return 2 * quads >= (n >= 500000 ? 29 : 43) * segments;
}

// D3Q19: where the two-rows or the folded kernel takes the padded rows (or the tiled
// one in a single tile: 63 x 7 x 400 10.2 and 6.2; elsewhere its halo rows cost more:
// 131 x 3 x 150 6.2 and 7.6), so not with FP64 storage, rows of more than 512 nodes or
// 16-bit rows of other than whole 16 bytes, which stay on the one-thread-per-node
// kernel and only slow it down (513 x 40 x 40 26.8 and 29.4, BF16 51^3 8.2 and 9.5;
// FP64 45^3 66, 148 on the tiled kernel), and only where the fast kernels' longer
// start pays (us a step, natural and padded rows, FP32: closed 33^3 3.7 and 4.0,
// 37^3 4.2 and 3.8, 63^3 9.5 and 5.1; periodic, with the images' extra launch,
// 51^3 6.3 and 6.7, 55^3 7.8 and 6.8, 79^3 16.2 and 10.5).
static bool pad_pays_3d(const Geometry& g, int precision, int kernel) {
  const int64_t n = (int64_t)(g.nx - g.pad) * g.ny * g.nz;
  if (n < ((g.periodic & 1u) ? 150000 : 50000)) return false;
  return kernel == MACLAB_KERNEL_ROWS2 || kernel == MACLAB_KERNEL_FOLDED ||
         (kernel == MACLAB_KERNEL_TILED && precision != MACLAB_F64 && g.nx <= 64);
}

// At least 17 nodes wide, so that two quads lie between the two x-walls and no
// quad holds both.  Padded and natural rows run kernels that sum in different orders,
// so the slabs of a domain all follow the choice of the whole.
void pad_rows(Geometry* g, int precision, int64_t planes) {
  const bool px = (g->periodic & 1u) != 0;
  if (g->nx % 4 == 0 || g->nx < 17 || (g->d == 2 && px)) return;
  Geometry p = *g;
  p.pad = (g->nx + (px ? 2 : 0) + 3) / 4 * 4 - g->nx;
  p.nx += p.pad;
  p.n = (int64_t)p.nx * p.ny * p.nz;
  p.ilv = 1;
  p.hx = p.nx / 2;
  Geometry whole = p;
  (g->d == 2 ? whole.ny : whole.nz) = (int)planes;
  whole.n = (int64_t)whole.nx * whole.ny * whole.nz;
  const int kernel = pick_step_kernel(whole, precision);
  if (g->d == 2 ? pad_pays_2d(whole, precision, kernel) : pad_pays_3d(whole, precision, kernel)) *g = p;
}

static const char* kernel_name(const Geometry& g, int precision, int kernel) {
  if (kernel == MACLAB_KERNEL_ROWS2) {
    static const char* rows2[4] = {"step_rows2<D3Q19,f64>", "step_rows2<D3Q19,f32>", "step_rows2<D3Q19,bf16>",
                                   "step_rows2<D3Q19,f16>"};
    return rows2[precision & 3];
  }
  if (kernel == MACLAB_KERNEL_FOLDED) {
    static const char* fold[4] = {"step_fold<D3Q19,f64>", "step_fold<D3Q19,f32>", "step_fold<D3Q19,bf16>",
                                  "step_fold<D3Q19,f16>"};
    return fold[precision & 3];
  }
  if (kernel == MACLAB_KERNEL_BLOCK) {
    static const char* blk[4] = {"step_block<D2Q9,f64>", "step_block<D2Q9,f32>", "step_block<D2Q9,bf16>",
                                 "step_block<D2Q9,f16>"};
    return blk[precision & 3];
  }
  if (kernel == MACLAB_KERNEL_SEGMENT) {
    static const char* seg[4] = {"segment<D2Q9,f64>", "segment<D2Q9,f32>", "segment<D2Q9,bf16>",
                                 "segment<D2Q9,f16>"};
    return seg[precision & 3];
  }
  static const char* names[2][2][4] = {
      {{"step_naive<D2Q9,f64>", "step_naive<D2Q9,f32>", "step_naive<D2Q9,bf16>",
        "step_naive<D2Q9,f16>"},
       {"step_naive<D3Q19,f64>", "step_naive<D3Q19,f32>", "step_naive<D3Q19,bf16>",
        "step_naive<D3Q19,f16>"}},
      {{"step_tiled<D2Q9,f64>", "step_tiled<D2Q9,f32>", "step_tiled<D2Q9,bf16>",
        "step_tiled<D2Q9,f16>"},
       {"step_tiled<D3Q19,f64>", "step_tiled<D3Q19,f32>", "step_tiled<D3Q19,bf16>",
        "step_tiled<D3Q19,f16>"}}};
  return names[kernel == MACLAB_KERNEL_TILED ? 1 : 0][g.lattice == kD2Q9 ? 0 : 1][precision & 3];
}

static KernelInfo describe_kernel(const Geometry& g, int precision, int kernel, int ty, int tz) {
  if (kernel == MACLAB_KERNEL_TILED)
    return KernelInfo{MACLAB_KERNEL_TILED, 1, 1, tiled_threads(g, precision, ty, tz),
                      kernel_name(g, precision, kernel)};
  if (kernel == MACLAB_KERNEL_FOLDED)
    return KernelInfo{MACLAB_KERNEL_FOLDED, 1, 1, fold_threads(g, precision, ty),
                      kernel_name(g, precision, kernel)};
  if (kernel == MACLAB_KERNEL_ROWS2)
    return KernelInfo{MACLAB_KERNEL_ROWS2, 1, 1, rows2_threads(g, precision, ty), kernel_name(g, precision, kernel)};
  if (kernel == MACLAB_KERNEL_BLOCK)
    return KernelInfo{MACLAB_KERNEL_BLOCK, block_steps(g, precision, ty), 1,
                      block_threads(g, precision, block_steps(g, precision, ty)),
                      kernel_name(g, precision, kernel)};

  if (kernel == MACLAB_KERNEL_SEGMENT) {
    const int depth = segment_depth(g, precision, ty);
    return KernelInfo{MACLAB_KERNEL_SEGMENT, depth, 1, depth == 2 ? 128 : 256, kernel_name(g, precision, kernel)};
  }
  return KernelInfo{MACLAB_KERNEL_REFERENCE, 1, 1, 256, kernel_name(g, precision, kernel)};
}

static cudaError_t launch_step_kernel(const StepLaunch& s, cudaStream_t stream, int kernel) {
  switch (kernel) {
    case MACLAB_KERNEL_REFERENCE:
      return s.g.lattice == kD2Q9 ? launch_naive_lat<kD2Q9>(s, stream)
                                  : launch_naive_lat<kD3Q19>(s, stream);
    case MACLAB_KERNEL_TILED:
      return launch_tiled(s, stream, s.ty, s.tz);
    case MACLAB_KERNEL_FOLDED:
      return launch_fold(s, stream, s.ty, s.tz);
    case MACLAB_KERNEL_ROWS2:
      return launch_rows2(s, stream, s.ty, s.tz);
    case MACLAB_KERNEL_BLOCK:
      return launch_block(s, stream, s.seg_steps);
    case MACLAB_KERNEL_SEGMENT:
      if (!s.seg_inst || !s.seg_items) return cudaErrorInvalidValue;
      if (s.seg_steps == 2)
        return launch_batch_step2(s.precision, s.seg_inst, s.seg_items, s.seg_n_items, s.cur, s.seg_blocks,
                                  (s.g.pad & 1) != 0, stream, s.overlap);
      if (s.seg_depth != 1) return cudaErrorInvalidValue;  // cut for another segment width
      return launch_batch_step(s.precision, s.seg_inst, s.seg_items, s.seg_n_items, s.cur, s.seg_blocks,
                               (s.g.pad & 1) != 0, stream, s.overlap);
    default:
      return cudaErrorInvalidValue;
  }
}

KernelInfo describe_step_kernel(const Geometry& g, int precision, int kernel, int ty, int tz) {
  KernelInfo k = describe_kernel(g, precision, kernel, ty, tz);
  if (wrap_columns(g)) ++k.launches;  // the periodic images
  return k;
}

cudaError_t launch_step(const StepLaunch& s, cudaStream_t stream, int kernel) {
  const cudaError_t e = launch_step_kernel(s, stream, kernel);
  if (e != cudaSuccess || !wrap_columns(s.g)) return e;
  return launch_wrap_columns(s.g, s.precision, s.out, stream, s.overlap);
}

}  // namespace maclab
