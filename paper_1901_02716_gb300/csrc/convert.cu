// convert.cu -- unit maps at the boundary of the library.
//
// Physical (rho, u) <-> stored lattice state (drho = rho / rho0 - 1, ut = u / e)
// with e = 6 nu / dx (Eq. (6)).  Wall nodes take their wall id's values
// (procedure step (iv): physical variables are retained on walls).  User
// arrays are in logical order; the state and the device node-type copy in
// storage order.
//
// The maps are defined in FP64 and rounded once to the arithmetic type.  Done
// literally that costs two FP64 operations and two conversions per value on a
// pipe of two lanes per SM: it bounded these kernels (512^3 FP32: 3.18 ms for
// 4.3 GB in and out, 20 % of the copy bandwidth).  With 32-bit user arrays and 32-bit
// arithmetic the same values come from the FP32 pipe (UnitMap):
//  * rho0 a power of two: v / rho0 - 1 and rho0 (1 + drho) are one exact
//    scaling and one FP32 rounding, as from FP64;
//  * e and 1 / e as a sum of two floats (48 bits): the leading product's error
//    is exact from an fma, so the one rounding that counts is the last, and
//    only a value within 2^-23 ulp of a rounding boundary can differ.
// Other rho0, an e whose two floats would leave the normal range, and FP64
// arrays or storage keep the FP64 form.
// Now bound by memory: 512^3 FP32 set 0.77 ms, get 0.61 ms (5.6 and 7.0 TB/s);
// setting no longer copies the state to the other buffer either (0.64 ms more).

#include "units.cuh"

namespace maclab {

// Both state buffers are given: wall nodes are written into both (the step
// kernels never write them), fluid nodes into s0 only, as every step writes
// all fluid nodes of the buffer it fills.
template <typename S, typename T, bool FAST, typename I, int U>
__global__ void __launch_bounds__(256) set_physical_k(Geometry g, const T* __restrict__ rho, const T* __restrict__ u,
                                                      UnitMap m, const uint8_t* __restrict__ node_type,
                                                      const double* __restrict__ wall_lat, int n_wall_ids,
                                                      S* __restrict__ s0, S* __restrict__ s1) {
  using MP = Map<S, FAST>;
  const int64_t N = g.n, NU = m.nu;  // field strides: state, user arrays
  const int d = g.d;
  for_units<I, U>(g, [&](int64_t i, int64_t j, int x) {
    if constexpr (U != kNode) {
      Four<S> q[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (f > d) continue;
        T v[4];
        ld_user<U, T>(g, f == 0 ? rho : u + (f - 1) * NU, j, x, v);
#pragma unroll
        for (int c = 0; c < 4; ++c) q[f].v[c] = f == 0 ? MP::rho_in(v[c], m) : MP::u_in(v[c], m);
      }
      bool any = false;
      if (node_type) {
        const uchar4 k4 = *reinterpret_cast<const uchar4*>(node_type + i);
        const int k[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (k[c] > 0 && k[c] <= n_wall_ids) {
            any = true;
            const double* w = wall_lat + 4 * (k[c] - 1);
#pragma unroll
            for (int f = 0; f < 4; ++f)
              if (f <= d) q[f].v[c] = Store<S>::to(typename Store<S>::C(w[f]));
          }
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (f > d) continue;
        *reinterpret_cast<Four<S>*>(s0 + f * N + i) = q[f];
        if (any) *reinterpret_cast<Four<S>*>(s1 + f * N + i) = q[f];
      }
    } else {
      const int k = node_type ? (int)node_type[i] : 0;
      if (k > 0 && k <= n_wall_ids) {
        const double* w = wall_lat + 4 * (k - 1);
        for (int f = 0; f <= d; ++f) s0[f * N + i] = s1[f * N + i] = Store<S>::to(typename Store<S>::C(w[f]));
      } else {
        s0[i] = MP::rho_in(rho[j], m);
        for (int c = 0; c < d; ++c) s0[(1 + c) * N + i] = MP::u_in(u[c * N + j], m);
      }
    }
  });
}

template <typename S>
__global__ void fill_walls_k(int d, int64_t N, const uint8_t* __restrict__ node_type,
                             const double* __restrict__ wall_lat, int n_wall_ids,
                             S* __restrict__ state) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)node_type[i];
    if (k > 0 && k <= n_wall_ids) {
      const double* w = wall_lat + 4 * (k - 1);
      state[i] = Store<S>::to(typename Store<S>::C(w[0]));
      for (int c = 0; c < d; ++c) state[(1 + c) * N + i] = Store<S>::to(typename Store<S>::C(w[1 + c]));
    }
  }
}

// Per-node wall values: every wall node (node type > 0) takes the given
// physical (rho, u), in both state buffers (the step kernels never write a
// wall node, so whichever buffer is current reads them); fluid entries of the
// arrays are not read.
template <typename S, typename T, bool FAST, typename I, int U>
__global__ void __launch_bounds__(256) set_walls_k(Geometry g, const T* __restrict__ rho, const T* __restrict__ u,
                                                   UnitMap m, const uint8_t* __restrict__ node_type,
                                                   S* __restrict__ s0, S* __restrict__ s1) {
  using MP = Map<S, FAST>;
  const int64_t N = g.n, NU = m.nu;
  for_units<I, U>(g, [&](int64_t i, int64_t j, int x) {
    if constexpr (U != kNode) {
      const uchar4 k4 = *reinterpret_cast<const uchar4*>(node_type + i);
      const bool wall[4] = {k4.x != 0, k4.y != 0, k4.z != 0, k4.w != 0};
      if (!(wall[0] | wall[1] | wall[2] | wall[3])) return;
      for (int f = 0; f <= g.d; ++f) {
        T v[4];
        ld_user<U, T>(g, f == 0 ? rho : u + (f - 1) * NU, j, x, v);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (wall[c]) s0[f * N + i + c] = s1[f * N + i + c] = f == 0 ? MP::rho_in(v[c], m) : MP::u_in(v[c], m);
      }
    } else {
      if (node_type[i] == 0) return;
      s0[i] = s1[i] = MP::rho_in(rho[j], m);
      for (int c = 0; c < g.d; ++c) s0[(1 + c) * N + i] = s1[(1 + c) * N + i] = MP::u_in(u[c * NU + j], m);
    }
  });
}

// The wall nodes of one raw state into the other buffer.  W: nodes a thread looks at,
// four where the fields are whole quads (one by one the look alone took longer than
// copying a whole 16-bit state: 128^3 BF16 16.1 us a maclab_set_lattice_state, 12.3).
template <typename S, int W>
__global__ void __launch_bounds__(256) copy_walls_k(int d, int64_t N, const uint8_t* __restrict__ node_type,
                                                    const S* __restrict__ src, S* __restrict__ dst) {
  const int64_t i = W * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
  if (i >= N) return;
  if constexpr (W == 4) {
    const uchar4 k = *reinterpret_cast<const uchar4*>(node_type + i);
    const bool wall[4] = {k.x != 0, k.y != 0, k.z != 0, k.w != 0};
    if (!(wall[0] | wall[1] | wall[2] | wall[3])) return;
    Four<S> v[4];
#pragma unroll
    for (int f = 0; f < 4; ++f)
      if (f <= d) v[f] = *reinterpret_cast<const Four<S>*>(src + f * N + i);
#pragma unroll
    for (int f = 0; f < 4; ++f)
      if (f <= d) {
        if (wall[0] & wall[1] & wall[2] & wall[3]) {
          *reinterpret_cast<Four<S>*>(dst + f * N + i) = v[f];
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (wall[c]) dst[f * N + i + c] = v[f].v[c];
        }
      }
  } else {
    if (node_type[i] == 0) return;
    for (int f = 0; f <= d; ++f) dst[f * N + i] = src[f * N + i];
  }
}

template <typename S>
static cudaError_t copy_walls_t(const Geometry& g, const uint8_t* nt, const void* src, void* dst, cudaStream_t st) {
  if (g.n % 4 == 0)
    copy_walls_k<S, 4><<<(unsigned)((g.n / 4 + 255) / 256), 256, 0, st>>>(g.d, g.n, nt, (const S*)src, (S*)dst);
  else
    copy_walls_k<S, 1><<<(unsigned)((g.n + 255) / 256), 256, 0, st>>>(g.d, g.n, nt, (const S*)src, (S*)dst);
  return cudaGetLastError();
}

// Rows of planes [p0, p0 + count) between padded storage and the raw layout
// (kQuad1 units of the rows; `rows` rows a field).  Into the state, quads with walls
// (node_type, of the state's rows) go to the other buffer as well where it is given.
template <typename S, typename I, bool TO_RAW>
__global__ void __launch_bounds__(256) repack_k(Geometry g, int64_t row0, int64_t rows, S* __restrict__ state,
                                                S* __restrict__ raw, S* __restrict__ other,
                                                const uint8_t* __restrict__ node_type) {
  const int64_t N = g.n, NU = rows * (g.nx - g.pad);
  Geometry part = g;  // the planes' rows only
  part.n = rows * g.nx;
  for_units<I, kQuad1>(part, [&](int64_t i, int64_t j, int x) {
    const int64_t at = row0 * g.nx + i;
    const bool walls = !TO_RAW && other && *reinterpret_cast<const uint32_t*>(node_type + at) != 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      if (f > g.d) continue;
      Four<S>* const q = reinterpret_cast<Four<S>*>(state + f * N + at);
      if constexpr (TO_RAW) {
        const Four<S> v = *q;
        st_user<kQuad1, S>(g, raw + f * NU, j, x, v.v);
      } else {
        Four<S> v;
        ld_user<kQuad1, S>(g, raw + f * NU, j, x, v.v);
        *q = v;
        if (walls) *reinterpret_cast<Four<S>*>(other + f * N + at) = v;
      }
    }
  });
}

template <typename S, typename T, bool FAST, typename I, int U>
__global__ void __launch_bounds__(256) get_physical_k(Geometry g, const S* __restrict__ state, UnitMap m,
                                                      T* __restrict__ rho, T* __restrict__ u) {
  using MP = Map<S, FAST>;
  const int64_t N = g.n, NU = m.nu;  // field strides: state, user arrays
  const int d = g.d;
  for_units<I, U>(g, [&](int64_t i, int64_t j, int x) {
    if constexpr (U != kNode) {
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        if (f > d) continue;
        const Four<S> q = *reinterpret_cast<const Four<S>*>(state + f * N + i);
        T v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          v[c] = f == 0 ? MP::template rho_out<T>(q.v[c], m) : MP::template u_out<T>(q.v[c], m);
        st_user<U, T>(g, f == 0 ? rho : u + (f - 1) * NU, j, x, v);
      }
    } else {
      rho[j] = MP::template rho_out<T>(state[i], m);
      for (int c = 0; c < d; ++c) u[c * N + j] = MP::template u_out<T>(state[(1 + c) * N + i], m);
    }
  });
}

template <typename S, typename T, bool FAST>
static cudaError_t set_t(const Geometry& g, const void* rho, const void* u, const UnitMap& m, const uint8_t* nt,
                         const double* wl, int nw, void* s0, void* s1, cudaStream_t st) {
  return by_unit(g, unit_of(g, rho, u, 2 * sizeof(T)), [&](unsigned grid, unsigned threads, auto index, auto unit) {
    set_physical_k<S, T, FAST, decltype(index), decltype(unit)::value>
        <<<grid, threads, 0, st>>>(g, (const T*)rho, (const T*)u, m, nt, wl, nw, (S*)s0, (S*)s1);
    return cudaGetLastError();
  });
}

template <typename S>
static cudaError_t set_s(const Geometry& g, const void* rho, const void* u, int dtype, double rho0, double e,
                         const uint8_t* nt, const double* wl, int nw, void* s0, void* s1, cudaStream_t st) {
  UnitMap m;
  const bool fast = unit_map(g, rho0, e, &m);
  if (dtype == MACLAB_DTYPE_F64) return set_t<S, double, false>(g, rho, u, m, nt, wl, nw, s0, s1, st);
  if constexpr (!std::is_same<S, double>::value)
    if (fast) return set_t<S, float, true>(g, rho, u, m, nt, wl, nw, s0, s1, st);
  return set_t<S, float, false>(g, rho, u, m, nt, wl, nw, s0, s1, st);
}

cudaError_t launch_set_physical(const Geometry& g, int precision, const void* rho, const void* u, int dtype,
                                double rho0, double e, const uint8_t* nt, const double* wl, int nw, void* state,
                                void* other, cudaStream_t st) {
  switch (precision) {
    case MACLAB_F64: return set_s<double>(g, rho, u, dtype, rho0, e, nt, wl, nw, state, other, st);
    case MACLAB_F32: return set_s<float>(g, rho, u, dtype, rho0, e, nt, wl, nw, state, other, st);
    case MACLAB_BF16_STORE: return set_s<__nv_bfloat16>(g, rho, u, dtype, rho0, e, nt, wl, nw, state, other, st);
    case MACLAB_F16_STORE: return set_s<__half>(g, rho, u, dtype, rho0, e, nt, wl, nw, state, other, st);
  }
  return cudaErrorInvalidValue;
}

template <typename S, typename T, bool FAST>
static cudaError_t get_t(const Geometry& g, const void* state, const UnitMap& m, void* rho, void* u, cudaStream_t st) {
  return by_unit(g, unit_of(g, rho, u, 2 * sizeof(T)), [&](unsigned grid, unsigned threads, auto index, auto unit) {
    get_physical_k<S, T, FAST, decltype(index), decltype(unit)::value>
        <<<grid, threads, 0, st>>>(g, (const S*)state, m, (T*)rho, (T*)u);
    return cudaGetLastError();
  });
}

template <typename S>
static cudaError_t get_s(const Geometry& g, const void* state, void* rho, void* u, int dtype, double rho0, double e,
                         cudaStream_t st) {
  UnitMap m;
  const bool fast = unit_map(g, rho0, e, &m);
  if (dtype == MACLAB_DTYPE_F64) return get_t<S, double, false>(g, state, m, rho, u, st);
  if constexpr (!std::is_same<S, double>::value)
    if (fast) return get_t<S, float, true>(g, state, m, rho, u, st);
  return get_t<S, float, false>(g, state, m, rho, u, st);
}

cudaError_t launch_get_physical(const Geometry& g, int precision, const void* state, void* rho, void* u, int dtype,
                                double rho0, double e, cudaStream_t st) {
  switch (precision) {
    case MACLAB_F64: return get_s<double>(g, state, rho, u, dtype, rho0, e, st);
    case MACLAB_F32: return get_s<float>(g, state, rho, u, dtype, rho0, e, st);
    case MACLAB_BF16_STORE: return get_s<__nv_bfloat16>(g, state, rho, u, dtype, rho0, e, st);
    case MACLAB_F16_STORE: return get_s<__half>(g, state, rho, u, dtype, rho0, e, st);
  }
  return cudaErrorInvalidValue;
}

template <typename S, typename T, bool FAST>
static cudaError_t walls_t(const Geometry& g, const void* rho, const void* u, const UnitMap& m, const uint8_t* nt,
                           void* s0, void* s1, cudaStream_t st) {
  return by_unit(g, unit_of(g, rho, u, 2 * sizeof(T)), [&](unsigned grid, unsigned threads, auto index, auto unit) {
    set_walls_k<S, T, FAST, decltype(index), decltype(unit)::value>
        <<<grid, threads, 0, st>>>(g, (const T*)rho, (const T*)u, m, nt, (S*)s0, (S*)s1);
    return cudaGetLastError();
  });
}

template <typename S>
static cudaError_t walls_s(const Geometry& g, const void* rho, const void* u, int dtype, double rho0, double e,
                           const uint8_t* nt, void* s0, void* s1, cudaStream_t st) {
  UnitMap m;
  const bool fast = unit_map(g, rho0, e, &m);
  if (dtype == MACLAB_DTYPE_F64) return walls_t<S, double, false>(g, rho, u, m, nt, s0, s1, st);
  if constexpr (!std::is_same<S, double>::value)
    if (fast) return walls_t<S, float, true>(g, rho, u, m, nt, s0, s1, st);
  return walls_t<S, float, false>(g, rho, u, m, nt, s0, s1, st);
}

cudaError_t launch_set_wall_values(const Geometry& g, int precision, const void* rho, const void* u,
                                   int dtype, double rho0, double e, const uint8_t* nt, void* s0,
                                   void* s1, cudaStream_t st) {
  if (!nt) return cudaSuccess;
  switch (precision) {
    case MACLAB_F64: return walls_s<double>(g, rho, u, dtype, rho0, e, nt, s0, s1, st);
    case MACLAB_F32: return walls_s<float>(g, rho, u, dtype, rho0, e, nt, s0, s1, st);
    case MACLAB_BF16_STORE: return walls_s<__nv_bfloat16>(g, rho, u, dtype, rho0, e, nt, s0, s1, st);
    case MACLAB_F16_STORE: return walls_s<__half>(g, rho, u, dtype, rho0, e, nt, s0, s1, st);
  }
  return cudaErrorInvalidValue;
}

template <typename S>
static cudaError_t repack_t(const Geometry& g, void* state, void* raw, int64_t row0, int64_t rows, bool to_raw,
                            void* other, const uint8_t* nt, cudaStream_t st) {
  const unsigned grid = grid_for(rows * g.nx / 4);
  S* const s = (S*)state;
  S* const r = (S*)raw;
  S* const o = nt ? (S*)other : nullptr;
  if (small_index(g.n)) {
    if (to_raw) repack_k<S, uint32_t, true><<<grid, 256, 0, st>>>(g, row0, rows, s, r, o, nt);
    else repack_k<S, uint32_t, false><<<grid, 256, 0, st>>>(g, row0, rows, s, r, o, nt);
  } else {
    if (to_raw) repack_k<S, int64_t, true><<<grid, 256, 0, st>>>(g, row0, rows, s, r, o, nt);
    else repack_k<S, int64_t, false><<<grid, 256, 0, st>>>(g, row0, rows, s, r, o, nt);
  }
  return cudaGetLastError();
}

cudaError_t launch_repack(const Geometry& g, int precision, void* state, void* raw, int64_t p0, int64_t count,
                          bool to_raw, cudaStream_t st, void* other, const uint8_t* nt) {
  const int64_t plane_rows = g.d == 3 ? g.ny : 1;
  switch (storage_bytes(precision)) {
    case 8: return repack_t<double>(g, state, raw, p0 * plane_rows, count * plane_rows, to_raw, other, nt, st);
    case 4: return repack_t<float>(g, state, raw, p0 * plane_rows, count * plane_rows, to_raw, other, nt, st);
    case 2: return repack_t<uint16_t>(g, state, raw, p0 * plane_rows, count * plane_rows, to_raw, other, nt, st);
  }
  return cudaErrorInvalidValue;
}

// One thread copies a row's two images in one field.
template <typename S>
__global__ void __launch_bounds__(256) wrap_columns_k(int64_t count, int nx, int first, int last, int image0,
                                                      S* __restrict__ state) {
  pdl_wait();  // the step before this kernel has completed and its writes are visible
  pdl_launch_next();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  S* const row = state + k * nx;  // fields follow one another: row k of the whole state
  row[image0] = row[first];
  row[nx - 1] = row[last];
}

template <typename S>
static cudaError_t wrap_t(const Geometry& g, void* state, cudaStream_t st, int overlap) {
  const int64_t count = g.n / g.nx * (g.d + 1);
  const int nx = g.nx - g.pad;
  return launch_kernel(wrap_columns_k<S>, dim3((unsigned)((count + 255) / 256)), dim3(256), 0, st, overlap, count, g.nx,
                       mem_x(g, 0), mem_x(g, nx - 1), mem_x(g, nx), (S*)state);
}

cudaError_t launch_wrap_columns(const Geometry& g, int precision, void* state, cudaStream_t st, int overlap) {
  switch (storage_bytes(precision)) {
    case 8: return wrap_t<double>(g, state, st, overlap);
    case 4: return wrap_t<float>(g, state, st, overlap);
    case 2: return wrap_t<uint16_t>(g, state, st, overlap);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_copy_walls(const Geometry& g, int precision, const uint8_t* nt, const void* src, void* dst,
                              cudaStream_t st) {
  if (!nt) return cudaSuccess;
  switch (storage_bytes(precision)) {
    case 8: return copy_walls_t<double>(g, nt, src, dst, st);
    case 4: return copy_walls_t<float>(g, nt, src, dst, st);
    case 2: return copy_walls_t<uint16_t>(g, nt, src, dst, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fill_walls(const Geometry& g, int precision, const uint8_t* nt, const double* wl,
                              int nw, void* state, cudaStream_t st) {
  if (!nt) return cudaSuccess;
  switch (precision) {
    case MACLAB_F64:
      fill_walls_k<double><<<grid_for(g.n), 256, 0, st>>>(g.d, g.n, nt, wl, nw, (double*)state);
      break;
    case MACLAB_F32:
      fill_walls_k<float><<<grid_for(g.n), 256, 0, st>>>(g.d, g.n, nt, wl, nw, (float*)state);
      break;
    case MACLAB_BF16_STORE:
      fill_walls_k<__nv_bfloat16><<<grid_for(g.n), 256, 0, st>>>(g.d, g.n, nt, wl, nw,
                                                                 (__nv_bfloat16*)state);
      break;
    case MACLAB_F16_STORE:
      fill_walls_k<__half><<<grid_for(g.n), 256, 0, st>>>(g.d, g.n, nt, wl, nw, (__half*)state);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace maclab
