// units.cuh -- unit maps between physical values and the stored lattice state,
// and the walk over storage quads and user arrays (the kernels of convert.cu,
// which has the reasons, and the ends of the reverse pass in adjoint.cu).
#pragma once
#include <math.h>

#include <type_traits>

#include "common.cuh"

namespace maclab {

// The unit maps: stored = v * inv_rho0 - 1 and v * inv_e; physical = rho0 (1 + v) and e v.
struct UnitMap {
  double rho0, e, inv_rho0, inv_e;
  float f_rho0, f_inv_rho0;      // exact (rho0 a power of two)
  float e_hi, e_lo, ie_hi, ie_lo;  // e and 1 / e as sums of two floats
  int64_t nu;                      // nodes of the user arrays (their field stride)
};

// Whether the FP32 forms above apply.
static bool unit_map(const Geometry& g, double rho0, double e, UnitMap* m) {
  m->nu = g.n / g.nx * (g.nx - g.pad);
  m->rho0 = rho0;
  m->e = e;
  m->inv_rho0 = 1.0 / rho0;
  m->inv_e = 1.0 / e;
  m->f_rho0 = (float)rho0;
  m->f_inv_rho0 = (float)m->inv_rho0;
  m->e_hi = (float)e;
  m->e_lo = (float)(e - (double)m->e_hi);
  m->ie_hi = (float)m->inv_e;
  m->ie_lo = (float)(m->inv_e - (double)m->ie_hi);
  int x = 0;
  const bool pow2 = frexp(rho0, &x) == 0.5 && x > -60 && x < 60;
  return pow2 && e > 0x1p-60 && e < 0x1p60;
}

// v (hi + lo), rounded once; infinities and NaN as in v * hi.
__device__ __forceinline__ float mul_pair(float v, float hi, float lo) {
  const float p = __fmul_rn(v, hi);
  const float s = __fadd_rn(p, __fmaf_rn(v, lo, __fmaf_rn(v, hi, -p)));
  return s == s ? s : p;
}

// FAST: 32-bit values and the FP32 forms.
template <typename S, bool FAST>
struct Map {
  using C = typename Store<S>::C;
  template <typename T>
  __device__ __forceinline__ static S rho_in(T v, const UnitMap& m) {
    if constexpr (FAST) return Store<S>::to(__fmaf_rn(v, m.f_inv_rho0, -1.0f));
    else return Store<S>::to(C((double)v * m.inv_rho0 - 1.0));
  }
  template <typename T>
  __device__ __forceinline__ static S u_in(T v, const UnitMap& m) {
    if constexpr (FAST) return Store<S>::to(mul_pair(v, m.ie_hi, m.ie_lo));
    else return Store<S>::to(C((double)v * m.inv_e));
  }
  template <typename T>
  __device__ __forceinline__ static T rho_out(S v, const UnitMap& m) {
    if constexpr (FAST) return __fmul_rn(m.f_rho0, __fadd_rn(1.0f, Store<S>::from(v)));
    else return (T)(m.rho0 * (1.0 + (double)Store<S>::from(v)));
  }
  template <typename T>
  __device__ __forceinline__ static T u_out(S v, const UnitMap& m) {
    if constexpr (FAST) return mul_pair(Store<S>::from(v), m.e_hi, m.e_lo);
    else return (T)(m.e * (double)Store<S>::from(v));
  }
};

template <typename T>
struct alignas(2 * sizeof(T)) Two {
  T x, y;
};
template <typename S>
struct alignas(4 * sizeof(S) > 16 ? 16 : 4 * sizeof(S)) Four {
  S v[4];
};

// The kernels walk the user arrays in order (a warp touches contiguous runs of
// each user array, which may be page-locked host memory read or written over
// the host link).  kQuad2 (interleaved rows without padding, user arrays
// aligned to two values): a thread takes one storage quad, the nodes (2t,
// 2t + H, 2t + 1, 2t + 1 + H) of a row, i.e. two runs of two user values per
// field and one wide store, so a warp moves whole sectors on both sides.
// kQuad1 (padded rows or unaligned user arrays): the same quad with single user
// values, of which the one or two beyond the domain's last node do not exist.
// kNode (natural rows): a thread takes one node, at the same place on both
// sides.  I: index type (32 bits wherever the count allows, as the division by
// the row length is the largest integer cost).
enum Unit { kNode, kQuad1, kQuad2 };

// fn(storage index, user index, x of the unit's first node)
template <typename I, int U, typename Fn>
__device__ __forceinline__ void for_units(const Geometry& g, Fn&& fn) {
  const I units = (I)(U != kNode ? g.n / 4 : g.n);
  for (I k = (I)blockIdx.x * blockDim.x + threadIdx.x; k < units; k += (I)gridDim.x * blockDim.x) {
    if constexpr (U == kNode) {
      fn((int64_t)k, (int64_t)k, 0);
    } else {
      const I per_row = (I)(g.nx / 4);
      const I row = k / per_row;
      const int x = 2 * (int)(k - row * per_row);
      fn((int64_t)4 * k, (int64_t)row * (g.nx - g.pad) + x, x);
    }
  }
}

// Nodes (x, x + H, x + 1, x + 1 + H) of a user row, j the index of x; those past
// the end of a padded row read as its first node (launch_wrap_columns then puts
// the periodic images in place) and are not written.
template <int U, typename T>
__device__ __forceinline__ void ld_user(const Geometry& g, const T* p, int64_t j, int x, T (&v)[4]) {
  if constexpr (U == kQuad2) {
    const Two<T> a = *reinterpret_cast<const Two<T>*>(p + j);
    const Two<T> b = *reinterpret_cast<const Two<T>*>(p + j + g.hx);
    v[0] = a.x;
    v[1] = b.x;
    v[2] = a.y;
    v[3] = b.y;
  } else {
    const int last = g.nx - g.pad - 1 - g.hx;
    v[0] = p[j];
    v[1] = p[x <= last ? j + g.hx : j - x];
    v[2] = p[j + 1];
    v[3] = p[x + 1 <= last ? j + 1 + g.hx : j - x];
  }
}
template <int U, typename T>
__device__ __forceinline__ void st_user(const Geometry& g, T* p, int64_t j, int x, const T (&v)[4]) {
  if constexpr (U == kQuad2) {
    *reinterpret_cast<Two<T>*>(p + j) = Two<T>{v[0], v[2]};
    *reinterpret_cast<Two<T>*>(p + j + g.hx) = Two<T>{v[1], v[3]};
  } else {
    const int last = g.nx - g.pad - 1 - g.hx;
    p[j] = v[0];
    p[j + 1] = v[2];
    if (x <= last) p[j + g.hx] = v[1];
    if (x + 1 <= last) p[j + 1 + g.hx] = v[3];
  }
}

// Blocks of 256 threads for n threads' worth of units, at most 2^20 (each
// thread then takes several): a thread's few loads are all it has in flight,
// so the block scheduler, not a loop, keeps the SMs full.
static unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > (1 << 20)) b = 1 << 20;
  return (unsigned)(b < 1 ? 1 : b);
}

// 32-bit unit indices where neither the count nor a grid stride past it overflows.
static bool small_index(int64_t units) { return units < ((int64_t)1 << 31); }

static Unit unit_of(const Geometry& g, const void* a, const void* b, size_t bytes) {
  if (!g.ilv) return kNode;
  return !g.pad && (reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) % bytes == 0 ? kQuad2 : kQuad1;
}

// launch(blocks, threads, index type, std::integral_constant<int, unit>) for the unit
// and node count.  Fewer than 2^18 units go in blocks of 64 threads, so that they reach
// every SM evenly: with FP64 maps, on a pipe of two lanes an SM, 64^2 took four SMs
// (get 14.4 us whole call, 13.0 in small blocks).
template <typename Fn>
static cudaError_t by_unit(const Geometry& g, Unit unit, Fn&& launch) {
  const int64_t units = unit == kNode ? g.n : g.n / 4;
  const unsigned threads = units < (1 << 18) ? 64 : 256;
  const unsigned grid = units < (1 << 18) ? (unsigned)((units + 63) / 64) : grid_for(units);
  auto with_index = [&](auto index) {
    switch (unit) {
      case kNode: return launch(grid, threads, index, std::integral_constant<int, kNode>{});
      case kQuad1: return launch(grid, threads, index, std::integral_constant<int, kQuad1>{});
      default: return launch(grid, threads, index, std::integral_constant<int, kQuad2>{});
    }
  };
  return small_index(g.n) ? with_index(uint32_t{}) : with_index(int64_t{});
}

// Running sum of one thread: FP64 for FP64 storage; float-float (Knuth's
// two-sum, the error of every FP32 addition kept in lo) otherwise, so the
// per-node terms, formed in FP32, are added without FP64 arithmetic.
template <typename C>
struct NuAcc {
  double v = 0.0;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ double value() const { return v; }
};
template <>
struct NuAcc<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
    hi = s;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

}  // namespace maclab
