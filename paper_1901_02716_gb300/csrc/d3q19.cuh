// d3q19.cuh -- the D3Q19 update (Eqs. (2), (4), (5)) factored by rows and planes.
//
// With T_a = A + c.B + sum_i c_i^2 P_ii + sum_{i<j} c_i c_j P_ij (step_tiled.cuh)
// and the integer weights 36 w = 12 (rest), 2 (axes), 1 (edges), the nineteen terms
// need not be formed and summed one by one.  A source node sends along x
//   a+- = S +- B_x (S = A + P_xx),  b+- = B_y +- P_xy,  d+- = B_z +- P_xz,
//   e = P_yy,  f = P_zz,
// five values each way.  With L, R its row neighbours' values and own ones for
// c_x = 0, a row sums at each x (weights 2 for c_x = 0, 1 else; `1` marks sums with c_x)
//   sA = a+L + a-R, dA = a+L - a-R, and likewise of b, d, e, f,
//   U = 2 (A + e) + sA + sE,  Q = 2 B_y + sB,  V = dA + dE,  Q1 = dB,
//   W = 2 (A + f) + sA + sF,  D = 2 B_z + sD,  X = dA + dF,  D1 = dD,
// which give all that moves within the plane x, y and the plane x, z:
//   to its own row and plane      R: 12 A + 2 sA      M_x: 2 dA
//   to the row c_y away           R: G = U + c_y Q    M_x: H = V + c_y Q1    M_y: c_y G
//   to the plane c_z away         R: K = W + c_z D    M_x: X + c_z D1        M_z: c_z K
// The four edges of the plane y, z are single terms,
//   T(c_y, c_z) = (A + e + f + c_y B_y) + c_z (B_z + c_y P_yz)   R, M_y: c_y, M_z: c_z.
// So four values (G, H, T of c_z = +1 and -1) cross from row to row, without a
// shift in x, and what a plane sends on has M_z = +-R: between planes a march
// carries three sums for the plane it has just sent to (R, M_x, M_y) and four for
// the plane before it.  79 operations a node where forming and summing the
// nineteen terms took 106, and 7 sums held where it took 12.
// Every sum adds its own row first, then the row below, then the row above, so
// results do not depend on how rows and planes are dealt to threads.
#pragma once
#include "step_tiled.cuh"

namespace maclab {

// What one node pair sends.  NU: the terms of the viscosity mode, g_a / w_a =
// drho + rho (3/2 u.u - 9/2 (c.u)^2), i.e. T_a without B and with P negated.
template <typename C>
struct D3Node {
  using P = typename Pair<C>::P;
  P A, by, bz, e, f, Ae, Af;  // Ae = A + e, Af = A + f
  P ap, bp, dp;          // c_x = +1
  P am, bm, dm;          // c_x = -1
  P tpp, tpm, tmp, tmm;  // T(c_y, c_z) for c_x = 0
};

template <typename C, bool NU>
__device__ __forceinline__ D3Node<C> d3_node(typename Pair<C>::P r, typename Pair<C>::P u, typename Pair<C>::P v,
                                             typename Pair<C>::P w) {
  using O = Pair<C>;
  using P = typename O::P;
  D3Node<C> n;
  const P g = O::fma(r, O::splat(C(3)), O::splat(C(3)));  // 3 rho
  // products that enter sums: never contracted, so that every instance rounds alike
  const P bx = O::mul_exact(g, u), by = O::mul_exact(g, v), bz = O::mul_exact(g, w);
  const P qx = O::mul(bx, u), qy = O::mul(by, v), qz = O::mul(bz, w);  // 3 rho u_i^2
  const P cxy = O::mul(bx, v), cxz = O::mul(bx, w), cyz = O::mul(by, w);
  constexpr C s = NU ? C(-1) : C(1);
  n.A = O::fma(O::fma(bz, w, O::fma(by, v, qx)), O::splat(s * C(-0.5)), r);
  const P S = O::fma(qx, O::splat(s * C(1.5)), n.A);
  n.e = O::mul_exact(qy, O::splat(s * C(1.5)));
  n.f = O::mul_exact(qz, O::splat(s * C(1.5)));
  n.Ae = O::fma(qy, O::splat(s * C(1.5)), n.A);
  n.Af = O::fma(qz, O::splat(s * C(1.5)), n.A);
  const P h = O::fma(qz, O::splat(s * C(1.5)), n.Ae);
  const P p3 = O::splat(s * C(3)), m3 = O::splat(s * C(-3));
  if constexpr (NU) {
    n.ap = n.am = S;
    n.by = n.bz = O::splat(C(0));
    n.bp = O::mul_exact(cxy, p3);
    n.bm = O::mul_exact(cxy, m3);
    n.dp = O::mul_exact(cxz, p3);
    n.dm = O::mul_exact(cxz, m3);
    n.tpp = n.tmm = O::fma(cyz, p3, h);
    n.tpm = n.tmp = O::fma(cyz, m3, h);
  } else {
    n.ap = O::add(S, bx);
    n.am = O::sub(S, bx);
    n.by = by;
    n.bz = bz;
    n.bp = O::fma(cxy, p3, by);
    n.bm = O::fma(cxy, m3, by);
    n.dp = O::fma(cxz, p3, bz);
    n.dm = O::fma(cxz, m3, bz);
    const P hp = O::add(h, by), hm = O::sub(h, by);
    const P kp = O::fma(cyz, p3, bz), km = O::fma(cyz, m3, bz);
    n.tpp = O::add(hp, kp);
    n.tpm = O::sub(hp, kp);
    n.tmp = O::add(hm, km);
    n.tmm = O::sub(hm, km);
  }
  return n;
}

// The row's sums at one x.
template <typename C>
struct D3Row {
  using P = typename Pair<C>::P;
  P sA, dA;              // own row and plane (with A)
  P gp, hp, gm, hm;      // rows above and below
  P kp, xp, km, xm;      // planes above and below
};

// l: the node pair at x - 1, r: at x + 1 (of each only what moves this way is read)
template <typename C, bool NU>
__device__ __forceinline__ D3Row<C> d3_row(const D3Node<C>& n, const D3Node<C>& l, const D3Node<C>& r) {
  using O = Pair<C>;
  using P = typename O::P;
  const P two = O::splat(C(2));
  D3Row<C> w;
  w.sA = O::add(l.ap, r.am);
  w.dA = O::sub(l.ap, r.am);
  P Q = O::add(l.bp, r.bm), D = O::add(l.dp, r.dm);
  if constexpr (!NU) {
    Q = O::fma(n.by, two, Q);
    D = O::fma(n.bz, two, D);
  }
  const P Q1 = O::sub(l.bp, r.bm), D1 = O::sub(l.dp, r.dm);
  const P U = O::add(O::fma(n.Ae, two, w.sA), O::add(l.e, r.e));
  const P W = O::add(O::fma(n.Af, two, w.sA), O::add(l.f, r.f));
  const P V = O::add(w.dA, O::sub(l.e, r.e));
  const P X = O::add(w.dA, O::sub(l.f, r.f));
  w.gp = O::add(U, Q);
  w.gm = O::sub(U, Q);
  w.hp = O::add(V, Q1);
  w.hm = O::sub(V, Q1);
  w.kp = O::add(W, D);
  w.km = O::sub(W, D);
  w.xp = O::add(X, D1);
  w.xm = O::sub(X, D1);
  return w;
}

}  // namespace maclab
