// d2q9.cuh -- the D2Q9 update (Eqs. (2), (4), (5)) factored by rows.
//
// The D2Q9 weights are the product of the weights (1, 4, 1) / 6 of the two
// axes, so the nine terms w36_a T_a of a node need not be formed and summed one
// by one.  With T_a = A + c.B + sum_i c_i^2 P_ii + c_x c_y P_xy (step_tiled.cuh)
// a source node sends along x only
//   a = A, S + B_x, S - B_x      (c_x = 0, +1, -1; S = A + P_xx),
//   b = B_y, B_y + P_xy, B_y - P_xy    and    e = P_yy,
// of which T = a + c_y b + c_y^2 e.  A row's sums over the sources x, x - 1, x + 1
//   P, P1: weights (4, 1, 1) and c_x of a;  Q, Q1 of b;  E, E1 of e
// give what the row adds to the row c_y away (weight 4 for c_y = 0, else 1):
//   R (36 drho'):  c_y = 0: 4 P          c_y = +-1: G+- = (P + E) +- Q
//   M_x:                    4 P1                    H+- = (P1 + E1) +- Q1
//   M_y:                    0                       +- G+-
// 34 operations a node (14 per source, 15 per row sum, 5 to add three rows)
// where the nine terms took 47, and only two values, not three, cross from row
// to row, without a shift in x.  Every kernel of the lattice sums in the order
// written here (rows y - 1, y, y + 1), so they agree bit for bit.  The constants
// that multiply first-order quantities (3, 3/2, 1/2, 4) are exact.
#pragma once
#include "step_tiled.cuh"

namespace maclab {

// What one node pair sends along its row.
template <typename C>
struct D9Node {
  using P = typename Pair<C>::P;
  P A, by, e;            // c_x = 0
  P ap, bp, am, bm;      // c_x = +1, c_x = -1 (e as above)
};

template <typename C>
__device__ __forceinline__ D9Node<C> d9_node(typename Pair<C>::P r, typename Pair<C>::P u, typename Pair<C>::P v) {
  using O = Pair<C>;
  using P = typename O::P;
  D9Node<C> n;
  const P g = O::fma(r, O::splat(C(3)), O::splat(C(3)));  // 3 rho
  // products that enter sums: never contracted, so that every kernel rounds alike
  const P bx = O::mul_exact(g, u);
  n.by = O::mul_exact(g, v);
  const P qx = O::mul(bx, u), qy = O::mul(n.by, v);  // 3 rho u_i^2
  n.A = O::fma(O::fma(n.by, v, qx), O::splat(C(-0.5)), r);
  n.e = O::mul_exact(qy, O::splat(C(1.5)));
  const P S = O::fma(qx, O::splat(C(1.5)), n.A);
  const P c = O::mul(bx, v);  // 3 rho u_x u_y
  n.ap = O::add(S, bx);
  n.am = O::sub(S, bx);
  n.bp = O::fma(c, O::splat(C(3)), n.by);
  n.bm = O::fma(c, O::splat(C(-3)), n.by);
  return n;
}

// What a row adds at one x: to its own row (p, p1), the row above (gp, hp) and
// the row below (gm, hm).
template <typename C>
struct D9Row {
  using P = typename Pair<C>::P;
  P p, p1, gp, hp, gm, hm;
};

// own: the node; (apl, bpl, el) of the node at x - 1, (amr, bmr, er) at x + 1.
template <typename C>
__device__ __forceinline__ D9Row<C> d9_row(typename Pair<C>::P A, typename Pair<C>::P by, typename Pair<C>::P e,
                                           typename Pair<C>::P apl, typename Pair<C>::P bpl, typename Pair<C>::P el,
                                           typename Pair<C>::P amr, typename Pair<C>::P bmr, typename Pair<C>::P er) {
  using O = Pair<C>;
  using P = typename O::P;
  const P four = O::splat(C(4));
  D9Row<C> w;
  w.p = O::fma(A, four, O::add(apl, amr));
  w.p1 = O::sub(apl, amr);
  const P q = O::fma(by, four, O::add(bpl, bmr)), q1 = O::sub(bpl, bmr);
  const P U = O::add(w.p, O::fma(e, four, O::add(el, er)));
  const P V = O::add(w.p1, O::sub(el, er));
  w.gp = O::add(U, q);
  w.gm = O::sub(U, q);
  w.hp = O::add(V, q1);
  w.hm = O::sub(V, q1);
  return w;
}

// Sums (36 drho', 36 m_x, 36 m_y) of a destination row as its sources arrive:
// begin with what the row below sent (gp, hp), add the row itself, then the row above.
template <typename C>
__device__ __forceinline__ void d9_own(typename Pair<C>::P (&s)[3], typename Pair<C>::P gp, typename Pair<C>::P hp,
                                       const D9Row<C>& w) {
  using O = Pair<C>;
  s[0] = O::fma(w.p, O::splat(C(4)), gp);
  s[1] = O::fma(w.p1, O::splat(C(4)), hp);
  s[2] = gp;
}
template <typename C>
__device__ __forceinline__ void d9_above(typename Pair<C>::P (&s)[3], typename Pair<C>::P gm, typename Pair<C>::P hm) {
  using O = Pair<C>;
  s[0] = O::add(s[0], gm);
  s[1] = O::add(s[1], hm);
  s[2] = O::sub(s[2], gm);
}

// The new state from the sums (Eq. (5): u' = M / (36 + R) + F).
template <typename C>
__device__ __forceinline__ void d9_state(const typename Pair<C>::P (&s)[3], const typename Pair<C>::P (&force)[2],
                                         typename Pair<C>::P (&v)[3]) {
  using O = Pair<C>;
  const typename O::P inv = O::rcp(O::add(O::splat(C(36)), s[0]));
  v[0] = O::mul(s[0], O::splat(C(1.0 / 36.0)));
  v[1] = O::fma(s[1], inv, force[0]);
  v[2] = O::fma(s[2], inv, force[1]);
}

// A lane's quad of a row: pairs a = (2t, 2t + H) and b = (2t + 1, 2t + 1 + H).
// The left neighbour of pair a is the previous lane's pair b, the right one of
// pair b the next lane's pair a; left(v) and right(v) give those lanes' v.
template <typename C, typename Left, typename Right>
__device__ __forceinline__ void d9_quad(const typename Pair<C>::P (&st)[3][2], D9Row<C> (&w)[2], Left&& left,
                                        Right&& right) {
  const D9Node<C> a = d9_node<C>(st[0][0], st[1][0], st[2][0]);
  const D9Node<C> b = d9_node<C>(st[0][1], st[1][1], st[2][1]);
  w[0] = d9_row<C>(a.A, a.by, a.e, left(b.ap, 0), left(b.bp, 1), left(b.e, 2), b.am, b.bm, b.e);
  w[1] = d9_row<C>(b.A, b.by, b.e, a.ap, a.bp, a.e, right(a.am, 0), right(a.bm, 1), right(a.e, 2));
}

// The tiled kernel's row: see its declaration.
template <typename C, int MODE, int BXC>
__device__ __forceinline__ void row_update_2d(const typename Pair<C>::P (&st)[3][2], typename Pair<C>::P (&ap)[2][3],
                                              typename Pair<C>::P (&ac)[2][3], typename Pair<C>::P (&an)[2][3],
                                              const SmemBase<typename Pair<C>::P>& sb, bool active) {
  using O = Pair<C>;
  using P = typename O::P;
  constexpr int XS = Cols<BXC>::W;  // stride between slots
  if (active) {
    const D9Node<C> a = d9_node<C>(st[0][0], st[1][0], st[2][0]);
    const D9Node<C> b = d9_node<C>(st[0][1], st[1][1], st[2][1]);
    const P to_r[3] = {b.ap, b.bp, b.e}, to_l[3] = {a.am, a.bm, a.e};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sb.x_own[k * XS] = to_r[k];
      if (sb.wl) sb.x_sl[k * XS] = O::swap(to_r[k]);
      sb.x_own[(3 + k) * XS] = to_l[k];
      if (sb.wr) sb.x_sr[(3 + k) * XS] = O::swap(to_l[k]);
    }
  }
  __syncthreads();
  if (active) {
    D9Row<C> w[2];
    d9_quad<C>(st, w, [&](P, int k) { return sb.x_l[k * XS]; }, [&](P, int k) { return sb.x_r[(3 + k) * XS]; });
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if constexpr (MODE != kFirst) d9_above<C>(ap[q], w[q].gm, w[q].hm);
      if constexpr (MODE == kMid) d9_own<C>(ac[q], ac[q][0], ac[q][1], w[q]);
      if constexpr (MODE != kLast) {
        an[q][0] = an[q][2] = w[q].gp;
        an[q][1] = w[q].hp;
      }
    }
  }
  __syncthreads();  // the row's slots are the next row's (one buffer, whatever the planes use)
}

}  // namespace maclab
