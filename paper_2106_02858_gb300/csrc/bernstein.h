// The Bernstein form of the degree-q polynomials on a tetrahedron, the basis of the field vectors
// inside an FP64 handle (FP32 handles hold nodal values): coefficient c_b of B_b = q! / (b0! b1! b2! b3!) l0^b0 l1^b1 l2^b2 l3^b3
// sits at the place of the equispaced node b / q (lattice_index order), so faces, permutations
// and neighbour codes are those of the nodes.  In this basis the operators of the DG scheme are
// sparse (for the nodal values they are dense):
//   * a derivative lowers the degree by differences, (d_k F)_a = q (c_{a + e_k} - c_{a + e_0}) for
//     |a| = q - 1, and raising the degree back adds ((a_i + 1) / q) of it to coefficient a + e_i;
//   * the lift of a flux g on face f, M^{-1} times the face mass, is a face-local product
//     h_b = sum_i (b_i + 1)^2 g_b + sum_{i != j} (b_i + 1) b_j g_{b + e_i - e_j} on the face's own
//     coefficients, and on the layer b_f = j behind it (-1)^j C(q, j) / (j + 1) times the j-fold
//     degree reduction of h, (r)_a = sum_i ((a_i + 1) / (q - j)) h_{a + e_i} per step;
//   * the mass matrix is a sum of squares, M = s sum_g X_g X_g^T over all |g| <= q with
//     X_g(c) = sum_b prod_i C(b_i, g_i) c_b, s = (q!)^2 / (2q + 3)!: X of degree q is c itself, and
//     each lower degree is one contraction, X_g = (1 / k) sum_i (g_i + 1) X_{g + e_i} with k = q - |g|.
// (Section 5.2.2, Eq. DG_semidiscrete / ode_system; identities of the Bernstein basis, e.g. Chan and Warburton, "GPU-accelerated Bernstein-Bezier discontinuous Galerkin methods for
// wave problems", SIAM J. Sci. Comput. 39 (2017).)  All weights are small integers or rationals.
#pragma once

#include "common.h"

namespace cmcg {

struct Bary4 {
  int b[4];
};
// Barycentric indices of node n of the order-q lattice (inverse of lattice_index).
constexpr Bary4 bary_of(int q, int n) {
  int m = 0;
  for (int k = 0; k <= q; ++k)
    for (int j = 0; j <= q - k; ++j)
      for (int i = 0; i <= q - k - j; ++i, ++m)
        if (m == n) return Bary4{{q - i - j - k, i, j, k}};
  return Bary4{{0, 0, 0, 0}};
}
constexpr int node_at(int q, const Bary4& x) { return lattice_index(q, x.b[1], x.b[2], x.b[3]); }
// Index of face-local lattice point (w0, w1, w2) of degree q (w2 outermost, w1 fastest).
constexpr int face_index(int q, int w1, int w2) {
  int idx = 0;
  for (int k = 0; k < w2; ++k) idx += q - k + 1;
  return idx + w1;
}
struct Bary3 {
  int b[3];
};
constexpr Bary3 face_bary_of(int q, int n) {
  int m = 0;
  for (int w2 = 0; w2 <= q; ++w2)
    for (int w1 = 0; w1 <= q - w2; ++w1, ++m)
      if (m == n) return Bary3{{q - w1 - w2, w1, w2}};
  return Bary3{{0, 0, 0}};
}

// Index tables of order Q, used with compile-time indices only.
template <int Q>
struct BernTab {
  static constexpr int NA = np_of(Q - 1);  // coefficients of degree Q - 1
  int up[NA][4];                           // coefficient a + e_i
  int upw[NA][4];                          // a_i + 1
  int face[4][nfp_of(Q)];                  // volume index of face-local coefficient
  int l0[nfp_of(Q)][nfp_of(Q)];            // the face-local product h = l0 g, less the common term:
  bool in_sum[nfp_of(Q)];                  // rows of this set all hold the sum of g over the set (P1: all
                                           // face coefficients, P2: the edge coefficients), added once
  int red[Q + 1][nfp_of(Q)][3];            // [j][a][i]: index (degree Q - j + 1) of a + e_i; weight a_i + 1 below
  int redw[Q + 1][nfp_of(Q)][3];
  int layer[4][Q + 1][nfp_of(Q)];          // [f][j][a]: volume index of layer j's coefficient a (|a| = Q - j)
};
template <int Q>
constexpr BernTab<Q> make_bern() {
  BernTab<Q> t{};
  for (int m = 0; m < BernTab<Q>::NA; ++m) {
    const Bary4 a = bary_of(Q - 1, m);
    for (int i = 0; i < 4; ++i) {
      Bary4 u = a;
      u.b[i] += 1;
      t.up[m][i] = node_at(Q, u);
      t.upw[m][i] = a.b[i] + 1;
    }
  }
  for (int n = 0; n < nfp_of(Q); ++n) {
    const Bary3 w = face_bary_of(Q, n);
    int d = 0;
    for (int i = 0; i < 3; ++i) d += (w.b[i] + 1) * (w.b[i] + 1);
    t.l0[n][n] = d;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        if (i == j || w.b[j] == 0) continue;
        Bary3 u = w;
        u.b[i] += 1;
        u.b[j] -= 1;
        t.l0[n][face_index(Q, u.b[1], u.b[2])] = (w.b[i] + 1) * w.b[j];
      }
  }
  for (int n = 0; n < nfp_of(Q); ++n) {
    const Bary3 w = face_bary_of(Q, n);
    t.in_sum[n] = Q == 1 || (Q == 2 && w.b[0] * w.b[1] + w.b[0] * w.b[2] + w.b[1] * w.b[2] > 0);
  }
  for (int n = 0; n < nfp_of(Q); ++n)
    for (int m = 0; m < nfp_of(Q); ++m)
      if (t.in_sum[n] && t.in_sum[m]) t.l0[n][m] -= 1;
  for (int f = 0; f < 4; ++f)
    for (int j = 0; j <= Q; ++j)
      for (int n = 0; n < nfp_of(Q - j); ++n) {
        const Bary3 w = face_bary_of(Q - j, n);
        Bary4 x{{0, 0, 0, 0}};
        x.b[f] = j;
        for (int s = 0; s < 3; ++s) x.b[FACE_VERTS[f][s]] = w.b[s];
        t.layer[f][j][n] = node_at(Q, x);
        if (j == 0) t.face[f][n] = t.layer[f][0][n];
        if (f == 0 && j > 0)
          for (int i = 0; i < 3; ++i) {
            Bary3 u = w;
            u.b[i] += 1;
            t.red[j][n][i] = face_index(Q - j + 1, u.b[1], u.b[2]);
            t.redw[j][n][i] = w.b[i] + 1;
          }
      }
  return t;
}
// Factor of layer j's unnormalised reductions: (-1)^j C(Q, j) / (j + 1) / (Q (Q - 1) ... (Q - j + 1))
// = (-1)^j / (j + 1)!.
constexpr double layer_weight(int j) {
  double w = 1.0;
  for (int k = 2; k <= j + 1; ++k) w /= k;
  return (j & 1) ? -w : w;
}

// Coefficients <-> values at the nodes.  A node whose barycentric indices have one, two or three
// nonzeros depends on the coefficients of its vertex, edge or face only; the tables hold the
// nonzero weights of the (unit lower-dimensional) Bernstein values and of their inverse.
struct BasisTab {
  int n;              // entries
  int col[10];
  double w[10];
};
constexpr double bern_value(int q, const Bary4& x, const Bary4& a) {  // B_a at the node x / q
  double v = 1;
  int k = 0;
  for (int i = 0; i < 4; ++i)
    for (int r = 1; r <= a.b[i]; ++r) {
      ++k;
      v = v * (double(k) * x.b[i]) / (double(r) * q);
    }
  return v;
}
constexpr BasisTab to_node_row(int q, int n) {
  BasisTab t{};
  const Bary4 x = bary_of(q, n);
  for (int m = 0; m < np_of(q); ++m) {
    const double v = bern_value(q, x, bary_of(q, m));
    if (v != 0) {
      t.col[t.n] = m;
      t.w[t.n++] = v;
    }
  }
  return t;
}
// Row n of the inverse: vertices are their values; an edge coefficient follows from its edge's
// values (q = 2: 2 u1 - (u0 + u2) / 2; q = 3: (-5 u0 + 18 u1 - 9 u2 + 2 u3) / 6), the face
// coefficient of q = 3 from its face's ((27 u_c + 2 sum_v u - (9 / 2) sum_e u) / 6).
constexpr BasisTab to_bern_row(int q, int n) {
  BasisTab t{};
  const Bary4 x = bary_of(q, n);
  int nz = 0;
  for (int i = 0; i < 4; ++i) nz += x.b[i] != 0;
  for (int m = 0; m < np_of(q); ++m) {
    const Bary4 a = bary_of(q, m);
    bool in = true;  // a lies on the vertex / edge / face of x
    int nza = 0;
    for (int i = 0; i < 4; ++i) {
      if (a.b[i] != 0 && x.b[i] == 0) in = false;
      nza += a.b[i] != 0;
    }
    if (!in) continue;
    double w = 0;
    if (nz == 1) w = 1;
    else if (nz == 2) {
      int d = 0;  // lattice distance of a from x along the edge, towards x's nearer vertex first
      int big = -1;
      for (int i = 0; i < 4; ++i)
        if (x.b[i] != 0 && (big < 0 || x.b[i] > x.b[big])) big = i;
      d = a.b[big];
      if (q == 2) w = d == 1 ? 2.0 : -0.5;
      else w = d == 3 ? -5.0 / 6 : d == 2 ? 3.0 : d == 1 ? -1.5 : 1.0 / 3;
    } else {
      w = nza == 3 ? 4.5 : nza == 1 ? 1.0 / 3 : -0.75;
    }
    t.col[t.n] = m;
    t.w[t.n++] = w;
  }
  return t;
}
template <int Q>
struct BasisRows {
  BasisTab r[np_of(Q)];
};
template <int Q>
constexpr BasisRows<Q> make_to_node() {
  BasisRows<Q> t{};
  for (int n = 0; n < np_of(Q); ++n) t.r[n] = to_node_row(Q, n);
  return t;
}
template <int Q>
constexpr BasisRows<Q> make_to_bern() {
  BasisRows<Q> t{};
  for (int n = 0; n < np_of(Q); ++n) t.r[n] = to_bern_row(Q, n);
  return t;
}

// Layout of a field vector.  A half tile is 16 tetrahedra, a row of 32 values the coefficient n of
// component c of their electric (even) and magnetic (odd) fields: one thread pair per tetrahedron
// reads a row as one 128-byte line (FP32).
constexpr int HTILE = 16;
__host__ __device__ constexpr int64_t field_at(int np, int64_t i, int field, int c, int n) {
  return (i >> 4) * int64_t(96) * np + (c * np + n) * 32 + 2 * int(i & 15) + field;
}

}  // namespace cmcg
