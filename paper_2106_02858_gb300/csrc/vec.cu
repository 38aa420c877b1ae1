// Vector kernels of the CMCG outer loop (Section 2.2, Algorithm cmcg):
// conversion between the boundary layout [tet][comp][node] (nodal values, double) and
// the handle's fields (field_at; nodal values in FP32, Bernstein coefficients in FP64),
// fused CG updates, and the
// (eps, mu)-weighted inner product (Eq. innerproduct)
//     (X, Y) = sum_K |det A_K| sum_c w_c sum_ij X_c[i] Mref[i][j] Y_c[j],
// w_c = eps_K on E rows, mu_K on H rows, accumulated in FP64 whatever the
// storage precision.  Reductions are deterministic: one partial per block
// (warp shuffles, then shared memory in a fixed order) and one finalising
// block that sums the partials in a fixed order.
#include "bernstein.h"

namespace cmcg {
namespace {

// One warp converts one component of a half tile: lane 2t + f takes field f of tetrahedron t, its
// nodes being contiguous in the boundary arrays.  x0, x1: the arrays of the two fields, at
// [tet * stride + c * Np] (x1 null: zeros).
template <int Q, typename R>
__global__ void __launch_bounds__(128) to_internal_kernel(const double* x0, const double* x1, int64_t stride, R* in,
                                                          const int32_t* e_of_i, int64_t nti, const double* per_tet) {
  constexpr int NP = np_of(Q);
  constexpr BasisRows<Q> T = make_to_bern<Q>();
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t ht = w / 3;
  const int c = int(w % 3), l = threadIdx.x & 31;
  if (ht * HTILE >= nti) return;
  const int32_t e = e_of_i[ht * HTILE + (l >> 1)];
  const double* x = (l & 1) ? x1 : x0;
  double u[NP];
#pragma unroll
  for (int n = 0; n < NP; ++n) u[n] = 0;
  if (e >= 0 && x) {
    x += e * stride + c * NP;
    const double s = per_tet ? per_tet[e] : 1.0;
#pragma unroll
    for (int n = 0; n < NP; ++n) u[n] = x[n] * s;
  }
  R* o = in + ht * (96 * NP) + c * NP * 32 + l;
#pragma unroll
  for (int n = 0; n < NP; ++n) {
    double v = u[n];
    if constexpr (sizeof(R) == 8) {
      v = T.r[n].w[0] * u[T.r[n].col[0]];
#pragma unroll
      for (int k = 1; k < 10; ++k)
        if (k < T.r[n].n) v = fma(T.r[n].w[k], u[T.r[n].col[k]], v);
    }
    o[n * 32] = R(v);
  }
}

template <int Q, typename R>
__global__ void __launch_bounds__(128) to_external_kernel(const R* in, double* x0, double* x1, int64_t stride,
                                                          const int32_t* e_of_i, int64_t nti) {
  constexpr int NP = np_of(Q);
  constexpr BasisRows<Q> T = make_to_node<Q>();
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t ht = w / 3;
  const int c = int(w % 3), l = threadIdx.x & 31;
  if (ht * HTILE >= nti) return;
  const int32_t e = e_of_i[ht * HTILE + (l >> 1)];
  double u[NP];
#pragma unroll
  for (int n = 0; n < NP; ++n) u[n] = double(in[ht * (96 * NP) + (c * NP + n) * 32 + l]);
  if (e < 0) return;
  double* x = ((l & 1) ? x1 : x0) + e * stride + c * NP;
#pragma unroll
  for (int n = 0; n < NP; ++n) {
    double v = u[n];
    if constexpr (sizeof(R) == 8) {
      v = T.r[n].w[0] * u[T.r[n].col[0]];
#pragma unroll
      for (int k = 1; k < 10; ++k)
        if (k < T.r[n].n) v = fma(T.r[n].w[k], u[T.r[n].col[k]], v);
    }
    x[n] = v;
  }
}

// o = a x + b y on the tiles of the problems with mask[p] != 0 (problem of tile t: tprob[t], or 0).
template <typename R>
__global__ void lincomb_masked_kernel(R* o1, R* o2, R* o3, double a, const R* x, double b, const R* y, int64_t n,
                                      int64_t tile_len, const int32_t* tprob, const int32_t* mask) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = tprob ? tprob[i / tile_len] : 0;
    if (!mask[p]) continue;
    double v = a * double(x[i]);
    if (y) v += b * double(y[i]);
    const R r = R(v);
    if (o1) o1[i] = r;
    if (o2) o2[i] = r;
    if (o3) o3[i] = r;
  }
}

template <typename R>
__global__ void lincomb_kernel(R* o1, R* o2, R* o3, double a, const R* x, double b, const R* y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double v = a * double(x[i]);
    if (y) v += b * double(y[i]);
    const R r = R(v);
    if (o1) o1[i] = r;
    if (o2) o2[i] = r;
    if (o3) o3[i] = r;
  }
}

// The element inner product on nodal values (FP32 fields): s_c = sum_i x_i (sum_j M_ij y_j), FP64.
__constant__ double cM1[4 * 4];
__constant__ double cM2[10 * 10];
__constant__ double cM3[20 * 20];

template <int Q>
__device__ __forceinline__ double cM(int idx) {
  if constexpr (Q == 1) return cM1[idx];
  else if constexpr (Q == 2) return cM2[idx];
  else return cM3[idx];
}
template <int Q>
__device__ __forceinline__ double nodal_dot(const double (&x)[np_of(Q)], const double (&y)[np_of(Q)]) {
  constexpr int NP = np_of(Q);
  double s = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double t = 0;
#pragma unroll
    for (int j = 0; j < NP; ++j) t = fma(cM<Q>(i * NP + j), y[j], t);
    s = fma(x[i], t, s);
  }
  return s;
}

// The element inner product on Bernstein coefficients (FP64 fields) as a sum of squares (bernstein.h): x^T M y = s sum_g X_g Y_g over the
// degree-q coefficients and their contractions to every lower degree.  At GB300's FP64 rate the
// operations bound these kernels: 60 contractions per vector and 35 products per pair at P3 (20 and
// 15 at P2) where the dense mass matrix takes 420 (110).
template <int Q>
struct MassTab {
  int dn[Q + 1][np_of(Q)][4];  // [k][g][i]: index of g + e_i in degree Q - k + 1, |g| = Q - k
  int w[Q + 1][np_of(Q)][4];   // g_i + 1
};
template <int Q>
constexpr MassTab<Q> make_mass() {
  MassTab<Q> t{};
  for (int k = 1; k <= Q; ++k)
    for (int m = 0; m < np_of(Q - k); ++m)
      for (int i = 0; i < 4; ++i) {
        Bary4 g = bary_of(Q - k, m);
        g.b[i] += 1;
        t.dn[k][m][i] = node_at(Q - k + 1, g);
        t.w[k][m][i] = g.b[i];
      }
  return t;
}
constexpr double mass_scale(int q) { return q == 1 ? 1.0 / 120 : q == 2 ? 1.0 / 1260 : 1.0 / 10080; }

// x becomes its contraction to degree Q - k (x k!: the contractions are kept unnormalised).
template <int Q, int K>
__device__ __forceinline__ void contract(double (&x)[np_of(Q)]) {
  constexpr MassTab<Q> T = make_mass<Q>();
  double r[np_of(Q - K)];
#pragma unroll
  for (int m = 0; m < np_of(Q - K); ++m) {
    double v = T.w[K][m][0] == 1 ? x[T.dn[K][m][0]] : T.w[K][m][0] * x[T.dn[K][m][0]];
#pragma unroll
    for (int i = 1; i < 4; ++i) v = fma(double(T.w[K][m][i]), x[T.dn[K][m][i]], v);
    r[m] = v;
  }
#pragma unroll
  for (int m = 0; m < np_of(Q - K); ++m) x[m] = r[m];
}
// xx += sum_g (x_g / k!)^2 over this degree and all lower ones (XX), xy the same with x_g y_g (XY).
template <int Q, int K, bool XX, bool XY>
__device__ __forceinline__ void mass_levels(double (&x)[np_of(Q)], double (&y)[np_of(Q)], double& xx, double& xy) {
  if constexpr (K > 0) {
    contract<Q, K>(x);
    if constexpr (XY) contract<Q, K>(y);
  }
  constexpr int f = K == 2 ? 2 : K == 3 ? 6 : 1;  // K!
  double a = 0, b = 0;
#pragma unroll
  for (int m = 0; m < np_of(Q - K); ++m) {
    if constexpr (XX) a = fma(x[m], x[m], a);
    if constexpr (XY) b = fma(x[m], y[m], b);
  }
  if constexpr (XX) xx = fma(a, 1.0 / (f * f), xx);
  if constexpr (XY) xy = fma(b, 1.0 / (f * f), xy);
  if constexpr (K < Q) mass_levels<Q, K + 1, XX, XY>(x, y, xx, xy);
}

// Block b of the table covers its tetrahedra in order, two threads each: the thread's internal
// tetrahedron, or -1 when past the block's range.
__device__ __forceinline__ int64_t block_tet(const BlockTable& bt) {
  const int b = blockIdx.x, k = threadIdx.x >> 1;
  if (k >= bt.ntet[b]) return -1;
  const int64_t t = bt.tet0[b] + k;
  return int64_t(bt.half_at[t >> 4]) * HTILE + (t & 15);
}

// Sum over the block of the odd threads' values: a warp's shuffle tree over 32 consecutive
// tetrahedra, then the four warps' sums in order (valid in thread 0).
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double tet[DOT_TETS];
  __shared__ double sh[DOT_TETS / 32];
  __syncthreads();  // a previous call's reads are done
  if (threadIdx.x & 1) tet[threadIdx.x >> 1] = v;
  __syncthreads();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (w < DOT_TETS / 32) {
    double x = tet[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (l == 0) sh[w] = x;
  }
  __syncthreads();
  double s = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < DOT_TETS / 32; ++i) s += sh[i];
  return s;
}

// The tetrahedron's products xx = (x, x) and xy = (x, y), valid in the odd thread; `load(c, x, y)`
// loads component c of the thread's field.  FP32 fields keep one chain over the six components: the
// odd thread goes on from the even thread's sum over E.
template <int Q, typename R, bool XX, bool XY, typename Load>
__device__ __forceinline__ void tet_dots(bool live, double w, double& xx, double& xy, Load&& load) {
  constexpr int NP = np_of(Q);
  double px[3] = {0, 0, 0}, py[3] = {0, 0, 0};
  if (live)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double x[NP], y[NP];
      load(c, x, y);
      if constexpr (sizeof(R) == 8) {
        mass_levels<Q, 0, XX, XY>(x, y, px[c], py[c]);
      } else {
        if constexpr (XY) py[c] = nodal_dot<Q>(x, y);
        if constexpr (XX) px[c] = nodal_dot<Q>(x, x);
      }
    }
  if constexpr (sizeof(R) == 8) w *= mass_scale(Q);
  auto chain = [&](const double (&p)[3]) {
    double s = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) s = fma(w, p[c], s);
    const double e = __shfl_xor_sync(0xffffffffu, s, 1);
    if (threadIdx.x & 1) {
      s = e;
#pragma unroll
      for (int c = 0; c < 3; ++c) s = fma(w, p[c], s);
    }
    return s;
  };
  if constexpr (XX) xx = chain(px);
  if constexpr (XY) xy = chain(py);
}

// A = Uw - WT; partials (D, A) and (D, D).
template <int Q, typename R>
__global__ void __launch_bounds__(DOT_THREADS) cg_after_adjoint_kernel(const R* Uw, const R* WT, R* A, const R* D,
                                                                      const double* wdot, double* partials,
                                                                      const BlockTable bt, const int32_t* pactive) {
  constexpr int NP = np_of(Q);
  const bool act = !pactive || pactive[bt.prob[blockIdx.x]];
  const int64_t t = block_tet(bt);
  const bool live = act && t >= 0;
  const int64_t o = live ? field_at(NP, t, threadIdx.x & 1, 0, 0) : 0;
  double da = 0, dd = 0;
  tet_dots<Q, R, true, true>(live, live ? wdot[2 * t + (threadIdx.x & 1)] : 0.0, dd, da,
                       [&](int c, double (&x)[NP], double (&y)[NP]) {
#pragma unroll
                         for (int n = 0; n < NP; ++n) {
                           const int64_t k = o + (c * NP + n) * 32;
                           const R v = R(double(Uw[k]) - double(WT[k]));
                           A[k] = v;
                           y[n] = double(v);
                           x[n] = double(D[k]);
                         }
                       });
  const double s = block_sum(da);
  const double s2 = block_sum(dd);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = s;
    partials[gridDim.x + blockIdx.x] = s2;
  }
}

// U0 += alpha_p D; R -= alpha_p A; partial (R, R).
template <int Q, typename R>
__global__ void __launch_bounds__(DOT_THREADS) cg_update_kernel(R* U0, R* Rv, const R* D, const R* A, const double* wdot,
                                                               const Scalars* sc, double* partials, const BlockTable bt,
                                                               const int32_t* pactive) {
  constexpr int NP = np_of(Q);
  const int p = bt.prob[blockIdx.x];
  const bool act = !pactive || pactive[p];
  const int64_t t = block_tet(bt);
  const bool live = act && t >= 0;
  const double alpha = act ? sc[p].alpha : 0.0;
  const int64_t o = live ? field_at(NP, t, threadIdx.x & 1, 0, 0) : 0;
  double rr = 0, unused = 0;
  tet_dots<Q, R, true, false>(live, live ? wdot[2 * t + (threadIdx.x & 1)] : 0.0, rr, unused,
                        [&](int c, double (&x)[NP], double (&y)[NP]) {
#pragma unroll
                          for (int n = 0; n < NP; ++n) {
                            const int64_t k = o + (c * NP + n) * 32;
                            U0[k] = R(double(U0[k]) + alpha * double(D[k]));
                            const R r = R(double(Rv[k]) - alpha * double(A[k]));
                            Rv[k] = r;
                            x[n] = double(r);
                          }
                        });
  const double s = block_sum(rr);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

template <int Q, typename R>
__global__ void __launch_bounds__(DOT_THREADS) dot_kernel(const R* X, const R* Y, const double* wdot, double* partials,
                                                         const BlockTable bt) {
  constexpr int NP = np_of(Q);
  const int64_t t = block_tet(bt);
  const bool live = t >= 0;
  const int64_t o = live ? field_at(NP, t, threadIdx.x & 1, 0, 0) : 0;
  double acc = 0, unused = 0;
  tet_dots<Q, R, false, true>(live, live ? wdot[2 * t + (threadIdx.x & 1)] : 0.0, unused, acc,
                       [&](int c, double (&x)[NP], double (&y)[NP]) {
#pragma unroll
                         for (int n = 0; n < NP; ++n) {
                           x[n] = double(X[o + (c * NP + n) * 32]);
                           y[n] = double(Y[o + (c * NP + n) * 32]);
                         }
                       });
  const double s = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// Rows [tet][6][Np] into field vectors.
template <typename R>
__global__ void scatter_rows_kernel(R* dst_re, R* dst_im, const double* src_re, const double* src_im,
                                    const int64_t* tet, int64_t count, int np) {
  const int64_t rows = 6 * np, n = count * rows;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = i / rows;
    const int k = int(i % rows);
    const int64_t o = field_at(np, tet[e], k / (3 * np), k / np % 3, k % np);
    dst_re[o] = R(src_re[i]);
    dst_im[o] = R(src_im[i]);
  }
}

template <typename R>
__global__ void halo_kernel(R* v, const int64_t* dst, const int64_t* src, int64_t n, int np) {
  const int64_t rows = 6 * np, total = n * rows;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = i / rows;
    const int k = int(i % rows), f = k & 1, m = k >> 1;  // the two fields of a coefficient are adjacent
    v[field_at(np, dst[e], f, 0, m)] = v[field_at(np, src[e], f, 0, m)];
  }
}

__global__ void zero_wdot_kernel(double* wdot, const int64_t* tets, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = tets[i];
    wdot[2 * t] = 0.0;
    wdot[2 * t + 1] = 0.0;
  }
}

// sigma/eps of internal tetrahedra [0, nti) of one problem: val[e] * scale[e] for the external
// tetrahedron e = e_of_i[i] (0 on padding).
template <typename R>
__global__ void set_sigma_kernel(R* geo, const double* val, const double* scale, const int32_t* e_of_i, int64_t nti) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nti; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t e = e_of_i[i];
    const R s = e >= 0 ? R(val[e] * scale[e]) : R(0);
    constexpr int gs = sizeof(R) == 4 ? GEO_S32 : GEO_S64, size = sizeof(R) == 4 ? GEO32 : GEO64;
    R* g = geo + (i >> 4) * size + gs * 16 + GEO_SIGMA * 32 + 2 * (i & 15);
    g[0] = s;
    g[1] = s;
  }
}

// D = R + beta_p D; Uw = D (active problems only).
template <typename R>
__global__ void cg_direction_kernel(R* D, R* Uw, const R* Rv, const Scalars* sc, const int32_t* tprob,
                                    const int32_t* pactive, int64_t n, int64_t tile_len) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = tprob ? tprob[i / tile_len] : 0;
    if (pactive && !pactive[p]) continue;
    const R v = R(double(Rv[i]) + sc[p].beta * double(D[i]));
    D[i] = v;
    Uw[i] = v;
  }
}

__global__ void finalize_kernel(const double* partials, const BlockTable bt, Scalars* sc, int32_t* pactive,
                                const int32_t* used, int which, double tol) {
  __shared__ double sh[256];
  const int p = blockIdx.x;
  const int b0 = bt.coupled ? 0 : bt.pb0[p], b1 = bt.coupled ? bt.nblk : bt.pb0[p + 1];
  auto reduce = [&](const double* part) {
    double s = 0;
    for (int i = b0 + threadIdx.x; i < b1; i += blockDim.x) s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
      __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
  };
  const double tot = reduce(partials);
  // which == 1: (D, D)_M of the same blocks, stored after the (D, A) partials
  const double dd = which == 1 ? reduce(partials + bt.nblk) : 0.0;
  if (threadIdx.x != 0) return;
  Scalars& S = sc[p];
  if (which == 3) {
    S.rr_new = tot;
    return;
  }
  if (which == 4) {  // as 0, for the problems of `used` only (the others are left untouched)
    if (!used || !used[p]) return;
    S.rr = tot;
    S.rr0 = tot;
    S.iters = 0;
    S.status = isfinite(tot) ? 0 : CMCG_ERR_NONFINITE;
    if (pactive) pactive[p] = (S.status == 0 && tot > 0 && sqrt(tot) > tol * sqrt(tot)) ? 1 : 0;
    return;
  }
  if (which == 0) {
    S.rr = tot;
    S.rr0 = tot;
    S.iters = 0;
    S.status = isfinite(tot) ? 0 : CMCG_ERR_NONFINITE;
    const bool in = !used || used[p];
    if (pactive) pactive[p] = (in && S.status == 0 && tot > 0 && sqrt(tot) > tol * sqrt(tot)) ? 1 : 0;
    return;
  }
  if (pactive && !pactive[p]) return;
  if (!isfinite(tot)) {
    S.status = CMCG_ERR_NONFINITE;
    if (pactive) pactive[p] = 0;
    return;
  }
  if (which == 1) {
    S.dA = tot;
    // (D, A) = |(I - P) D|^2 <= (1 + |P|)^2 |D|^2.  A CFL-stable period map is not a
    // contraction in this norm (non-normal transient growth; |P D| / |D| reaches about 3
    // along the CG directions of the test meshes), but a step beyond the stability limit
    // grows by orders of magnitude per period: |(I - P) D| > 100 |D| means |P| > 99.
    if (tot > 1e4 * dd) {
      S.status = CMCG_ERR_UNSTABLE;
      S.alpha = 0;
      if (pactive) pactive[p] = 0;
    } else if (!(tot > 0)) {
      S.status = CMCG_ERR_CG_BREAKDOWN;
      S.alpha = 0;
      if (pactive) pactive[p] = 0;
    } else {
      S.alpha = S.rr / tot;
    }
  } else {  // which == 2
    S.rr_new = tot;
    S.beta = S.rr > 0 ? tot / S.rr : 0.0;
    S.rr = tot;
    S.iters += 1;
    if (pactive && !(sqrt(tot) > tol * sqrt(S.rr0))) pactive[p] = 0;
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 64) b = 152 * 64;
  if (b < 1) b = 1;
  return int(b);
}

}  // namespace

#define CMCG_BY_ORDER(q, KERNEL, blocks, threads, ...)                          \
  do {                                                                          \
    if ((q) == 1) KERNEL<1, R><<<blocks, threads, 0, s>>>(__VA_ARGS__);         \
    else if ((q) == 2) KERNEL<2, R><<<blocks, threads, 0, s>>>(__VA_ARGS__);    \
    else KERNEL<3, R><<<blocks, threads, 0, s>>>(__VA_ARGS__);                  \
  } while (0)

void upload_dot_mass(int q, const double* M) {
  const int np = np_of(q);
  if (q == 1) cudaMemcpyToSymbol(cM1, M, sizeof(double) * np * np);
  else if (q == 2) cudaMemcpyToSymbol(cM2, M, sizeof(double) * np * np);
  else cudaMemcpyToSymbol(cM3, M, sizeof(double) * np * np);
}

template <typename R>
void launch_to_internal(int q, const double* x0, const double* x1, int64_t stride, R* in, const int32_t* e_of_i,
                        int64_t nti, const double* per_tet, cudaStream_t s) {
  const unsigned blocks = unsigned((nti / HTILE * 3 + 3) / 4);  // four warps a block
  CMCG_BY_ORDER(q, to_internal_kernel, blocks, 128, x0, x1, stride, in, e_of_i, nti, per_tet);
}
template <typename R>
void launch_to_external(int q, const R* in, double* x0, double* x1, int64_t stride, const int32_t* e_of_i, int64_t nti,
                        cudaStream_t s) {
  const unsigned blocks = unsigned((nti / HTILE * 3 + 3) / 4);
  CMCG_BY_ORDER(q, to_external_kernel, blocks, 128, in, x0, x1, stride, e_of_i, nti);
}
template <typename R>
void launch_lincomb3_masked(R* o1, R* o2, R* o3, double a, const R* x, double b, const R* y, int64_t n, int np,
                            const int32_t* tprob, const int32_t* mask, cudaStream_t s) {
  lincomb_masked_kernel<R><<<grid_for(n, 256), 256, 0, s>>>(o1, o2, o3, a, x, b, y, n, int64_t(6) * np * TILE, tprob,
                                                            mask);
}
template <typename R>
void launch_lincomb3(R* o1, R* o2, R* o3, double a, const R* x, double b, const R* y, int64_t n, cudaStream_t s) {
  lincomb_kernel<R><<<grid_for(n, 256), 256, 0, s>>>(o1, o2, o3, a, x, b, y, n);
}

template <typename R>
void launch_cg_after_adjoint(int q, const R* Uw, const R* WT, R* A, const R* D, const double* wdot, double* partials,
                             const BlockTable& bt, const int32_t* pactive, cudaStream_t s) {
  CMCG_BY_ORDER(q, cg_after_adjoint_kernel, bt.nblk, DOT_THREADS, Uw, WT, A, D, wdot, partials, bt, pactive);
}
template <typename R>
void launch_cg_update(int q, R* U0, R* Rv, const R* D, const R* A, const double* wdot, const Scalars* sc,
                      double* partials, const BlockTable& bt, const int32_t* pactive, cudaStream_t s) {
  CMCG_BY_ORDER(q, cg_update_kernel, bt.nblk, DOT_THREADS, U0, Rv, D, A, wdot, sc, partials, bt, pactive);
}
template <typename R>
void launch_dot(int q, const R* X, const R* Y, const double* wdot, double* partials, const BlockTable& bt,
                cudaStream_t s) {
  CMCG_BY_ORDER(q, dot_kernel, bt.nblk, DOT_THREADS, X, Y, wdot, partials, bt);
}
template <typename R>
void launch_scatter_rows(R* dst_re, R* dst_im, const double* src_re, const double* src_im, const int64_t* tet,
                         int64_t count, int np, cudaStream_t s) {
  if (count <= 0) return;
  scatter_rows_kernel<R><<<grid_for(count * 6 * np, 256), 256, 0, s>>>(dst_re, dst_im, src_re, src_im, tet, count,
                                                                         np);
}
template <typename R>
void launch_halo(R* v, const int64_t* dst, const int64_t* src, int64_t n, int np, cudaStream_t s) {
  if (n <= 0) return;
  halo_kernel<R><<<grid_for(n * 6 * np, 256), 256, 0, s>>>(v, dst, src, n, np);
}
void launch_zero_wdot(double* wdot, const int64_t* tets, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  zero_wdot_kernel<<<grid_for(n, 256), 256, 0, s>>>(wdot, tets, n);
}
template <typename R>
void launch_set_sigma(R* geo, const double* val, const double* scale, const int32_t* e_of_i, int64_t nti,
                      cudaStream_t s) {
  if (nti <= 0) return;
  set_sigma_kernel<R><<<grid_for(nti, 256), 256, 0, s>>>(geo, val, scale, e_of_i, nti);
}
template <typename R>
void launch_cg_direction(R* D, R* Uw, const R* Rv, const Scalars* sc, const int32_t* tprob, const int32_t* pactive,
                         int64_t n, int np, cudaStream_t s) {
  cg_direction_kernel<R><<<grid_for(n, 256), 256, 0, s>>>(D, Uw, Rv, sc, tprob, pactive, n, int64_t(6) * np * TILE);
}
void launch_finalize(const double* partials, const BlockTable& bt, Scalars* sc, int32_t* pactive, const int32_t* used,
                     int which, double tol, cudaStream_t s) {
  finalize_kernel<<<bt.nprob, 256, 0, s>>>(partials, bt, sc, pactive, used, which, tol);
}

#define CMCG_INST(R)                                                                                                  \
  template void launch_to_internal<R>(int, const double*, const double*, int64_t, R*, const int32_t*, int64_t,         \
                                      const double*, cudaStream_t);                                                   \
  template void launch_to_external<R>(int, const R*, double*, double*, int64_t, const int32_t*, int64_t, cudaStream_t); \
  template void launch_lincomb3<R>(R*, R*, R*, double, const R*, double, const R*, int64_t, cudaStream_t);             \
  template void launch_lincomb3_masked<R>(R*, R*, R*, double, const R*, double, const R*, int64_t, int,                 \
                                          const int32_t*, const int32_t*, cudaStream_t);                                \
  template void launch_cg_after_adjoint<R>(int, const R*, const R*, R*, const R*, const double*, double*,              \
                                           const BlockTable&, const int32_t*, cudaStream_t);                          \
  template void launch_cg_update<R>(int, R*, R*, const R*, const R*, const double*, const Scalars*, double*,          \
                                    const BlockTable&, const int32_t*, cudaStream_t);                                 \
  template void launch_dot<R>(int, const R*, const R*, const double*, double*, const BlockTable&, cudaStream_t);      \
  template void launch_scatter_rows<R>(R*, R*, const double*, const double*, const int64_t*, int64_t, int,        \
                                       cudaStream_t);                                                              \
  template void launch_set_sigma<R>(R*, const double*, const double*, const int32_t*, int64_t, cudaStream_t);        \
  template void launch_halo<R>(R*, const int64_t*, const int64_t*, int64_t, int, cudaStream_t);                        \
  template void launch_cg_direction<R>(R*, R*, const R*, const Scalars*, const int32_t*, const int32_t*, int64_t,     \
                                       int, cudaStream_t);
CMCG_INST(float)
CMCG_INST(double)

}  // namespace cmcg
