// The stage of dg_stage.cuh on nodal values, FP32 handles; included by dg_stage.cuh inside its
// anonymous namespace, once per order.
//
// Reference derivatives: at P1 and P2 the entries of D_r, D_s, D_t are small whole numbers and
// half of them (P1) and 58% (P2) are zero; with the loops unrolled the zeros cost nothing and the
// others are immediate operands.  At P3 they, and the lift at every order, are constant-bank
// operands.  Each output value's sums run in a fixed order (derivatives over j, the lift over faces
// and face nodes), whatever the split.
//
// Issue slots and the latency of a half tile's first loads bound it, not the FP32 pipe (7 of 15.5 us at
// 81,648 P2 tetrahedra) or the bytes (11 us).  So two values go through one packed instruction
// wherever two neighbours have the same factor or the same place in a sum; the pipe's rate is that of
// single ones, but warp instructions and time of that stage were 13.2 M and 19.2 us with single ones,
// 11.1 M and 16.5 us with the lift packed, 9.1 M and 15.5 us with the fluxes and, at P2, the volume
// sums too.  Twelve warps of 168 registers per SM, in blocks of two (48,000 tetrahedra: 9.7 us in blocks
// of four, 9.5 of two; one-warp blocks 12.9); sixteen of 128 registers take 10.6 us there.
__constant__ float cD[CMCG_Q == 3 ? 3 * NPQ * NPQ : 1];
__constant__ __align__(8) float cL[4 * NFPQ * NPQ];  // [face node][node]

// Multiply-add and product of two values at once, each rounded once as by fmaf and *; the same names
// for one value.
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n.reg .b64 x, y, z, r;\nmov.b64 x, {%2, %3};\nmov.b64 y, {%4, %5};\nmov.b64 z, {%6, %7};\n"
      "fma.rn.f32x2 r, x, y, z;\nmov.b64 {%0, %1}, r;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b) {
  float2 d;
  asm("{\n.reg .b64 x, y, r;\nmov.b64 x, {%2, %3};\nmov.b64 y, {%4, %5};\n"
      "mul.rn.f32x2 r, x, y;\nmov.b64 {%0, %1}, r;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
template <typename T>
__device__ __forceinline__ T splat(float a) {
  if constexpr (sizeof(T) == 8) return {a, a};
  else return a;
}
// phi[n - I0] += L[n][k] fl for the nodes n = I0 .. I0 + NN - 1 and face node k, two nodes per
// instruction.
template <int I0, int NN>
__device__ __forceinline__ void nodal_lift(float (&phi)[NN], float fl, int k) {
  const float* L = cL + k * NPQ;
#pragma unroll
  for (int n = I0 & ~1; n < I0 + NN; n += 2) {
    if (n >= I0 && n + 1 < I0 + NN) {
      const float2 w = *reinterpret_cast<const float2*>(L + n);
      const float2 r = vfma(w, splat<float2>(fl), {phi[n - I0], phi[n + 1 - I0]});
      phi[n - I0] = r.x;
      phi[n + 1 - I0] = r.y;
    } else {
      const int m = n < I0 ? n + 1 : n;
      phi[m - I0] = fmaf(L[m], fl, phi[m - I0]);
    }
  }
}

// D_b[i][j] of orders 1 and 2, exact: nodal values -> Bernstein coefficients -> differences raised
// back to degree q -> values (all weights are dyadic there).
struct NodalD {
  float d[3][NPQ][NPQ];
};
constexpr NodalD make_nodal_d() {
  NodalD t{};
  if (CMCG_Q == 3) return t;
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
  constexpr BasisRows<CMCG_Q> N = make_to_node<CMCG_Q>(), I = make_to_bern<CMCG_Q>();
  for (int j = 0; j < NPQ; ++j) {
    double c[NPQ] = {};  // Bernstein coefficients of the nodal basis function j
    for (int m = 0; m < NPQ; ++m)
      for (int k = 0; k < I.r[m].n; ++k)
        if (I.r[m].col[k] == j) c[m] = I.r[m].w[k];
    for (int b = 0; b < 3; ++b) {
      double e[NPQ] = {};
      for (int a = 0; a < BernTab<CMCG_Q>::NA; ++a)
        for (int i = 0; i < 4; ++i) e[B.up[a][i]] += B.upw[a][i] * (c[B.up[a][b + 1]] - c[B.up[a][0]]);
      for (int i = 0; i < NPQ; ++i) {
        double v = 0;
        for (int k = 0; k < N.r[i].n; ++k) v += N.r[i].w[k] * e[N.r[i].col[k]];
        t.d[b][i][j] = float(v);
      }
    }
  }
  return t;
}

// The flux of a face at one or two of its nodes: jumps X and the partner's Y, normal n, (k1, k2).
template <typename T>
__device__ __forceinline__ void flux_nodes(T (&fl)[3], const T (&X)[3], const T (&Y)[3], float n0, float n1, float n2,
                                           float k1, float k2) {
  const float n[3] = {n0, n1, n2};
  const T nY = vfma(splat<T>(n2), Y[2], vfma(splat<T>(n0), Y[0], vmul(splat<T>(n1), Y[1])));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int a = (c + 1) % 3, b = (c + 2) % 3;
    const T nX = vfma(splat<T>(n[a]), X[b], vmul(splat<T>(-n[b]), X[a]));  // (n x X)_c
    const T tY = vfma(splat<T>(-n[c]), nY, Y[c]);                         // (Y - n (n.Y))_c
    fl[c] = vfma(splat<T>(k1), nX, vmul(splat<T>(k2), tY));
  }
}
// The flux of face f at its nodes: normal n, (k1, k2), trace weight wt, neighbour trace tr.
__device__ __forceinline__ void nodal_flux(float (&fl)[3][NFPQ], const float (&tr)[3][NFPQ], const float (&v)[3][NPQ],
                                           float n0, float n1, float n2, float k1, float k2, float wt, int f) {
  constexpr FaceTab FM = make_fmask(CMCG_Q);
#pragma unroll
  for (int jf = 0; jf < NFPQ; jf += 2) {
    if (jf + 1 < NFPQ) {
      float2 X[3], Y[3], F[3];
#pragma unroll
      for (int c = 0; c < 3; ++c)
        X[c] = {fmaf(wt, tr[c][jf], -v[c][FM.v[f][jf]]), fmaf(wt, tr[c][jf + 1], -v[c][FM.v[f][jf + 1]])};
#pragma unroll
      for (int c = 0; c < 3; ++c)
        Y[c] = {__shfl_xor_sync(0xffffffffu, X[c].x, 1), __shfl_xor_sync(0xffffffffu, X[c].y, 1)};
      flux_nodes<float2>(F, X, Y, n0, n1, n2, k1, k2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        fl[c][jf] = F[c].x;
        fl[c][jf + 1] = F[c].y;
      }
    } else {
      float X[3], Y[3], F[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) X[c] = fmaf(wt, tr[c][jf], -v[c][FM.v[f][jf]]);
#pragma unroll
      for (int c = 0; c < 3; ++c) Y[c] = __shfl_xor_sync(0xffffffffu, X[c], 1);
      flux_nodes<float>(F, X, Y, n0, n1, n2, k1, k2);
#pragma unroll
      for (int c = 0; c < 3; ++c) fl[c][jf] = F[c];
    }
  }
}

// Shared memory of a warp (floats): the half tile's geometry and its rows of base (SPLIT == 1 only:
// the other splits read the few base values they need directly), copied asynchronously 16 bytes a
// lane; then the warp's fluxes (SPLIT > 1).
template <int SPLIT>
constexpr int nodal_smem() {
  return GEO32 + (SPLIT == 1 ? HS : 4 / SPLIT * NFPQ * 3 * 32);
}
// n floats (a multiple of 4) from src to dst, both 16-byte aligned, by the warp.
__device__ __forceinline__ void warp_copy_async(float* dst, const float* src, int n, int l) {
#pragma unroll
  for (int k = 0; k < n; k += 128)
    if (k + 4 * l < n) cp_async_16(dst + k + 4 * l, src + k + 4 * l);
  cp_async_commit();
}

// One part (warp p of SPLIT) of a half tile's stage (every warp of a half tile takes the same exits).
template <int SPLIT, int P>
__device__ __forceinline__ void nodal_part(const StageArgs<float>& a, int64_t ht, int l, int warp, float* xs) {
  constexpr int NP = NPQ, NFP = NFPQ, NF = 4 / SPLIT, F0 = P * NF;
  constexpr int I0 = P * NP / SPLIT, NN = (P + 1) * NP / SPLIT - I0;  // output values of this part
  constexpr NodalD D = make_nodal_d();
  const int prob = a.tprob ? a.tprob[ht >> 1] : 0;
  const StageCoef<float> cf = a.coef[prob];
  if (!cf.active) return;
  const int half = l & 1;
  float* gsm = xs + warp * nodal_smem<SPLIT>();
  warp_copy_async(gsm, a.geo + ht * GEO32, GEO32, l);
  Neighbour<float> nb[NF];
#pragma unroll
  for (int ff = 0; ff < NF; ++ff) nb[ff] = find_neighbour(a, ht, l, F0 + ff);

  grid_dep_wait();
  grid_dep_launch();
  if (a.pactive && !a.pactive[prob]) {  // CG converged for this problem (written by the CG kernels)
    cp_async_wait<0>();
    return;
  }
  const int64_t own = ht * HS + l;  // the thread's field; its output is the partner's, own ^ 1
  // One face's traces at a time: the first face's are loaded before the volume sums, each next
  // face's as soon as the flux has used the last ones', before that face's lift.
  float tr[3][NFP];
  load_trace(tr, a.vin, nb[0]);
  float v[3][NP];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int n = 0; n < NP; ++n) v[c][n] = a.vin[own + (c * NP + n) * 32];
  if (SPLIT == 1 && a.out) {
    warp_copy_async(gsm + GEO32, a.base + ht * HS, HS, l);
    cp_async_wait<1>();
  } else {
    cp_async_wait<0>();
  }
  __syncwarp();
  const float* gs = gsm + (l >> 1);
  const float* gp = gsm + GEO_S32 * 16 + l;
  float G[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) G[k] = gs[k * 16];
  const float sv = gp[0] * a.sH;
  float phi[3][NN];
#pragma unroll
  for (int ii = 0; ii < NN; ++ii) {
    const int i = I0 + ii;
    if constexpr (CMCG_Q == 1) {  // sums of two terms: nothing to pack (4,374 tetrahedra: 2.7 us packed, 2.45 so)
      float d[3][3];  // [direction][component]
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        bool first = true;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          if (D.d[b][i][j] == 0.0f) continue;
#pragma unroll
          for (int c = 0; c < 3; ++c) d[b][c] = first ? D.d[b][i][j] * v[c][j] : fmaf(D.d[b][i][j], v[c][j], d[b][c]);
          first = false;
        }
      }
      // d/dx_ax of component c = sum_b G[b][ax] d[b][c]
      auto dx = [&](int ax, int c) { return fmaf(G[2 * 3 + ax], d[2][c], fmaf(G[0 * 3 + ax], d[0][c], G[1 * 3 + ax] * d[1][c])); };
      phi[0][ii] = sv * (dx(1, 2) - dx(2, 1));
      phi[1][ii] = sv * (dx(2, 0) - dx(0, 2));
      phi[2][ii] = sv * (dx(0, 1) - dx(1, 0));
    } else {
      float2 d10[3];  // d/db of components (1, 0)
      float d2[3];    // of component 2
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        bool first = true;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          if (CMCG_Q < 3 && D.d[b][i][j] == 0.0f) continue;
          const float w = CMCG_Q < 3 ? D.d[b][i][j] : cD[(b * NP + i) * NP + j];
          const float2 v10 = {v[1][j], v[0][j]}, ww = {w, w};
          d10[b] = first ? vmul(ww, v10) : vfma(ww, v10, d10[b]);
          d2[b] = first ? vmul(w, v[2][j]) : vfma(w, v[2][j], d2[b]);
          first = false;
        }
      }
      // d/dx_ax of component c = sum_b G[b][ax] d[b][c], two at a time
      auto sum = [&](float2 g0, float2 e0, float2 g1, float2 e1, float2 g2, float2 e2) {
        return vfma(g2, e2, vfma(g0, e0, vmul(g1, e1)));
      };
      const float2 z = sum(splat<float2>(G[2]), d10[0], splat<float2>(G[5]), d10[1], splat<float2>(G[8]), d10[2]);
      const float2 xy = sum({G[0], G[1]}, d10[0], {G[3], G[4]}, d10[1], {G[6], G[7]}, d10[2]);
      const float2 xy2 = sum({G[0], G[1]}, splat<float2>(d2[0]), {G[3], G[4]}, splat<float2>(d2[1]), {G[6], G[7]},
                             splat<float2>(d2[2]));
      phi[0][ii] = sv * (xy2.y - z.x);
      phi[1][ii] = sv * (z.y - xy2.x);
      phi[2][ii] = sv * (xy.x - xy.y);
    }
  }
  float bv[3][NN], jv[3][NN];
  float* mine = gsm + GEO32 + l;  // this warp's fluxes (SPLIT > 1)
#pragma unroll
  for (int ff = 0; ff < NF; ++ff) {
    if (ff + 1 == NF) {
      if (SPLIT > 1 && a.out) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int n = 0; n < NN; ++n) bv[c][n] = a.base[(own ^ 1) + (c * NP + I0 + n) * 32];
      }
      if (a.j && a.nharm <= 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) load_source<float, NN>(jv[c], a.j + own, c, I0);
      }
    }
    const int f = F0 + ff;
    float fl[3][NFP];
    nodal_flux(fl, tr, v, gs[(9 + 3 * f) * 16], gs[(10 + 3 * f) * 16], gs[(11 + 3 * f) * 16],
               gp[(1 + 2 * f) * 32] * a.sH, gp[(2 + 2 * f) * 32], nb[ff].c, f);
    if (ff + 1 < NF) load_trace(tr, a.vin, nb[ff + 1 < NF ? ff + 1 : 0]);
    if constexpr (SPLIT == 1) {
#pragma unroll
      for (int jf = 0; jf < NFP; ++jf)
#pragma unroll
        for (int c = 0; c < 3; ++c) nodal_lift<I0, NN>(phi[c], fl[c][jf], (F0 + ff) * NFP + jf);
    } else {
#pragma unroll
      for (int jf = 0; jf < NFP; ++jf)
#pragma unroll
        for (int c = 0; c < 3; ++c) mine[((ff * NFP + jf) * 3 + c) * 32] = fl[c][jf];
    }
  }
  if constexpr (SPLIT > 1) {  // every face's flux from shared memory, in the order of the faces
    asm volatile("bar.sync %0, %1;\n" ::"r"(1 + warp / SPLIT), "n"(32 * SPLIT) : "memory");
    const float* all = xs + (warp / SPLIT) * SPLIT * nodal_smem<SPLIT>() + GEO32 + l;
#pragma unroll
    for (int k = 0; k < 4 * NFP; ++k) {
      float fl[3];
#pragma unroll
      for (int c = 0; c < 3; ++c)
        fl[c] = all[(k / (NF * NFP)) * nodal_smem<SPLIT>() + ((k % (NF * NFP)) * 3 + c) * 32];
#pragma unroll
      for (int c = 0; c < 3; ++c) nodal_lift<I0, NN>(phi[c], fl[c], k);
    }
  }
  if (SPLIT == 1 && a.out) {
    cp_async_wait<0>();
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NN; ++n) bv[c][n] = gsm[GEO32 + (c * NP + n) * 32 + (l ^ 1)];
  }
  const float sigma = a.sigma ? gp[GEO_SIGMA * 32] : 0.0f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    add_data<float, NN>(phi[c], jv[c], a, cf, own, c, I0, half, sigma);
    if (a.fre) accumulate_filter<float, NN>(a, cf, phi[c], own, c, I0);  // forward sweeps with the filter only
    if (a.out) {
#pragma unroll
      for (int n = 0; n < NN; ++n) a.out[(own ^ 1) + (c * NP + I0 + n) * 32] = fmaf(cf.c_out, phi[c][n], bv[c][n]);
    }
  }
}
