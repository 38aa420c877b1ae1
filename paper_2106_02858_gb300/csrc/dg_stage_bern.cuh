// The stage of dg_stage.cuh on Bernstein coefficients (bernstein.h), FP64 handles; included by
// dg_stage.cuh inside its anonymous namespace, once per order.  GB300 does two FP64 operations per
// clock and SM, so the operations are the cost, and in this basis both terms are sparse:
//
//   curl:  the 4 x 3 differences c_{a + e_k} - c_{a + e_0} of each degree-(q - 1) index a,
//          the chain rule and curl on those (27 operations), and a weight a_i + 1 into each
//          of the four coefficients a + e_i: 390 operations per field at P3, 156 at P2,
//          where the dense derivatives and their chain rule take 4,080 and 1,140;
//   flux:  f is tangential, so X is projected on the face's frame (t1, t2) once, two numbers
//          instead of three go through the shuffle and the lift, and f = k1 [(k y1 - x2) t1 +
//          (k y2 + x1) t2], k = k2 / k1, is put back together on the lifted coefficients;
//   lift:  the face-local product of at most seven integer weights per row, then one degree
//          reduction per layer behind the face: 76 operations per face and flux component at
//          P3, 33 at P2, where the dense lift takes 200 and 60.
//
// 10,368 P2 tetrahedra: 144 us per stage with the dense matrices, 52 so; 384 P1 16 and 6.0.  A warp's FP64
// instruction holds its SM quarter's unit for 64 cycles, so four warps of one block share a small
// mesh's half tile (SPLIT 4) as well as four SMs would (a cluster of one-warp blocks: 7.7 us).

// The curl: index m's share of (scale * curl F) in phi, G already scaled by the material factor.
__device__ __forceinline__ void add_curl(double (&phi)[3][NPQ], const double (&v)[3][NPQ], const double (&G)[9], int m) {
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
  double d[3][3];  // [direction][component]
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) d[k][c] = v[c][B.up[m][k + 1]] - v[c][B.up[m][0]];
  double w[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {  // component c: d_{c+1} F_{c+2} - d_{c+2} F_{c+1}
    const int p = (c + 1) % 3, q = (c + 2) % 3;
    w[c] = G[0 * 3 + p] * d[0][q];
    w[c] = fma(G[1 * 3 + p], d[1][q], w[c]);
    w[c] = fma(G[2 * 3 + p], d[2][q], w[c]);
    w[c] = fma(-G[0 * 3 + q], d[0][p], w[c]);
    w[c] = fma(-G[1 * 3 + q], d[1][p], w[c]);
    w[c] = fma(-G[2 * 3 + q], d[2][p], w[c]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 3; ++c) phi[c][B.up[m][i]] = fma(double(B.upw[m][i]), w[c], phi[c][B.up[m][i]]);
}

// The lift of face f's flux k1 (g1 t1 + g2 t2) into phi.
__device__ __forceinline__ void add_lift(double (&phi)[3][NPQ], const double (&g)[2][NFPQ], const double (&t)[6], double k1, int f) {
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
  double h[2][NFPQ];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    double s = double(0);
    bool any = false;
#pragma unroll
    for (int n = 0; n < NFPQ; ++n)
      if (B.in_sum[n]) {
        s = any ? s + g[k][n] : g[k][n];
        any = true;
      }
#pragma unroll
    for (int n = 0; n < NFPQ; ++n) {
      bool first = !B.in_sum[n];
      double x = B.in_sum[n] ? s : double(0);
#pragma unroll
      for (int m = 0; m < NFPQ; ++m)
        if (B.l0[n][m] != 0) {
          x = first ? double(B.l0[n][m]) * g[k][m] : fma(double(B.l0[n][m]), g[k][m], x);
          first = false;
        }
      h[k][n] = x;
    }
  }
#pragma unroll
  for (int j = 0; j <= CMCG_Q; ++j) {
    const int nj = (CMCG_Q - j + 1) * (CMCG_Q - j + 2) / 2;
    if (j > 0) {  // one degree reduction
      double r[2][NFPQ];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int n = 0; n < NFPQ; ++n)
          if (n < nj)
            r[k][n] = fma(double(B.redw[j][n][2]), h[k][B.red[j][n][2]],
                          fma(double(B.redw[j][n][1]), h[k][B.red[j][n][1]], double(B.redw[j][n][0]) * h[k][B.red[j][n][0]]));
#pragma unroll
        for (int n = 0; n < NFPQ; ++n)
          if (n < nj) h[k][n] = r[k][n];
      }
    }
    const double lk = double(layer_weight(j)) * k1;
    double tj[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) tj[k] = lk * t[k];
#pragma unroll
    for (int n = 0; n < NFPQ; ++n)
      if (n < nj)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          phi[c][B.layer[f][j][n]] = fma(h[0][n], tj[c], fma(h[1][n], tj[3 + c], phi[c][B.layer[f][j][n]]));
  }
}

// What a warp needs of one face before the previous stage has ended.
struct BernFace {
  double t[6], k1, k;
  Neighbour<double> nb;
};
__device__ __forceinline__ BernFace load_bern_face(const StageArgs<double>& a, int64_t ht, int l, int f) {
  BernFace F;
  const double* gs = a.geo + ht * GEO64 + (9 + 6 * f) * 16 + (l >> 1);
#pragma unroll
  for (int k = 0; k < 6; ++k) F.t[k] = gs[k * 16];
  const double* gp = a.geo + ht * GEO64 + GEO_S64 * 16 + (1 + 2 * f) * 32 + l;
  F.k1 = gp[0] * a.sH;
  F.k = gp[32] * a.sH;
  F.nb = find_neighbour(a, ht, l, f);
  return F;
}

// The flux of face f in its frame, divided by k1: own field v, neighbour trace tr.
__device__ __forceinline__ void bern_flux(double (&g)[2][NFPQ], const double (&tr)[3][NFPQ], const double (&v)[3][NPQ],
                                          const double (&t)[6], double cf, double k, int f) {
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
#pragma unroll
  for (int n = 0; n < NFPQ; ++n) {
    double X[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) X[c] = fma(cf, tr[c][n], -v[c][B.face[f][n]]);
    const double x1 = fma(t[2], X[2], fma(t[1], X[1], t[0] * X[0]));
    const double x2 = fma(t[5], X[2], fma(t[4], X[1], t[3] * X[0]));
    const double y1 = __shfl_xor_sync(0xffffffffu, x1, 1), y2 = __shfl_xor_sync(0xffffffffu, x2, 1);
    g[0][n] = fma(k, y1, -x2);
    g[1][n] = fma(k, y2, x1);
  }
}

// One part (warp p of SPLIT) of a half tile's stage; returns with the block's barriers unused
// unless SPLIT > 1 (every warp of a half tile takes the same exits).
template <int SPLIT, int P>
__device__ __forceinline__ void bern_part(const StageArgs<double>& a, int64_t ht, int l, int warp, double* xs) {
  constexpr int NP = NPQ, NA = BernTab<CMCG_Q>::NA, NF = 4 / SPLIT, F0 = P * NF;
  constexpr int I0 = P * NP / SPLIT, NN = (P + 1) * NP / SPLIT - I0;  // output coefficients finished here
  const int prob = a.tprob ? a.tprob[ht >> 1] : 0;
  const StageCoef<double> cf = a.coef[prob];
  if (!cf.active) return;
  const int half = l & 1;
  double G[9];
  {
    const double* gs = a.geo + ht * GEO64 + (l >> 1);
    const double* gp = a.geo + ht * GEO64 + GEO_S64 * 16 + l;
    const double sv = gp[0] * a.sH;
#pragma unroll
    for (int k = 0; k < 9; ++k) G[k] = gs[k * 16] * sv;
  }
  BernFace F[NF];
#pragma unroll
  for (int ff = 0; ff < NF; ++ff) F[ff] = load_bern_face(a, ht, l, F0 + ff);
  const double sigma = a.sigma ? a.geo[ht * GEO64 + (GEO_S64 * 16 + GEO_SIGMA * 32) + l] : double(0);

  grid_dep_wait();
  grid_dep_launch();
  if (a.pactive && !a.pactive[prob]) return;  // CG converged for this problem (written by the CG kernels)
  const int64_t own = ht * HS + l;  // the thread's field; its output is the partner's, own ^ 1
  // Traces run one face ahead of their use.
  double tr[2][3][NFPQ];
  load_trace(tr[0], a.vin, F[0].nb);
  double v[3][NP];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int n = 0; n < NP; ++n) v[c][n] = a.vin[own + (c * NP + n) * 32];
  double phi[3][NP];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int n = 0; n < NP; ++n) phi[c][n] = double(0);
#pragma unroll
  for (int m = P * NA / SPLIT; m < (P + 1) * NA / SPLIT; ++m) add_curl(phi, v, G, m);
  double bv[3][NN];
#pragma unroll
  for (int ff = 0; ff < NF; ++ff) {
    if (ff + 1 < NF) load_trace(tr[(ff + 1) & 1], a.vin, F[ff + 1].nb);
    if (ff + 1 == NF && a.out) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int n = 0; n < NN; ++n) bv[c][n] = a.base[(own ^ 1) + (c * NP + I0 + n) * 32];
    }
    double g[2][NFPQ];
    bern_flux(g, tr[ff & 1], v, F[ff].t, F[ff].nb.c, F[ff].k, F0 + ff);
    add_lift(phi, g, F[ff].t, F[ff].k1, F0 + ff);
  }
  double out[3][NN];
  if constexpr (SPLIT > 1) {
    // Partial sums of the other parts' coefficients to shared memory, the others' of ours back.
    double* mine = xs + warp * (3 * NP * 32) + l;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NP; ++n)
        if (n < I0 || n >= I0 + NN) mine[(c * NP + n) * 32] = phi[c][n];
    asm volatile("bar.sync %0, %1;\n" ::"r"(1 + warp / SPLIT), "n"(32 * SPLIT) : "memory");
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NN; ++n) {
        double s = phi[c][I0 + n];
#pragma unroll
        for (int k = 0; k < SPLIT; ++k)
          if (k != P) s += xs[((warp / SPLIT) * SPLIT + k) * (3 * NP * 32) + (c * NP + I0 + n) * 32 + l];
        out[c][n] = s;
      }
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NN; ++n) out[c][n] = phi[c][n];
  }
  // one branch around everything that few stages have: the common stage's last operations stay
  // together (with a branch per component and term the 384-tetrahedron P1 stage took 7.6 us, so 6.4;
  // 10,368 P2 tetrahedra 57.7 and 52.8)
  if (a.j || a.sigma || a.bre || a.fre) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double jv[NN] = {};
      if (a.j && a.nharm <= 0) load_source<double, NN>(jv, a.j + own, c, I0);
      add_data<double, NN>(out[c], jv, a, cf, own, c, I0, half, sigma);
      if (a.fre) accumulate_filter<double, NN>(a, cf, out[c], own, c, I0);  // forward sweeps with the filter only
    }
  }
  if (a.out) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NN; ++n) a.out[(own ^ 1) + (c * NP + I0 + n) * 32] = bv[c][n] + cf.c_out * out[c][n];
  }
}

