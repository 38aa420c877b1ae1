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
// 10,368 P2 tetrahedra: 144 us per stage with the dense matrices, 48 so; 384 P1 16 and 5.8.  A warp's FP64
// instruction holds its SM quarter's unit for 64 cycles, so four warps of one block share a small
// mesh's half tile (SPLIT 4) as well as four SMs would (a cluster of one-warp blocks: 7.7 us).

// Component c of the curl of index m, d_{c+1} F_{c+2} - d_{c+2} F_{c+1}, G already scaled by the material
// factor: it goes into the output with weight a_i + 1 at each of the four coefficients a + e_i.
__device__ __forceinline__ double curl_of(const double (&v)[3][NPQ], const double (&G)[9], int m, int c) {
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
  const int p = (c + 1) % 3, q = (c + 2) % 3;
  auto d = [&](int k, int e) { return v[e][B.up[m][k + 1]] - v[e][B.up[m][0]]; };  // direction k, component e
  double w = G[0 * 3 + p] * d(0, q);
  w = fma(G[1 * 3 + p], d(1, q), w);
  w = fma(G[2 * 3 + p], d(2, q), w);
  w = fma(-G[0 * 3 + q], d(0, p), w);
  w = fma(-G[1 * 3 + q], d(1, p), w);
  return fma(-G[2 * 3 + q], d(2, p), w);
}

// Coefficients of the layers 0 .. j - 1 behind a face.
constexpr int layer_at(int j) {
  int s = 0;
  for (int i = 0; i < j; ++i) s += (CMCG_Q - i + 1) * (CMCG_Q - i + 2) / 2;
  return s;
}
static_assert(layer_at(CMCG_Q + 1) == NPQ, "the layers hold every coefficient once");

// The lift of a flux k1 (g1 t1 + g2 t2): frame(j, tj) is called with layer j's scaled frame, then
// coef(j, n, h1, h2) for each of its coefficients n, to which h1 tj[c] + h2 tj[3 + c] is to be added.
template <typename Frame, typename Coef>
__device__ __forceinline__ void lift_of(const double (&g)[2][NFPQ], const double (&t)[6], double k1, Frame&& frame, Coef&& coef) {
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
    frame(j, tj);
#pragma unroll
    for (int n = 0; n < NFPQ; ++n)
      if (n < nj) coef(j, n, h[0][n], h[1][n]);
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

// Shared memory of a half tile (values per lane), SPLIT > 1: the curl of every index, every face's
// lift before it is spread over the components, and the layers' scaled frames.
constexpr int BERN_W = 0;
constexpr int BERN_H = BERN_W + BernTab<CMCG_Q>::NA * 3;
constexpr int BERN_T = BERN_H + 4 * 2 * NPQ;
constexpr int BERN_SMEM = BERN_T + 4 * (CMCG_Q + 1) * 6;

// Source, conductivity, data and filter on part K, Np values at most, of the output values o0 .. o0 + NO - 1.
template <int K, int NO>
__device__ __forceinline__ void bern_terms(double (&out)[NO], const StageArgs<double>& a, const StageCoef<double>& cf,
                                           int64_t own, int o0, int half, double sigma) {
  constexpr int A = K * NPQ, N = NO - A < NPQ ? NO - A : NPQ;
  double p[N], jv[N] = {};
#pragma unroll
  for (int k = 0; k < N; ++k) p[k] = out[A + k];
  if (a.j && a.nharm <= 0) load_source<double, N>(jv, a.j + own, 0, o0 + A);
  add_data<double, N>(p, jv, a, cf, own, 0, o0 + A, half, sigma);
  if (a.fre) accumulate_filter<double, N>(a, cf, p, own, 0, o0 + A);  // forward sweeps with the filter only
#pragma unroll
  for (int k = 0; k < N; ++k) out[A + k] = p[k];
}

// One part (warp p of SPLIT) of a half tile's stage; returns with the block's barriers unused
// unless SPLIT > 1 (every warp of a half tile takes the same exits).
//
// Every output value's sum has one order whatever the split, the curl's indices and then the faces: a
// handle's split is chosen by timing and must not show in its results.  So the warps of a half tile
// don't exchange partial sums of the output but what goes into them: each computes its share of the
// curl and of the faces' lifts, and after the barrier finishes its share of the 3 Np output values.
// That is also 3 (SPLIT - 1) Np fewer operations per tetrahedron and field than adding partial sums up,
// and at P3 a warp need not hold all 60 sums (four warps a half tile, us per stage, with partial sums
// and so: 2,058 P3 tetrahedra 22.7 and 22.5, 10,368 98.7 and 92.5, 10,368 P2 51.0 and 48.3, 384 P1 6.1 and
// 5.8).  Both shares are cut by value, not by index or coefficient: the P1 curl has one index (one warp
// with all of it: 6.3), and P2's ten coefficients don't go into four (384 tetrahedra 12.3, so 11.95).
template <int SPLIT, int P>
__device__ __forceinline__ void bern_part(const StageArgs<double>& a, int64_t ht, int l, int warp, double* xs) {
  constexpr int NP = NPQ, NA = BernTab<CMCG_Q>::NA, NF = 4 / SPLIT, F0 = P * NF;
  // Output values finished here, value c Np + n being coefficient n of component c.
  constexpr int O0 = P * 3 * NP / SPLIT, NO = (P + 1) * 3 * NP / SPLIT - O0;
  constexpr BernTab<CMCG_Q> B = make_bern<CMCG_Q>();
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
  double out[NO];
#pragma unroll
  for (int k = 0; k < NO; ++k) out[k] = double(0);
  auto mine = [&](int c, int n) { return c * NP + n >= O0 && c * NP + n < O0 + NO; };
  auto add_curl = [&](int m, int c, double w) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (mine(c, B.up[m][i])) {
        double& o = out[c * NP + B.up[m][i] - O0];
        o = fma(double(B.upw[m][i]), w, o);
      }
  };
  auto add_coef = [&](int f, int j, int n, double h1, double h2, const double (&tj)[6]) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (mine(c, B.layer[f][j][n])) {
        double& o = out[c * NP + B.layer[f][j][n] - O0];
        o = fma(h1, tj[c], fma(h2, tj[3 + c], o));
      }
  };
  double* sm = xs + (warp / SPLIT) * (BERN_SMEM * 32) + l;  // SPLIT > 1
#pragma unroll
  for (int k = P * 3 * NA / SPLIT; k < (P + 1) * 3 * NA / SPLIT; ++k) {
    const double w = curl_of(v, G, k / 3, k % 3);
    if constexpr (SPLIT == 1) add_curl(k / 3, k % 3, w);
    else sm[(BERN_W + k) * 32] = w;
  }
  double bv[NO];
#pragma unroll
  for (int ff = 0; ff < NF; ++ff) {
    if (ff + 1 < NF) load_trace(tr[(ff + 1) & 1], a.vin, F[ff + 1].nb);
    if (ff + 1 == NF && a.out) {
#pragma unroll
      for (int k = 0; k < NO; ++k) bv[k] = a.base[(own ^ 1) + (O0 + k) * 32];
    }
    const int f = F0 + ff;
    double g[2][NFPQ];
    bern_flux(g, tr[ff & 1], v, F[ff].t, F[ff].nb.c, F[ff].k, f);
    double tj[6];
    lift_of(
        g, F[ff].t, F[ff].k1,
        [&](int j, const double (&t)[6]) {
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            if constexpr (SPLIT == 1) tj[k] = t[k];
            else sm[(BERN_T + (f * (CMCG_Q + 1) + j) * 6 + k) * 32] = t[k];
          }
        },
        [&](int j, int n, double h1, double h2) {
          if constexpr (SPLIT == 1) {
            add_coef(f, j, n, h1, h2, tj);
          } else {
            sm[(BERN_H + (f * NP + layer_at(j) + n) * 2) * 32] = h1;
            sm[(BERN_H + (f * NP + layer_at(j) + n) * 2 + 1) * 32] = h2;
          }
        });
  }
  if constexpr (SPLIT > 1) {
    asm volatile("bar.sync %0, %1;\n" ::"r"(1 + warp / SPLIT), "n"(32 * SPLIT) : "memory");
#pragma unroll
    for (int k = 0; k < 3 * NA; ++k) add_curl(k / 3, k % 3, sm[(BERN_W + k) * 32]);
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int j = 0; j <= CMCG_Q; ++j) {
        double tj[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) tj[k] = sm[(BERN_T + (f * (CMCG_Q + 1) + j) * 6 + k) * 32];
#pragma unroll
        for (int n = 0; n < NFPQ; ++n)
          if (n < (CMCG_Q - j + 1) * (CMCG_Q - j + 2) / 2)
            add_coef(f, j, n, sm[(BERN_H + (f * NP + layer_at(j) + n) * 2) * 32],
                     sm[(BERN_H + (f * NP + layer_at(j) + n) * 2 + 1) * 32], tj);
      }
  }
  // one branch around everything that few stages have: the common stage's last operations stay
  // together (with a branch per component and term the 384-tetrahedron P1 stage took 7.6 us, so 6.4;
  // 10,368 P2 tetrahedra 57.7 and 52.8)
  if (a.j || a.sigma || a.bre || a.fre) {
    bern_terms<0, NO>(out, a, cf, own, O0, half, sigma);
    if constexpr (NO > NP) bern_terms<1, NO>(out, a, cf, own, O0, half, sigma);
    if constexpr (NO > 2 * NP) bern_terms<2, NO>(out, a, cf, own, O0, half, sigma);
  }
  if (a.out) {
#pragma unroll
    for (int k = 0; k < NO; ++k) a.out[(own ^ 1) + (O0 + k) * 32] = fma(cf.c_out, out[k], bv[k]);
  }
}
