// The RK stage of dg_stage.cuh with the two dense contractions of the DG operator
// (Section 5.2.2, Eq. DG_semidiscrete / Eq. ode_system) on the 5th-generation
// tensor cores: the reference derivatives D_b F (b = r, s, t) of the own field
// and the lift LIFT . f of the face fluxes.  FP32 sweeps only; included by
// dg_stage.cuh inside its anonymous namespace, once per order.
//
// Mapping.  A CTA covers 64 tetrahedra (four half tiles) with two warpgroups.  Row r of
// every MMA (lane r of tensor memory, TMEM) belongs to threads r and 128 + r; as in
// dg_stage_kernel, rows 2k and 2k + 1 hold the electric and the magnetic field of one
// tetrahedron (each gives the other field's Phi).  Per row:
//
//   volume:  d_{c'}[(b, i)] = sum_j F_{c'}[j] D_b[i][j]      (3 MMAs chains, K = Np, N = 3 Np)
//   lift:    L_c[i]        = sum_k f_c[k] LIFT[i][k]        (3 chains, K = 4 Nfp, N = Np)
//
// with F the own field and f the face fluxes of the output field (computed on the
// CUDA cores as in dg_stage_kernel).  The A operands (per-row data) are written to
// TMEM with tcgen05.st; the B operands (reference matrices, shared by all rows)
// are staged in shared memory once per CTA by a bulk copy, in the K-major
// no-swizzle core-matrix layout (8 rows x 16 bytes per core matrix, LBO = 128
// bytes between core matrices along K, SBO between groups of 8 rows).  The chain
// rule with the tetrahedron's affine factors and the curl are applied to the
// derivatives read back from TMEM, on the CUDA cores.
//
// Precision (3xTF32).  Every FP32 value x is split x = hi + lo with hi = x
// rounded to TF32 (10 explicit mantissa bits) and lo = x - hi, of which the tensor
// core reads the leading TF32 bits; a product is hi_a hi_b + lo_a hi_b + hi_a lo_b
// (the lo_a lo_b term, ~2^-22 relative, is dropped), accumulated in FP32 in TMEM.
// The reference matrices are split on the host from double (both parts rounded).
//
// Warpgroup 0 (threads 0 to 127) runs the volume term: it writes the own field's operands,
// reads the derivatives back and applies the chain rule and the curl.  Warpgroup 1 meanwhile
// gathers the neighbour traces and computes the face fluxes, into shared memory.  Both write
// the lift's operands; warpgroup 0 adds the lift to components 0 and 1 and writes their output,
// warpgroup 1 component 2's.  One warpgroup doing all of this in turn took 10.2 us for a lone
// CTA (one warp per scheduler issuing 4,200 dependent instructions, 18% of the issue slots) and
// 13.3 us per stage of 12,288 P3 tetrahedra; two take 7.8 us and 12.0 us.
//
// An MMA takes 33 (N = 64) or 18 cycles (N = 32) when its operands are uniform registers of a
// converged warp and one elected lane issues it; issued from a branch for one lane, whose registers
// the hardware has to make uniform first, it took 118 and 61, more than everything else a warp does.
//
// Synchronisation.  The contractions run in four batches: volume of components 0 and 1, volume
// of 2, lift of 0 and 1, lift of 2.  The warps that write a batch's operands arrive on its
// rdy[], its MMAs are committed to its done[].  Volume component 2 uses component 0's columns
// again; then, all derivatives being read and all fluxes computed (one barrier of the CTA), the
// lift lays the columns out anew: three accumulators and two operands, component 2's in the
// place of component 0's once that has been read.  256 columns are held, so two CTAs share an
// SM.  All waits on mbarriers are bounded (about one second of %globaltimer), after which the
// CTA records CMCG_ERR_DEVICE_TIMEOUT in a.err, skips the dependent work, frees its TMEM and
// returns.  TMEM is allocated after the grid-dependency wait, so a CTA that starts early under
// programmatic dependent launch never holds TMEM while the previous stage still runs; the bulk
// copy of the reference matrices is issued before that wait.

constexpr int TC_ROWS = 128;
constexpr int TC_THREADS = 2 * TC_ROWS;
constexpr int TC_TETS = 64;
constexpr int TC_KV = (NPQ + 7) / 8 * 8;              // volume K (nodes), padded to the MMA K of 8
constexpr int TC_KL = (4 * NFPQ + 7) / 8 * 8;         // lift K (face nodes f Nfp + jf)
// Accumulator columns.  Volume: the derivatives of node i along b = 0, 1, 2 are neighbours, five
// nodes to a block of 16 columns (one TMEM load).  Lift: column i.
constexpr int TC_PER = NPQ < 5 ? NPQ : 5;
constexpr int TC_NV = NPQ / TC_PER * 16;
constexpr int TC_NL = (NPQ + 15) / 16 * 16;
static_assert(NPQ % TC_PER == 0, "whole blocks");
__host__ __device__ constexpr int tc_vcol(int b, int i) { return i / TC_PER * 16 + i % TC_PER * 3 + b; }
// TMEM columns.  Volume: buffer b at b TC_COLS / 2, its accumulator [0, NV) and its operand, hi
// [NV, NV + KV) and lo [NV + KV, NV + 2 KV).  Lift: accumulator of component c at c NL, operands 0
// and 1 (hi, then lo, KL columns each) behind the accumulators; component 2 uses operand 0.
constexpr int TC_LIFT_A = 3 * TC_NL;
constexpr int TC_NEED = 2 * (TC_NV + 2 * TC_KV) > TC_LIFT_A + 4 * TC_KL ? 2 * (TC_NV + 2 * TC_KV) : TC_LIFT_A + 4 * TC_KL;
constexpr int TC_COLS = TC_NEED <= 128 ? 128 : 256;
static_assert(TC_NEED <= TC_COLS, "two CTAs per SM need at most 256 TMEM columns each");

// Reference matrices for the MMAs (B operands), split hi / lo, in the core-matrix
// layout: [BV hi | BV lo | BL hi | BL lo], BV = NV x KV, BL = NL x KL (row-major
// in (n, k) through tc_cm_offset).  Written by upload_constants.
constexpr int TC_BV_BYTES = TC_NV * TC_KV * 4;
constexpr int TC_BL_BYTES = TC_NL * TC_KL * 4;
constexpr int TC_B_BYTES = 2 * TC_BV_BYTES + 2 * TC_BL_BYTES;
__device__ __align__(128) uint32_t gTcB[TC_B_BYTES / 4];

// Byte offset of element (row n, column k) of an (rows x K) K-major operand.
__host__ __device__ constexpr int tc_cm_offset(int n, int k, int K) {
  return ((n >> 3) * (K >> 2) + (k >> 2)) * 128 + (n & 7) * 16 + (k & 3) * 4;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: start address, LBO, SBO (bytes), no swizzle.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}

// Instruction descriptor of kind::tf32: D f32, A and B tf32, both K-major, M x N.
__host__ __device__ constexpr uint32_t tc_idesc(int m, int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(n >> 3) << 17) | (uint32_t(m >> 4) << 24);
}

// Round an FP32 bit pattern to TF32 (nearest, ties away from zero).
__device__ __forceinline__ uint32_t tf32_rn(uint32_t u) { return (u + 0x1000u) & 0xFFFFE000u; }
// x = hi + lo with hi = x rounded to TF32 and lo = x - hi exactly (|lo| <= 2^-11 |x|); the
// tensor core reads lo's leading TF32 bits (it truncates), which keeps hi + lo within 2^-21 |x|.
__device__ __forceinline__ void tf32_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = tf32_rn(__float_as_uint(x));
  lo = __float_as_uint(x - __uint_as_float(hi));
}

__device__ __forceinline__ void tmem_st8(uint32_t addr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(addr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&f)[16]) {
  uint32_t v[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(addr)
      : "memory");
#pragma unroll
  for (int k = 0; k < 16; ++k) f[k] = __uint_as_float(v[k]);
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// One MMA D[tmem d] (+)= A[tmem a] B[smem desc b]^T, M = 128, by one elected lane of a converged warp.
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, e;\nelect.sync _|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
      "@e tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Waits until the mbarrier completes phase `parity`; false after about one second.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  const uint64_t t0 = globaltimer();
  for (;;) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (globaltimer() - t0 > 1000000000ull) return false;
  }
}

// Reductions over the CTA (its warps arrive from their own code paths).
__device__ __forceinline__ bool cta_and(bool x) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, 3, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(uint32_t(x)), "n"(TC_THREADS)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ bool cta_or(bool x) { return !cta_and(!x); }

// Zero-padded K-column operand at TMEM address addr, split hi / lo: value k is val(k) for k < n.
// Columns [K0, K1) of it.
template <int K, int K0, int K1, typename Val>
__device__ __forceinline__ void tc_store_operand(uint32_t addr, int n, Val&& val) {
#pragma unroll
  for (int k0 = K0; k0 < K1; k0 += 8) {
    uint32_t hi[8], lo[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k0 + k < n) {
        tf32_split(val(k0 + k), hi[k], lo[k]);
      } else {
        hi[k] = 0u;
        lo[k] = 0u;
      }
    }
    tmem_st8(addr + k0, hi);
    tmem_st8(addr + K + k0, lo);
  }
}

// The MMAs of NC contractions in turn (one warp): D = A_lo B_hi + A_hi B_lo + A_hi B_hi over the K
// steps, then a commit to the mbarrier `bar` (also when skipped, so that waiters are released).
// Contraction x: accumulator d + x dd, operand hi ahi + x da; bhi: shared address of the B operand's
// hi part, its lo part blo bytes behind.
template <int K, int NC>
__device__ __forceinline__ void tc_issue(uint32_t d, uint32_t dd, uint32_t ahi, uint32_t da, uint32_t b, uint32_t blo,
                                         uint32_t idesc, uint32_t bar, bool go) {
  if (go) {
    constexpr uint32_t sbo = uint32_t(K / 4) * 128;
#pragma unroll
    for (int s = 0; s < K / 8; ++s) {
      const uint64_t bh = tc_desc(b + 256 * s, 128, sbo), bl = tc_desc(b + blo + 256 * s, 128, sbo);
#pragma unroll
      for (int x = 0; x < NC; ++x) tc_mma(d + x * dd, ahi + x * da + K + 8 * s, bh, idesc, s > 0 ? 1u : 0u);
#pragma unroll
      for (int x = 0; x < NC; ++x) tc_mma(d + x * dd, ahi + x * da + 8 * s, bl, idesc, 1u);
#pragma unroll
      for (int x = 0; x < NC; ++x) tc_mma(d + x * dd, ahi + x * da + 8 * s, bh, idesc, 1u);
    }
  }
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar)
      : "memory");
}

// The warp's part of an operand is written (and its reads of the accumulator are done).
__device__ __forceinline__ void tc_ready(uint32_t bar) {
  asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
  tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

template <int MINB>
__global__ void __launch_bounds__(TC_THREADS, MINB) dg_stage_tc(const StageArgs<float> a) {
  using R = float;
  constexpr int NP = NPQ, NFP = NFPQ;
  constexpr FaceTab FM = make_fmask(CMCG_Q);
  constexpr int KM = (TC_KL / 8 + 1) / 2 * 8;  // lift operand columns written by warpgroup 0, the rest by 1
  const int tid = threadIdx.x, wg = tid >> 7, row = tid & 127, warp = row >> 5, l = tid & 31, half = l & 1;
  const int64_t ht = int64_t(a.flip ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * (TC_ROWS / 32) + warp;
  const bool in_range = ht * HTILE < a.nti;  // warp-uniform

  // Batches 0, 1: volume of own components 0 and 1, then 2; 2, 3: lift of output components 0 and 1, then 2.
  __shared__ __align__(8) uint64_t bars[9];  // reference matrices; rdy[4]; done[4]
  __shared__ uint32_t tmem_base;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sB = smem_raw;                               // TC_B_BYTES
  R* fl = reinterpret_cast<R*>(smem_raw + TC_B_BYTES) + row;  // traces, then fluxes: component c of face node k at (c 4 Nfp + k) TC_ROWS
  R* ph = fl + 4 * NFP * 3 * TC_ROWS;                         // the volume term of component 2
  const bool jpre = a.j && a.nharm <= 0;

  int prob = 0;
  StageCoef<R> cf;
  cf.active = 0;
  if (in_range) {
    prob = a.tprob ? a.tprob[ht >> 1] : 0;
    cf = a.coef[prob];
  }
  bool live = in_range && cf.active;
  if (!cta_or(live)) return;  // CTA-uniform
  const uint32_t barB = smem_addr(&bars[0]), rdy = smem_addr(&bars[1]), done = smem_addr(&bars[5]);
  const uint32_t sb = smem_addr(sB);
  // The reference matrices (written only at handle creation) are copied before the grid
  // dependency: one bulk copy, completion counted in bytes on barB.
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(barB));
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(rdy + 8 * x), "r"(x < 2 ? 4 : 8));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(done + 8 * x));
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(barB), "r"(TC_B_BYTES) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(sb),
        "l"(gTcB), "r"(TC_B_BYTES), "r"(barB)
        : "memory");
  }

  // A warp without a half tile takes half tile 0's geometry and neighbours, and stores nothing.
  const int64_t hr = in_range ? ht : 0;
  const int64_t own = hr * HS + l;  // the thread's field; its output is the partner's, own ^ 1
  const R* gs = a.geo + hr * GEO32 + (l >> 1);
  const R* gp = a.geo + hr * GEO32 + GEO_S32 * 16 + l;
  uint32_t tmem = 0, trow = 0;  // this CTA's columns, this warp's lanes of them
  // Batch x's MMAs, by the warp that calls this (all operands warp-uniform).
  auto issue = [&](int x, bool ok) -> bool {
    ok = mbar_wait(barB, 0) && ok;
    ok = mbar_wait(rdy + 8 * x, 0) && ok;
    tc_fence_after();
    const bool go = __all_sync(0xffffffffu, ok);
    const uint32_t t = __shfl_sync(0xffffffffu, tmem, 0);
    constexpr uint32_t IV = tc_idesc(128, TC_NV), IL = tc_idesc(128, TC_NL), H = TC_COLS / 2, SL = 2 * TC_BV_BYTES;
    if (x == 0) tc_issue<TC_KV, 2>(t, H, t + TC_NV, H, sb, TC_BV_BYTES, IV, done + 8 * x, go);
    if (x == 1) tc_issue<TC_KV, 1>(t, 0, t + TC_NV, 0, sb, TC_BV_BYTES, IV, done + 8 * x, go);
    if (x == 2) tc_issue<TC_KL, 2>(t, TC_NL, t + TC_LIFT_A, 2 * TC_KL, sb + SL, TC_BL_BYTES, IL, done + 8 * x, go);
    if (x == 3) tc_issue<TC_KL, 1>(t + 2 * TC_NL, 0, t + TC_LIFT_A, 0, sb + SL, TC_BL_BYTES, IL, done + 8 * x, go);
    return ok;
  };
  const bool first = __shfl_sync(0xffffffffu, warp, 0) == 0;  // the warpgroup's first warp
  // Columns of the lift operand of component c (value k: flux k of the row), the warpgroup's share.
  auto store_lift = [&](int c) {
    const uint32_t addr = trow + TC_LIFT_A + (c == 1 ? 2 * TC_KL : 0);
    auto flux = [&](int k) { return fl[(c * 4 * NFP + k) * TC_ROWS]; };
    if (wg == 0) tc_store_operand<TC_KL, 0, KM>(addr, 4 * NFP, flux);
    else tc_store_operand<TC_KL, KM, TC_KL>(addr, 4 * NFP, flux);
  };
  // Component c: the lift added to the volume term p, data, filter, output.
  auto finish = [&](int c, R (&p)[NP], const R (&bv)[NP], const R (&jv)[NP], R sigma) {
#pragma unroll
    for (int k0 = 0; k0 < TC_NL; k0 += 16) {
      float t16[16];
      tmem_ld16(trow + c * TC_NL + k0, t16);
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (i / 16 * 16 == k0) p[i] += t16[i % 16];
    }
    if (!live) return;  // warp-uniform
    add_data<R, NP>(p, jv, a, cf, own, c, 0, half, sigma);
    if (a.fre) accumulate_filter<R, NP>(a, cf, p, own, c, 0);  // forward sweeps with the filter only
    if (a.out) {
#pragma unroll
      for (int n = 0; n < NP; ++n) a.out[(own ^ 1) + (c * NP + n) * 32] = bv[n] + cf.c_out * p[n];
    }
  };
  auto load_base = [&](R (&bv)[NP], int c) {
    if (a.out) {
#pragma unroll
      for (int n = 0; n < NP; ++n) bv[n] = a.base[(own ^ 1) + (c * NP + n) * 32];
    }
  };
  // Both warpgroups: fluxes computed, derivatives read.
  auto middle = [&]() {
    tc_fence_before();
    asm volatile("barrier.cta.sync 1, 256;\n" ::: "memory");
    tc_fence_after();
  };

  if (wg == 1) {
    // ---- warpgroup 1: neighbour traces, face fluxes
    Neighbour<R> nb[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      nb[f] = find_neighbour(a, hr, l, f);
      asm volatile("" : "+l"(nb[f].at), "+l"(nb[f].nodes));  // looked up before the wait
    }
    grid_dep_wait();
    grid_dep_launch();
    if (live && a.pactive && !a.pactive[prob]) live = false;  // CG converged (written by the CG kernels)
    if (!cta_or(live)) return;
    // Traces of a face two faces ahead of its fluxes, each face a group of copies.
    auto copy_face = [&](int f) {
      const R* p = a.vin + nb[f].at;
#pragma unroll
      for (int jf = 0; jf < NFP; ++jf) {
        const R* q = p + (unsigned(nb[f].nodes >> (5 * jf)) & 31u) * 32u;
#pragma unroll
        for (int c = 0; c < 3; ++c) cp_async_4(fl + (c * 4 * NFP + f * NFP + jf) * TC_ROWS, q + c * NP * 32);
      }
      cp_async_commit();
    };
    copy_face(0);
    R v[3][NP];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < NP; ++n) v[c][n] = a.vin[own + (c * NP + n) * 32];
    copy_face(1);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      if (f < 3) cp_async_wait<1>();
      else cp_async_wait<0>();
      if (f + 2 < 4) copy_face(f + 2 < 4 ? f + 2 : 0);
      const R n0 = gs[(9 + 3 * f) * 16], n1 = gs[(10 + 3 * f) * 16], n2 = gs[(11 + 3 * f) * 16];
      const R k1 = gp[(1 + 2 * f) * 32] * a.sH, k2 = gp[(2 + 2 * f) * 32];
      const R m0 = k1 * n0, m1 = k1 * n1, m2 = k1 * n2;  // k1 n, once per face
#pragma unroll
      for (int g = 0; g < NFP; g += 5) {  // five nodes at a time: independent chains
        R X[3][5], Y[3][5];
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (g + j < NFP)
#pragma unroll
            for (int c = 0; c < 3; ++c)
              X[c][j] = fmaf(nb[f].c, fl[(c * 4 * NFP + f * NFP + g + j) * TC_ROWS], -v[c][FM.v[f][g + j]]);
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (g + j < NFP)
#pragma unroll
            for (int c = 0; c < 3; ++c) Y[c][j] = __shfl_xor_sync(0xffffffffu, X[c][j], 1);
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (g + j < NFP) {
            const R nY = n0 * Y[0][j] + n1 * Y[1][j] + n2 * Y[2][j];
            R* s = fl + (f * NFP + g + j) * TC_ROWS;
            s[0 * 4 * NFP * TC_ROWS] = (m1 * X[2][j] - m2 * X[1][j]) + k2 * (Y[0][j] - n0 * nY);
            s[1 * 4 * NFP * TC_ROWS] = (m2 * X[0][j] - m0 * X[2][j]) + k2 * (Y[1][j] - n1 * nY);
            s[2 * 4 * NFP * TC_ROWS] = (m0 * X[1][j] - m1 * X[0][j]) + k2 * (Y[2][j] - n2 * nY);
          }
      }
    }
    middle();
    tmem = tmem_base;
    trow = tmem + (uint32_t(warp * 32) << 16);
    store_lift(0);
    store_lift(1);
    tc_ready(rdy + 8 * 2);
    R bv[NP];
    load_base(bv, 2);
    bool ok = true;
    if (first) ok = issue(2, ok);
    ok = mbar_wait(done + 8 * 2, 0) && ok;  // component 0's operand has been read
    tc_fence_after();
    store_lift(2);
    tc_ready(rdy + 8 * 3);
    if (first) ok = issue(3, ok);
    R p[NP], jv[NP];
    if (jpre) load_source<R, NP>(jv, a.j + own, 2, 0);
#pragma unroll
    for (int n = 0; n < NP; ++n) p[n] = ph[n * TC_ROWS];
    ok = mbar_wait(done + 8 * 3, 0) && ok;
    tc_fence_after();
    if (ok) finish(2, p, bv, jv, a.sigma ? gp[GEO_SIGMA * 32] : R(0));
    tc_fence_before();
    cta_and(ok);
    return;
  }

  // ---- warpgroup 0: volume, output
  R G[9];
  const R sv = gp[0] * a.sH;
#pragma unroll
  for (int m = 0; m < 9; ++m) G[m] = gs[m * 16] * sv;  // the material factor of Phi, folded into the chain rule
  const R sigma = a.sigma ? gp[GEO_SIGMA * 32] : R(0);
  grid_dep_wait();
  grid_dep_launch();
  if (live && a.pactive && !a.pactive[prob]) live = false;
  if (!cta_or(live)) {
    if (tid == 0) mbar_wait(barB, 0);  // the copy lands before the CTA's shared memory is released
    return;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&tmem_base)),
                 "r"(TC_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  R v[2][NP];  // the own field, component 2 in place of component 0's
  auto load_own = [&](int b, int c) {
#pragma unroll
    for (int n = 0; n < NP; ++n) v[b][n] = a.vin[own + (c * NP + n) * 32];
  };
  load_own(0, 0);
  load_own(1, 1);
  tc_fence_before();
  asm volatile("barrier.cta.sync 2, 128;\n" ::: "memory");  // TMEM address and mbarrier initialisation visible
  tc_fence_after();
  tmem = tmem_base;
  trow = tmem + (uint32_t(warp * 32) << 16);

  R phi[3][NP];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int i = 0; i < NP; ++i) phi[c][i] = R(0);
  // Volume result of own component cp (buffer b): derivatives along r, s, t, chain rule, curl.
  auto read_vol = [&](int b, int cp) {
    // curl F: component 0 = d1 F2 - d2 F1, 1 = d2 F0 - d0 F2, 2 = d0 F1 - d1 F0
    const int ap = cp == 0 ? 2 : cp == 1 ? 0 : 1;   // axis whose derivative enters with +
    const int am = cp == 0 ? 1 : cp == 1 ? 2 : 0;   // axis whose derivative enters with -
    const int cpl = cp == 0 ? 1 : cp == 1 ? 2 : 0;  // output component receiving + d_ap F_cp
    const int cmi = cp == 0 ? 2 : cp == 1 ? 0 : 1;  // output component receiving - d_am F_cp
#pragma unroll
    for (int i0 = 0; i0 < NP; i0 += TC_PER) {
      float d[16];
      tmem_ld16(trow + b * (TC_COLS / 2) + tc_vcol(0, i0), d);
#pragma unroll
      for (int i = i0; i < i0 + TC_PER; ++i) {
        const R d0 = d[3 * (i - i0)], d1 = d[3 * (i - i0) + 1], d2 = d[3 * (i - i0) + 2];
        phi[cpl][i] = fmaf(G[2 * 3 + ap], d2, fmaf(G[1 * 3 + ap], d1, fmaf(G[0 * 3 + ap], d0, phi[cpl][i])));
        phi[cmi][i] = fmaf(-G[2 * 3 + am], d2, fmaf(-G[1 * 3 + am], d1, fmaf(-G[0 * 3 + am], d0, phi[cmi][i])));
      }
    }
  };
  auto store_vol = [&](int b) {
    tc_store_operand<TC_KV, 0, TC_KV>(trow + b * (TC_COLS / 2) + TC_NV, NP, [&](int k) { return v[b][k]; });
  };
  store_vol(0);
  store_vol(1);
  tc_ready(rdy + 8 * 0);
  load_own(0, 2);
  bool ok = true;
  if (first) ok = issue(0, ok);
  ok = mbar_wait(done + 8 * 0, 0) && ok;
  tc_fence_after();
  store_vol(0);  // the operand has been read; the accumulator is read before the next MMAs are issued
  if (ok) read_vol(0, 0);
  tc_ready(rdy + 8 * 1);
  if (first) ok = issue(1, ok);
  if (ok) read_vol(1, 1);
  ok = mbar_wait(done + 8 * 1, 0) && ok;
  tc_fence_after();
  if (ok) read_vol(0, 2);
#pragma unroll
  for (int n = 0; n < NP; ++n) ph[n * TC_ROWS] = phi[2][n];

  middle();
  store_lift(0);
  store_lift(1);
  tc_ready(rdy + 8 * 2);
  R bv[2][NP];
  load_base(bv[0], 0);
  load_base(bv[1], 1);
  R jv[NP];
  if (jpre) load_source<R, NP>(jv, a.j + own, 0, 0);
  ok = mbar_wait(done + 8 * 2, 0) && ok;
  tc_fence_after();
  store_lift(2);
  tc_ready(rdy + 8 * 3);
  if (ok) {
    finish(0, phi[0], bv[0], jv, sigma);
    if (jpre) load_source<R, NP>(jv, a.j + own, 1, 0);
    finish(1, phi[1], bv[1], jv, sigma);
  }
  // Free TMEM (every thread's TMEM reads are complete).
  tc_fence_before();
  ok = cta_and(ok);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TC_COLS));
  }
  if (!ok && tid == 0 && a.err) atomicOr(a.err, 1);
}

// Dynamic shared memory of dg_stage_tc: reference matrices, traces / fluxes, the volume term of
// component 2.
constexpr size_t tc_smem() { return size_t(TC_B_BYTES) + size_t(4 * NFPQ * 3 + NPQ) * TC_ROWS * sizeof(float); }
// Resident CTAs per SM that the TMEM columns allow (512 per SM).
constexpr int TC_MINB = 2;

// The MMA operands of the reference matrices, split hi / lo from double, in the
// core-matrix layout of tc_cm_offset.
void tc_upload_reference(const RefMats& rm) {
  const int np = rm.np, nfp = rm.nfp;
  std::vector<uint32_t> buf(TC_B_BYTES / 4, 0u);
  auto rn = [](double x) -> uint32_t {  // round to TF32 (nearest) through FP32
    const float f = static_cast<float>(x);
    uint32_t u;
    std::memcpy(&u, &f, 4);
    return (u + 0x1000u) & 0xFFFFE000u;
  };
  auto put = [&](int base_bytes, int n, int k, int K, double x) {
    const uint32_t hi = rn(x);
    float fh;
    std::memcpy(&fh, &hi, 4);
    const uint32_t lo = rn(x - double(fh));
    buf[(base_bytes + tc_cm_offset(n, k, K)) / 4] = hi;
    buf[(base_bytes + (base_bytes == 0 ? TC_BV_BYTES : TC_BL_BYTES) + tc_cm_offset(n, k, K)) / 4] = lo;
  };
  const std::vector<double>* D[3] = {&rm.Dr, &rm.Ds, &rm.Dt};
  for (int b = 0; b < 3; ++b)
    for (int i = 0; i < np; ++i)
      for (int j = 0; j < np; ++j) put(0, tc_vcol(b, i), j, TC_KV, (*D[b])[size_t(i) * np + j]);
  for (int i = 0; i < np; ++i)
    for (int k = 0; k < 4 * nfp; ++k) put(2 * TC_BV_BYTES, i, k, TC_KL, rm.LIFT[size_t(i) * 4 * nfp + k]);
  cudaMemcpyToSymbol(gTcB, buf.data(), buf.size() * 4);
}
