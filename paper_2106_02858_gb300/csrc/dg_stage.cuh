// One explicit Runge-Kutta stage of the DG time-domain Maxwell scheme, for a
// fixed polynomial order CMCG_Q (included once per order by dg_q{1,2,3}.cu).
//
// Two lanes (2t, 2t + 1) share tetrahedron t of a half tile of 16: the even lane holds
// the electric field of K and computes Phi_H, the odd lane holds the magnetic field and
// computes Phi_E:
//
//   Phi_H =  mu^{-1} curl E + LIFT . fH,    Phi_E = -eps^{-1} curl H + LIFT . fE
//
// (Eq. ode_system: Phi(t, U) = Re(J e^{i w t}) + B U, strong form of the 3D upwind DG
// operator generalising Eq. DG_semidiscrete).  The curl of a thread's own field is all its
// volume term needs.  Face terms use jumps dE = E^+ - E^-, dH = H^+ - H^-; each thread
// forms the jump of its own field and the partner's arrives by lane shuffles.  With X its
// own jump and Y the partner's,
//
//   f = k1 (n x X) + k2 (Y - n (n . Y)),
//   (k1, k2) = (bH, aH) on the E lane  ->  fH = bH n x dE + aH dH_t,
//   (k1, k2) = (-bE, aE) on the H lane ->  fE = aE dE_t - bE n x dH,
//   aE = fscale / (eps (Z^- + Z^+)), bE = Z^+ aE, aH = fscale / (mu (Y^- + Y^+)), bH = Y^+ aH,
//
// which is -n x (H^ - H^-) and n x (E^ - E^-) for the upwind traces
// E^ = (Y^- E^- + Y^+ E^+ - (H^- - H^+) x n) / (Y^- + Y^+),
// H^ = (Z^- H^- + Z^+ H^+ + (E^- - E^+) x n) / (Z^- + Z^+);
// fscale folds the block-diagonal inverse mass into the lift.
//
// A boundary face names its own trace as its neighbour, and X = c tr - v with c = 1
// (interior), c = -1 | 1 (PEC mirror dE = -2 E^-, dH = 0) or c = 0 (impedance: zero outer
// state), so that every face node runs the same instructions.  The adjoint stage (Section
// 4.1.2, P* = Sigma P Sigma) flips the sign of every magnetic value read and of Phi_H: sH on
// the curl and on k1, no memory pass.
//
// Fields, geometry and data are laid out so that a warp's load is one line (field_at, GEO).
// FP32 fields are nodal values (dg_stage_nodal.cuh; P3 also dg_stage_tc.cuh), FP64 fields
// Bernstein coefficients (dg_stage_bern.cuh).
//
// SPLIT warps share a half tile, each with its share of the faces' fluxes and of the output
// values.  SPLIT > 1 shortens a warp's chain where a mesh is too small to fill the SMs.
#pragma once

#include <cstring>

#include "bernstein.h"

#ifndef CMCG_Q
#error "define CMCG_Q before including dg_stage.cuh"
#endif

namespace cmcg {
namespace {

constexpr int NPQ = np_of(CMCG_Q);
constexpr int NFPQ = nfp_of(CMCG_Q);
constexpr int HS = 96 * NPQ;  // values of a half tile of a field vector

// Own face node jf is node (cNB[face << 3 | perm] >> 5 jf) & 31 of the neighbour.
__constant__ unsigned long long cNB[4 * 8];

// Programmatic dependent launch: a stage may be launched while the previous
// stage is still running (once all its blocks are resident); before
// grid_dep_wait(), which returns once the previous grid has completed and its
// writes are visible, it reads only data that no kernel writes (geometry,
// neighbour codes, coefficient tables, tile problems).
// Without the launch attribute both are no-ops.
// The next stage may start its blocks: called first by grids of more blocks than SMs (81,648 P2
// tetrahedra 14.6 ms a sweep when called later, 14.4 so), by smaller ones after the grid dependency's
// wait, so that at most one stage waits.  There, called first, several stages pile up, and their
// waiting blocks make running ones double up on some SMs with others idle (sweeps: P2 FP32 1,296
// tetrahedra 994 us, 810 so; 2,058 1,378 and 1,015; P1 FP64 1,296 1,602 and 752).  The tensor-core
// stage calls it after the wait at every size (12,288 P3 tetrahedra: within 1% of calling it first).
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

__device__ __forceinline__ void cp_async_4(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_16(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Every sum of products here, in dg_stage_nodal.cuh and in dg_stage_bern.cuh is written as fma: what the
// compiler would fuse by itself may differ between the forms, which have to give the same bits.
//
// The conductivity, source and impedance-face terms of Phi on the output values n0 .. n0 + NN - 1
// of the thread (own: its place in the field layout, the partner's is own ^ 1).  The source on the
// E rows is, at the stage time, Re(J e^{i w t}) = s_cos J_re - s_sin J_im, or, in a sweep driven at
// several harmonics of a base frequency (a.nharm > 0), the sum over the harmonics of hcs[2h] J_re,h
// - hcs[2h+1] J_im,h.  The even lane reads J_re and the odd lane J_im, as one line (jv: already read,
// single frequency), and the odd lane, which computes Phi_E, adds both.
template <typename R, int NN>
__device__ __forceinline__ void load_source(R (&jv)[NN], const R* j, int c, int n0) {
#pragma unroll
  for (int n = 0; n < NN; ++n) jv[n] = j[(c * NPQ + n0 + n) * 32];
}
template <typename R, int NN>
__device__ __forceinline__ void add_source(R (&phi)[NN], const R (&jv)[NN], R cs, R sn, int half) {
#pragma unroll
  for (int n = 0; n < NN; ++n) {
    const R re = __shfl_xor_sync(0xffffffffu, jv[n], 1);
    if (half) phi[n] += fma(cs, re, -(sn * jv[n]));
  }
}
// Component c.
template <typename R, int NN>
__device__ __forceinline__ void add_data(R (&phi)[NN], const R (&jv)[NN], const StageArgs<R>& a, const StageCoef<R>& cf,
                                         int64_t own, int c, int n0, int half, R sigma) {
  const int64_t off = (own ^ 1) + (c * NPQ + n0) * 32;
  if (a.sigma && half) {  // Phi_E -= (sigma / eps) E (E is not flipped by Sigma)
#pragma unroll
    for (int n = 0; n < NN; ++n) phi[n] = fma(sigma, -a.vin[off + n * 32], phi[n]);
  }
  if (a.j) {
    if (a.nharm <= 0) {
      add_source<R, NN>(phi, jv, cf.s_cos, cf.s_sin, half);
    } else {
#pragma unroll 1
      for (int hh = 0; hh < a.nharm; ++hh) {
        R jh[NN];
        load_source<R, NN>(jh, a.j + hh * a.jstride + own, c, n0);
        add_source<R, NN>(phi, jh, a.hcs[2 * hh], a.hcs[2 * hh + 1], half);
      }
    }
  }
  if (a.bre) {  // impedance-face data, lifted (source sweeps only)
#pragma unroll
    for (int n = 0; n < NN; ++n) phi[n] += fma(cf.s_cos, a.bre[off + n * 32], -(cf.s_sin * a.bim[off + n * 32]));
  }
}

// The on-the-fly filter on component c of this thread's output values i0 .. i0 + NN - 1 (forward
// sweeps with the filter, first nested stage of each step): F += fa U + fb Phi.  A batch of rows of
// U and F is loaded before any of it is stored: vin, fre and fim are not known to be distinct, and a
// row-by-row read-modify-write would put every load behind the previous row's stores.
template <typename R, int NN>
__device__ __forceinline__ void accumulate_filter(const StageArgs<R>& a, const StageCoef<R>& cf, const R (&phi)[NN],
                                                  int64_t own, int c, int i0) {
  const int64_t off = (own ^ 1) + (c * NPQ + i0) * 32;
#pragma unroll
  for (int n0 = 0; n0 < NN; n0 += 10) {  // ten rows at a time
    R u[10], fr[10], fi[10];
#pragma unroll
    for (int n = 0; n < 10; ++n)
      if (n0 + n < NN) {
        u[n] = a.vin[off + (n0 + n) * 32];
        fr[n] = a.fre[off + (n0 + n) * 32];
        fi[n] = a.fim[off + (n0 + n) * 32];
      }
#pragma unroll
    for (int n = 0; n < 10; ++n)
      if (n0 + n < NN) {
        a.fre[off + (n0 + n) * 32] = fr[n] + fma(cf.fa_re, u[n], cf.fb_re * phi[n0 + n]);
        a.fim[off + (n0 + n) * 32] = fi[n] + fma(cf.fa_im, u[n], cf.fb_im * phi[n0 + n]);
      }
  }
}

// A face's neighbour: place of its value 0 of component 0 in a field vector, its face nodes, and
// the weight of its trace in the jump.
template <typename R>
struct Neighbour {
  int64_t at;
  unsigned long long nodes;
  R c;
};
template <typename R>
__device__ __forceinline__ Neighbour<R> find_neighbour(const StageArgs<R>& a, int64_t ht, int l, int f) {
  const int half = l & 1;
  const int32_t code = a.nbr[(ht * 4 + f) * 16 + (l >> 1)];
  const int perm = code & 7;
  Neighbour<R> n;
  n.c = perm < PERM_PEC ? R(1) : perm == PERM_IMP ? R(0) : half ? R(1) : R(-1);
  n.at = field_at(NPQ, code >> 5, half, 0, 0);
  n.nodes = cNB[code & 31];
  return n;
}
template <typename R>
__device__ __forceinline__ void load_trace(R (&tr)[3][NFPQ], const R* vin, const Neighbour<R>& nb) {
  const R* v = vin + nb.at;
#pragma unroll
  for (int n = 0; n < NFPQ; ++n) {
    const R* p = v + (unsigned(nb.nodes >> (5 * n)) & 31u) * 32u;
#pragma unroll
    for (int c = 0; c < 3; ++c) tr[c][n] = p[c * NPQ * 32];
  }
}

#include "dg_stage_bern.cuh"
#include "dg_stage_nodal.cuh"

template <int SPLIT, int P>
__device__ __forceinline__ void stage_part(const StageArgs<double>& a, int64_t ht, int l, int warp, double* xs) {
  bern_part<SPLIT, P>(a, ht, l, warp, xs);
}
template <int SPLIT, int P>
__device__ __forceinline__ void stage_part(const StageArgs<float>& a, int64_t ht, int l, int warp, float* xs) {
  nodal_part<SPLIT, P>(a, ht, l, warp, xs);
}

// WARPS warps per block; MINB: minimum resident blocks per SM requested from the compiler (caps
// registers at 65536 / (32 WARPS MINB)).  The forms are timed per handle (see api.cu).
template <typename R, int SPLIT, int WARPS, int MINB>
__global__ void __launch_bounds__(32 * WARPS, MINB) dg_stage_kernel(const StageArgs<R> a) {
  if (gridDim.x > unsigned(a.nsm)) grid_dep_launch();
  const int warp = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int64_t ht = (int64_t(a.flip ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * WARPS + warp) / SPLIT;
  if (ht * HTILE >= a.nti) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* xs = reinterpret_cast<R*>(smem_raw);
  if constexpr (SPLIT == 1) {
    stage_part<1, 0>(a, ht, l, warp, xs);
  } else if constexpr (SPLIT == 2) {
    if (warp & 1) stage_part<2, 1>(a, ht, l, warp, xs);
    else stage_part<2, 0>(a, ht, l, warp, xs);
  } else {
    switch (warp & 3) {
      case 0: stage_part<4, 0>(a, ht, l, warp, xs); break;
      case 1: stage_part<4, 1>(a, ht, l, warp, xs); break;
      case 2: stage_part<4, 2>(a, ht, l, warp, xs); break;
      default: stage_part<4, 3>(a, ht, l, warp, xs); break;
    }
  }
}

#include "dg_stage_tc.cuh"

// Dynamic shared memory: what the warps of a half tile exchange (FP64, SPLIT > 1), or geometry and base
// rows or fluxes (FP32).
template <typename R, int SPLIT, int WARPS>
constexpr size_t stage_smem() {
  if (sizeof(R) == 8) return SPLIT > 1 ? size_t(WARPS / SPLIT) * BERN_SMEM * 32 * sizeof(R) : 0;
  return size_t(WARPS) * nodal_smem<SPLIT>() * sizeof(R);
}
// Shared memory per block such that no SM takes more blocks than an even spread over the SMs gives it,
// for grids of more blocks than SMs (P1 FP32 24,576 tetrahedra 1,190 us a sweep without it, 1,040 so; 48,000
// 2,121 and 1,889).  Smaller grids are left alone: a whole SM to a block keeps other handles' kernels
// out (four handles of 4,374 P1 tetrahedra on four streams 1.29 ms so, 0.83 without).  P2 and P3 FP32 with two or
// four warps a half tile gain or lose by it (us a sweep without and with, P2 3,072 tetrahedra and four
// warps 1,838 and 1,991, 7,986 and two warps 2,468 and 2,334); the one-warp forms are faster at all these
// sizes (1,311 and 1,890), so they are left alone.  The P3 tensor-core stage takes more than any pad.
constexpr size_t SM_SHARED = 228 * 1024, BLOCK_RESERVED = 1024;
constexpr size_t MAX_DYNAMIC = 96 * 1024;  // above the largest need (P3 tensor cores 94 KB, FP64 73 KB) and pad (77 KB)
inline size_t spread_smem(size_t need, int64_t blocks, int nsm) {
  const int64_t per_sm = (blocks + nsm - 1) / nsm;
  const size_t pad = SM_SHARED / size_t(per_sm + 1) / 128 * 128 + 128 - BLOCK_RESERVED;  // per_sm + 1 such blocks don't fit
  return per_sm > 1 && per_sm < 32 && pad > need && (pad + BLOCK_RESERVED) * size_t(per_sm) <= SM_SHARED ? pad : need;
}
template <typename Arg>
void launch_k(void (*k)(Arg), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s, bool pdl,
              const Arg& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, a);
}

template <typename R, int SPLIT, int WARPS, int MINB>
void launch_form(const StageArgs<R>& a, cudaStream_t s, bool pdl) {
  constexpr bool spread = sizeof(R) == 8 || SPLIT == 1 || CMCG_Q == 1;
  constexpr size_t need = stage_smem<R, SPLIT, WARPS>();
  static_assert(need <= MAX_DYNAMIC, "shared memory");
  const int64_t warps = a.nti / HTILE * SPLIT, blocks = (warps + WARPS - 1) / WARPS;
  launch_k(dg_stage_kernel<R, SPLIT, WARPS, MINB>, unsigned(blocks), 32 * WARPS,
           spread ? spread_smem(need, blocks, a.nsm) : need, s, pdl, a);
}
template <typename R, int SPLIT, int WARPS, int MINB>
void allow_smem() {
  cudaFuncSetAttribute(dg_stage_kernel<R, SPLIT, WARPS, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       int(MAX_DYNAMIC));
}

}  // namespace

template <>
void launch_stage<CMCG_Q, float>(const StageArgs<float>& a, cudaStream_t s, int form, bool pdl) {
  switch (form) {
    case 1: launch_form<float, 1, 4, 4>(a, s, pdl); break;
    case 2: launch_form<float, 1, 4, 6>(a, s, pdl); break;
    case 3: launch_form<float, 2, 4, 3>(a, s, pdl); break;
    case 4: launch_form<float, 2, 4, 4>(a, s, pdl); break;
    case 5: launch_form<float, 4, 4, 4>(a, s, pdl); break;
    case STAGE_FORM_TC:
      launch_k(dg_stage_tc<TC_MINB>, unsigned((a.nti + TC_TETS - 1) / TC_TETS), TC_THREADS,
               spread_smem(tc_smem(), (a.nti + TC_TETS - 1) / TC_TETS, a.nsm), s, pdl, a);
      break;
    default: launch_form<float, 1, 2, 6>(a, s, pdl); break;
  }
}
template <>
void launch_stage<CMCG_Q, double>(const StageArgs<double>& a, cudaStream_t s, int form, bool pdl) {
  switch (form) {
    case 1: launch_form<double, 2, 2, 1>(a, s, pdl); break;
    case 2: launch_form<double, 4, 4, 1>(a, s, pdl); break;
    default: launch_form<double, 1, 4, 1>(a, s, pdl); break;
  }
}

template <>
void upload_constants<CMCG_Q>(const RefMats& rm) {
  // allow dynamic shared memory beyond the 48 KiB default
  allow_smem<float, 1, 2, 6>();
  allow_smem<float, 1, 4, 4>();
  allow_smem<float, 1, 4, 6>();
  allow_smem<float, 2, 4, 3>();
  allow_smem<float, 2, 4, 4>();
  allow_smem<float, 4, 4, 4>();
  allow_smem<double, 1, 4, 1>();
  allow_smem<double, 2, 2, 1>();
  allow_smem<double, 4, 4, 1>();
  cudaFuncSetAttribute(dg_stage_tc<TC_MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(MAX_DYNAMIC));
  cudaFuncSetAttribute(dg_stage_tc<TC_MINB>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       int(cudaSharedmemCarveoutMaxShared));  // two P3 CTAs per SM need 2 x 95 KB
  static_assert(tc_smem() <= MAX_DYNAMIC, "shared memory");
  tc_upload_reference(rm);
  std::vector<float> Df, Lf(rm.LIFT.size());  // LIFT: [node][face node]
  for (size_t k = 0; k < Lf.size(); ++k) Lf[(k % (4 * NFPQ)) * NPQ + k / (4 * NFPQ)] = float(rm.LIFT[k]);
  for (const std::vector<double>* D : {&rm.Dr, &rm.Ds, &rm.Dt}) Df.insert(Df.end(), D->begin(), D->end());
  if (CMCG_Q == 3) cudaMemcpyToSymbol(cD, Df.data(), sizeof(float) * Df.size());
  cudaMemcpyToSymbol(cL, Lf.data(), sizeof(float) * Lf.size());
  unsigned long long nb[4 * 8];
  for (int f = 0; f < 4; ++f)
    for (int p = 0; p < 8; ++p) {
      unsigned long long w = 0;
      for (int n = 0; n < NFPQ; ++n) {
        const int node = p < 6 ? rm.nbrnode[(f * 6 + p) * NFPQ + n] : rm.fmask[f * NFPQ + n];
        w |= (unsigned long long)(node) << (5 * n);
      }
      nb[f * 8 + p] = w;
    }
  cudaMemcpyToSymbol(cNB, nb, sizeof(nb));
}

}  // namespace cmcg
