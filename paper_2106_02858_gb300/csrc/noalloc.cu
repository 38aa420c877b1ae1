// cmcg_inner_noalloc: the (eps, mu)-weighted inner product of two nodal fields
// without any device allocation.
//
// Who needs it: callers that cannot call cudaMalloc at the point where they
// need the inner product -- code that owns all device memory through its own
// pool allocator (a framework's caching allocator), code running between
// stream-ordered work that must not be serialised (cudaMalloc and cudaFree can
// synchronise the device), and callers without a handle, since cmcg_create
// allocates the whole solver state.  The handle-based cmcg_inner reduces
// through a per-handle block-partials buffer allocated by cmcg_create; this
// variant reduces through one file-scope array instead.
//
// The array (NA_BLOCKS doubles, 19 KiB) is static device memory: every
// GPU that loads the library holds it until the process exits.  Host code only
// ever sees a stand-in for its name, so the device address is fetched with
// cudaGetSymbolAddress once per device, with that device current, and passed
// to the kernels.  Every call shares the array and finds the previous call's
// contents in it; nothing needs clearing because every entry a call reads was
// written earlier in the same call.  Calls that overlap on the GPU (two streams,
// or two host threads) race on the array.
#include <mutex>

#include "bernstein.h"

namespace cmcg {
namespace {

constexpr int NA_THREADS = 128;        // one partial per block
// Blocks, at most; larger meshes give every thread of every block the same number of components more: with
// the grid's stride, and the last pass partly idle, the figure below is 79 us instead of 68.
constexpr int NA_BLOCKS = 152 * 16;

static __device__ __align__(256) double g_na_partials[NA_BLOCKS];

// x^T M y of one component's nodal values on the unit tetrahedron.  M commutes with the renumberings
// of the four vertices, so it is a short form in sums that belong to a vertex i: s_i (P2: the midpoints
// of its three edges), a_i, b_i (P3: the near and the far nodes of its three edges), f_i (P3: the node
// of the opposite face), their totals over i, and the plain product over edge nodes, with whole
// coefficients (they follow from the simplex integrals; na_form evaluates P2's first line with 2/5 and
// 7.2 in their place, rounded):
//   P1 (x 120):    sum_i v v' + V V'
//   P2 (x 2520):   sum_i (5 v v' + 2 (v s' + s v') + 8 s s') + V V' - 3 (V S' + S V') + 2 S S' + 8 sum_e e e'
//   P3 (x 26880):  sum_i (14 v v' - 15 (v a' + a v') + 3 (v b' + b v') + 18 (v f' + f v') + 54 a a'
//                  - 27 (a b' + b a') - 54 (a f' + f a') + 216 f f') + 2 V V' + 3 (V A' + A V')
//                  + 18 (V F' + F V') + 216 F F' + 54 sum_e e e'
// 12, 57 and 135 operations where the dense matrix takes 20, 110 and 420: at GB300's FP64 rate (one
// warp instruction per 64 cycles and SM quarter) they bound the kernel, not the bytes.  81,648 P2
// tetrahedra: 131 us with the dense matrix, 68 us so (80 MB of fields; the operations alone 46 us).
// The error against exact sums is below the dense matrix's, whose entries were themselves rounded.
struct NaTab {
  int v[4], near[4][3], far[4][3], f[4], e[12], ne;
};
template <int Q>
constexpr NaTab make_na() {
  NaTab t{};
  for (int i = 0; i < 4; ++i) {
    Bary4 x{{0, 0, 0, 0}};
    x.b[i] = Q;
    t.v[i] = node_at(Q, x);
    int k = 0;
    for (int j = 0; j < 4; ++j) {
      if (j == i || Q == 1) continue;
      Bary4 y{{0, 0, 0, 0}}, z{{0, 0, 0, 0}};
      y.b[i] = Q - 1;
      y.b[j] = 1;
      z.b[j] = Q - 1;
      z.b[i] = 1;
      t.near[i][k] = node_at(Q, y);
      t.far[i][k++] = node_at(Q, z);
      if (Q == 3 || i < j) t.e[t.ne++] = node_at(Q, y);
    }
    Bary4 w{{1, 1, 1, 1}};
    w.b[i] = 0;
    if (Q == 3) t.f[i] = node_at(Q, w);
  }
  return t;
}
template <int Q>
__device__ __forceinline__ double na_form(const double (&x)[np_of(Q)], const double (&y)[np_of(Q)]) {
  constexpr NaTab T = make_na<Q>();
  double ee = 0;
#pragma unroll
  for (int k = 0; k < T.ne; ++k) ee = fma(x[T.e[k]], y[T.e[k]], ee);
  // 5 v v' + 2 (v s' + s v') + 8 s s' = 5 (v + 2/5 s)(v' + 2/5 s') + 7.2 s s', one fma less per vertex
  if constexpr (Q == 2) {
    double ww = 0, ss = 0, VX, VY, SX, SY;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double vx = x[T.v[i]], vy = y[T.v[i]];
      const double sx = x[T.near[i][0]] + x[T.near[i][1]] + x[T.near[i][2]];
      const double sy = y[T.near[i][0]] + y[T.near[i][1]] + y[T.near[i][2]];
      VX = i ? VX + vx : vx;
      VY = i ? VY + vy : vy;
      SX = i ? SX + sx : sx;
      SY = i ? SY + sy : sy;
      ww = fma(fma(0.4, sx, vx), fma(0.4, sy, vy), ww);
      ss = fma(sx, sy, ss);
    }
    const double r = fma(SX, fma(2.0, SY, -3.0 * VY), VX * fma(-3.0, SY, VY));
    return fma(5.0, ww, fma(7.2, ss, fma(8.0, ee, r))) * (1.0 / 2520);
  }
  double VX = 0, VY = 0, AX = 0, AY = 0, FX = 0, FY = 0, r = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double vx = x[T.v[i]], vy = y[T.v[i]];
    VX = i ? VX + vx : vx;
    VY = i ? VY + vy : vy;
    if constexpr (Q == 1) {
      r = fma(vx, vy, r);
    } else {
      const double ax = x[T.near[i][0]] + x[T.near[i][1]] + x[T.near[i][2]];
      const double ay = y[T.near[i][0]] + y[T.near[i][1]] + y[T.near[i][2]];
      const double bx = x[T.far[i][0]] + x[T.far[i][1]] + x[T.far[i][2]];
      const double by = y[T.far[i][0]] + y[T.far[i][1]] + y[T.far[i][2]];
      const double fx = x[T.f[i]], fy = y[T.f[i]];
      AX = i ? AX + ax : ax;
      AY = i ? AY + ay : ay;
      FX = i ? FX + fx : fx;
      FY = i ? FY + fy : fy;
      r = fma(vx, fma(14.0, vy, fma(-15.0, ay, fma(3.0, by, 18.0 * fy))), r);
      r = fma(ax, fma(-15.0, vy, fma(54.0, ay, fma(-27.0, by, -54.0 * fy))), r);
      r = fma(bx, fma(3.0, vy, -27.0 * ay), r);
      r = fma(fx, fma(18.0, vy, fma(-54.0, ay, 216.0 * fy)), r);
    }
  }
  if constexpr (Q == 1) return fma(VX, VY, r) * (1.0 / 120);
  r = fma(VX, fma(2.0, VY, fma(3.0, AY, 18.0 * FY)), r);
  r = fma(AX, 3.0 * VY, r);
  r = fma(FX, fma(18.0, VY, 216.0 * FY), r);
  return fma(54.0, ee, r) * (1.0 / 26880);
}

// Boundary layout: u, v are [tet][6][Np]; w is [tet][2] = (6|K| eps_K, 6|K| mu_K).  One thread per
// component of a tetrahedron, whose Np values are contiguous and follow the previous thread's; per
// times 128 components per block, the same for every block.
template <int Q>
__global__ void __launch_bounds__(NA_THREADS) na_dot_kernel(const double* __restrict__ u, const double* __restrict__ v,
                                                            const double* __restrict__ w, int64_t nt, int per,
                                                            double* __restrict__ partials) {
  constexpr int NP = np_of(Q);
  double acc = 0;
  int64_t k = (int64_t)blockIdx.x * per * NA_THREADS + threadIdx.x;
  for (int i = 0; i < per && k < 6 * nt; ++i, k += NA_THREADS) {
    double x[NP], y[NP];
#pragma unroll
    for (int n = 0; n < NP; ++n) {
      x[n] = u[k * NP + n];
      y[n] = v[k * NP + n];
    }
    const int64_t e = k / 6;
    acc = fma(w[2 * e + (k - 6 * e < 3 ? 0 : 1)], na_form<Q>(x, y), acc);
  }
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  __shared__ double sh[NA_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0;
    for (int i = 0; i < NA_THREADS / 32; ++i) s += sh[i];
    partials[blockIdx.x] = s;
  }
}

__global__ void na_finalize_kernel(const double* partials, int nblocks, double* __restrict__ out) {
  __shared__ double sh[256];
  double s = 0;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");  // launched while na_dot_kernel ends
  for (int i = threadIdx.x; i < nblocks; i += blockDim.x) s += partials[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

struct NaDevice {
  bool ready = false;
  double* partials = nullptr;  // device address of g_na_partials on this device
};
std::mutex g_na_mutex;
NaDevice g_na_dev[64];

// Once per device, with that device current: look up the scratch array's device address.
int na_setup(int device, double** partials) {
  std::lock_guard<std::mutex> lk(g_na_mutex);
  NaDevice& d = g_na_dev[device];
  if (!d.ready) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_na_partials) != cudaSuccess || p == nullptr) return CMCG_ERR_CUDA;
    d.partials = static_cast<double*>(p);
    d.ready = true;
  }
  *partials = d.partials;
  return CMCG_OK;
}

}  // namespace
}  // namespace cmcg

extern "C" int cmcg_inner_noalloc(int order, int64_t nt, const double* u, const double* v, const double* w,
                                  double* out, void* stream) {
  using namespace cmcg;
  if (order < 1 || order > 3 || nt < 1 || !u || !v || !w || !out) return CMCG_ERR_INVALID_ARG;
  if (nt > CMCG_NOALLOC_MAX_TETS) return CMCG_ERR_INVALID_ARG;  // the interface's limit
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return CMCG_ERR_NO_DEVICE;
  if (device < 0 || device >= 64) return CMCG_ERR_INVALID_ARG;
  double* partials = nullptr;
  int rc = na_setup(device, &partials);
  if (rc != CMCG_OK) return rc;
  const int64_t groups = (6 * nt + NA_THREADS - 1) / NA_THREADS;
  const int per = int((groups + NA_BLOCKS - 1) / NA_BLOCKS), nblocks = int((groups + per - 1) / per);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (order == 1) na_dot_kernel<1><<<nblocks, NA_THREADS, 0, s>>>(u, v, w, nt, per, partials);
  else if (order == 2) na_dot_kernel<2><<<nblocks, NA_THREADS, 0, s>>>(u, v, w, nt, per, partials);
  else na_dot_kernel<3><<<nblocks, NA_THREADS, 0, s>>>(u, v, w, nt, per, partials);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, na_finalize_kernel, static_cast<const double*>(partials), nblocks, out);
  return cudaGetLastError() == cudaSuccess ? CMCG_OK : CMCG_ERR_CUDA;
}
