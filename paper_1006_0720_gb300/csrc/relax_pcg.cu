// The relaxation's conjugate gradients with the multigrid preconditioner
// (FP64 vectors, matrix, residual and stopping test; FP32 V-cycle), nine
// components at once, in one of two forms:
//   * one cluster of CTAs per component runs its whole solve in one launch
//     (the components' iterations are independent of one another): no kernel
//     boundary and no host read between iterations;
//   * on large meshes the sweeps over the finest level are kernels over the
//     whole GPU and one more kernel, a cluster per component, runs the cycle
//     of the levels below.
// The components of one operator share its matrix, so the finest-level
// kernels take them in planes of three: {0, 4, 8} (the diagonal components,
// an operator each), {1, 2, 3} and {5, 6, 7} (one operator): a thread loads
// a row's indices once for three components instead of once each.
#include <algorithm>

#include "amg.cuh"
#include "common.cuh"
#include "cycle.cuh"

namespace pdfgb {

namespace {

constexpr int kPlaneBlock = 256;
// Levels above this many unknowns are swept by kernels over the whole GPU (at
// 79,600 unknowns 100 to 3,000 were equal, 6,000 slower).
constexpr int32_t kBelowMax = 1500;

__device__ __forceinline__ int plane_comp(int plane, int j) { return plane == 0 ? 4 * j : (plane == 1 ? 1 + j : 5 + j); }

struct Sys {
  int32_t n, nb;
  const int32_t *rp, *ci;
  const double* a[kRxVar];  // the operators, fixed unknowns with their diagonal only
  const uint8_t* wall;
  double *x, *r, *z, *p, *q, *part, *upart, *scal;
  float *r32, *x0;          // FP32 residual and W r, [9][n]
  int32_t* ctl;
};

using RxCycle = Cycle<float, kRxVar>;

// Block partials of the plane's three sums; true in the plane's last block,
// whose thread 0 then holds the totals in t (fixed order).  The values go
// through shared memory and one warp per sum adds them (13 FP64 additions
// per 256 values; a shuffle tree in every warp takes 40, and GB300's FP64
// pipe bounds these kernels).
__device__ __forceinline__ bool plane_total(double (&t)[3], double* part, int32_t* counter) {
  __shared__ double v[3][kPlaneBlock];
  __shared__ double tot[3];
  __shared__ bool last;
  const int32_t nb = gridDim.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto add = [&]() {  // tot = the sums of v
    __syncthreads();
    if (w < 3) {
      double a[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) a[k] = v[w][lane + 32 * k] + v[w][lane + 32 * (k + 4)];
      double s = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) tot[w] = s;
    }
    __syncthreads();
  };
#pragma unroll
  for (int j = 0; j < 3; ++j) v[j][threadIdx.x] = t[j];
  add();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < 3; ++j) part[(int64_t)j * nb + blockIdx.x] = tot[j];
    __threadfence();
    last = atomicAdd(counter, 1) == nb - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (!last) return false;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    double s = 0.0;
    for (int32_t k = threadIdx.x; k < nb; k += kPlaneBlock) s += __ldcg(part + (int64_t)j * nb + k);
    v[j][threadIdx.x] = s;
  }
  add();
#pragma unroll
  for (int j = 0; j < 3; ++j) t[j] = tot[j];
  return true;
}

// acc[j] += sum of a_j[k] x_j[ci[k]] over k = k0, k0 + g, ... < e for the three
// components of a plane: plane 0 has an operator each, the others share one
// (a1 = a2 = a0 unused).  Four entries at a time (see cy_row).
template <typename T>
__device__ __forceinline__ void plane_row(T (&acc)[3], bool own, int32_t k0, int32_t e, int g,
                                          const int32_t* __restrict__ ci, const T* __restrict__ a0,
                                          const T* __restrict__ a1, const T* __restrict__ a2,
                                          const T* __restrict__ x0, const T* __restrict__ x1,
                                          const T* __restrict__ x2) {
  for (int32_t k = k0; k < e; k += 4 * g) {
    int32_t j[4], at[4];
    T w[4], y[4][3];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      at[t] = k + t * g < e ? k + t * g : k;
      j[t] = __ldg(ci + at[t]);
      w[t] = __ldg(a0 + at[t]);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      y[t][0] = __ldg(x0 + j[t]);
      y[t][1] = __ldg(x1 + j[t]);
      y[t][2] = __ldg(x2 + j[t]);
    }
    if (own) {
      T w1[4], w2[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        w1[t] = __ldg(a1 + at[t]);
        w2[t] = __ldg(a2 + at[t]);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (k + t * g < e) {
          acc[0] += w[t] * y[t][0];
          acc[1] += w1[t] * y[t][1];
          acc[2] += w2[t] * y[t][2];
        }
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (k + t * g < e) {
          acc[0] += w[t] * y[t][0];
          acc[1] += w[t] * y[t][1];
          acc[2] += w[t] * y[t][2];
        }
    }
  }
}

// The plane's three vectors of [9][n] and operators of [kRxVar].
template <typename T>
struct PlaneVec {
  const T *v0, *v1, *v2;
  __device__ PlaneVec(const T* base, int64_t n, int plane)
      : v0(base + plane_comp(plane, 0) * n), v1(base + plane_comp(plane, 1) * n), v2(base + plane_comp(plane, 2) * n) {}
};
template <typename T>
__device__ __forceinline__ void plane_rows(T (&acc)[3], int plane, int32_t k0, int32_t e, int g, const int32_t* ci,
                                           const T* const (&a)[kRxVar], const T* x, int64_t n) {
  const PlaneVec<T> X(x, n, plane);
  const bool own = plane == 0;
  plane_row(acc, own, k0, e, g, ci, own ? a[0] : a[3], a[1], a[2], X.v0, X.v1, X.v2);
}

struct PlaneMask {
  bool on[3];
  bool any;
};
__device__ __forceinline__ PlaneMask plane_active(const int32_t* ctl, int plane) {
  PlaneMask m;
  m.any = false;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    m.on[j] = ctl[kRActive + plane_comp(plane, j)] != 0;
    m.any = m.any || m.on[j];
  }
  return m;
}

// The FP32 residual and x_0 = W r before the first cycle.
__global__ void __launch_bounds__(kPlaneBlock) k_rx_begin(Sys S, RxCycle C) {
  const int plane = blockIdx.y;
  const int32_t i = blockIdx.x * kPlaneBlock + threadIdx.x;
  if (i >= S.n) return;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int c = plane_comp(plane, j);
    const int64_t o = (int64_t)c * S.n + i;
    const float rf = (float)S.r[o];
    S.r32[o] = rf;
    S.x0[o] = C.lv[0].w[plane == 0 ? j : 3][i] * rf;
  }
}

// p = z + beta p, q = A z + beta q (= A p) and p . q for a plane (last block:
// alpha = r.z / p.q).  The latency of its
// gathers bounds it, the FP64 pipe half of that: at 79,600 unknowns 44 us
// with one component per thread (the indices and the shared matrix loaded
// nine and six times, shuffle sums), 39 us with three; the matrix in
// 32-row column-major slices, or eight entries in flight instead of four
// (126 registers), were no faster (39 and 47 us).
__global__ void __launch_bounds__(kPlaneBlock) k_rx_spmv(Sys S) {
  const int plane = blockIdx.y;
  if (S.ctl[kRDone]) return;
  const PlaneMask m = plane_active(S.ctl, plane);
  if (!m.any) return;
  const int32_t n = S.n, i = blockIdx.x * kPlaneBlock + threadIdx.x;
  double s[3] = {0.0, 0.0, 0.0};
  if (i < n) {
    double az[3] = {0.0, 0.0, 0.0};
    plane_rows<double>(az, plane, S.rp[i], S.rp[i + 1], 1, S.ci, S.a, S.z, n);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (!m.on[j]) continue;
      const int c = plane_comp(plane, j);
      const int64_t o = (int64_t)c * n + i;
      const double beta = S.scal[kRBeta + c];
      const double qn = az[j] + beta * S.q[o], pn = S.z[o] + beta * S.p[o];
      S.q[o] = qn;
      S.p[o] = pn;
      s[j] = qn * pn;
    }
  }
  if (!plane_total(s, S.part + (int64_t)plane * 3 * gridDim.x, S.ctl + kRCntSpmv + plane) || threadIdx.x != 0) return;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int c = plane_comp(plane, j);
    if (m.on[j]) S.scal[kRAlpha + c] = s[j] != 0.0 ? S.scal[kRRz + c] / s[j] : 0.0;
  }
}

// x += alpha p, r -= alpha q, the FP32 residual and x_0 = W r of the next
// cycle, r . r; the plane's last block counts the iteration and retires
// components at r.r <= rtol^2 b.b; the last of the three planes closes the
// iteration (stops the solve when no component is left, or at max_it).
__global__ void __launch_bounds__(kPlaneBlock) k_rx_update(Sys S, RxCycle C) {
  const int plane = blockIdx.y;
  if (S.ctl[kRDone]) return;
  const PlaneMask m = plane_active(S.ctl, plane);
  bool close = !m.any && blockIdx.x == 0 && threadIdx.x == 0;  // a plane without work still counts
  if (m.any) {
    const int32_t n = S.n, i = blockIdx.x * kPlaneBlock + threadIdx.x;
    double s[3] = {0.0, 0.0, 0.0};
    if (i < n) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (!m.on[j]) continue;
        const int c = plane_comp(plane, j);
        const int64_t o = (int64_t)c * n + i;
        const double alpha = S.scal[kRAlpha + c];
        S.x[o] += alpha * S.p[o];
        const double ri = S.r[o] - alpha * S.q[o];
        S.r[o] = ri;
        const float rf = (float)ri;
        S.r32[o] = rf;
        S.x0[o] = C.lv[0].w[plane == 0 ? j : 3][i] * rf;
        s[j] = ri * ri;
      }
    }
    if (plane_total(s, S.part + (int64_t)(3 + plane) * 3 * gridDim.x, S.ctl + kRCntUpd + plane) && threadIdx.x == 0) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int c = plane_comp(plane, j);
        if (!m.on[j]) continue;
        S.scal[kRRr + c] = s[j];
        S.ctl[kRIters + c] += 1;
        if (s[j] <= S.scal[kRTol2 + c]) S.ctl[kRActive + c] = 0;
      }
      close = true;
    }
  }
  if (!close) return;
  __threadfence();
  if (atomicAdd(S.ctl + kRCntClose, 1) != 2) return;
  S.ctl[kRCntClose] = 0;
  __threadfence();
  const int32_t it = S.ctl[kRIt] + 1;
  S.ctl[kRIt] = it;
  int n_active = 0;
  for (int c = 0; c < 9; ++c) n_active += __ldcg(S.ctl + kRActive + c);
  if (n_active == 0 || it >= S.ctl[kRMaxIt]) S.ctl[kRDone] = 1;
}

// b_{l+1} = S_l b_l and x_{l+1} = W b_{l+1} for a plane, G lanes per coarse row.
template <int G>
__global__ void __launch_bounds__(kPlaneBlock) k_rx_down(Sys S, RxCycle C, int l) {
  const int plane = blockIdx.y;
  if (S.ctl[kRDone]) return;
  if (!plane_active(S.ctl, plane).any) return;
  const CyLevel<float, kRxVar>& M = C.lv[l];
  const int32_t J = (blockIdx.x * kPlaneBlock + threadIdx.x) / G, lane = threadIdx.x % G;
  float s[3] = {0.0f, 0.0f, 0.0f};
  if (J < M.nc) plane_rows<float>(s, plane, M.s_rp[J] + lane, M.s_rp[J + 1], G, M.s_ci, M.s, M.b, M.n);
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
  if (J < M.nc && lane == 0) {
    const CyLevel<float, kRxVar>& N = C.lv[l + 1];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int64_t o = (int64_t)plane_comp(plane, j) * N.n + J;
      N.b[o] = s[j];
      N.x[o] = N.w[plane == 0 ? j : 3][J] * s[j];
    }
  }
}

// The cycle of levels C.first and below, one cluster per component: z of
// level C.first.
__global__ void __launch_bounds__(kCyThreads) k_rx_below(Sys S, RxCycle C) {
  extern __shared__ __align__(16) float lvl[];
  const uint32_t rank = cy_rank(), size = cy_size();
  const int c = blockIdx.x / size, v = cy_variant<kRxVar>(c);
  if (S.ctl[kRDone] || !S.ctl[kRActive + c]) return;
  const CyLevel<float, kRxVar>& M = C.lv[C.first];
  const int64_t o = (int64_t)c * M.n;
  const CyCorr<float> e = cy_below<false, false, float, kRxVar>(C, v, c, rank, size, M.b + o, lvl);
  const CyRows R = cy_rows(M.n, rank, size);
  if (e.local) cy_up<false, true>(M, v, R, M.b + o, M.x + o, e.e, M.z + o);
  else cy_up<false, false>(M, v, R, M.b + o, M.x + o, e.e, M.z + o);
}

// z = x + W (b - A x) + Q z_{l+1} on level l > 0 for a plane, G lanes per row.
template <int G>
__global__ void __launch_bounds__(kPlaneBlock) k_rx_up(Sys S, RxCycle C, int l) {
  const int plane = blockIdx.y;
  if (S.ctl[kRDone]) return;
  if (!plane_active(S.ctl, plane).any) return;
  const CyLevel<float, kRxVar>& M = C.lv[l];
  const int32_t i = (blockIdx.x * kPlaneBlock + threadIdx.x) / G, lane = threadIdx.x % G;
  float ax[3] = {0.0f, 0.0f, 0.0f}, qe[3] = {0.0f, 0.0f, 0.0f};
  if (i < M.n) {
    plane_rows<float>(ax, plane, M.a_rp[i] + lane, M.a_rp[i + 1], G, M.a_ci, M.a, M.x, M.n);
    plane_rows<float>(qe, plane, M.q_rp[i] + lane, M.q_rp[i + 1], G, M.q_ci, M.q, C.lv[l + 1].z, M.nc);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      ax[j] += __shfl_xor_sync(0xffffffffu, ax[j], o);
      qe[j] += __shfl_xor_sync(0xffffffffu, qe[j], o);
    }
  if (i < M.n && lane == 0) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int64_t o = (int64_t)plane_comp(plane, j) * M.n + i;
      M.z[o] = M.x[o] + M.w[plane == 0 ? j : 3][i] * (M.b[o] - ax[j]) + qe[j];
    }
  }
}

// z = x_0 + W (r - A x_0) + Q z_1 on the finest level for a plane, z = 0 on
// the fixed unknowns, r . z (last block: beta, or 0 at the start).
__global__ void __launch_bounds__(kPlaneBlock) k_rx_up0(Sys S, RxCycle C, int first) {
  const int plane = blockIdx.y;
  if (S.ctl[kRDone]) return;
  const PlaneMask m = plane_active(S.ctl, plane);
  if (!m.any) return;
  const CyLevel<float, kRxVar>& M = C.lv[0];
  const int32_t n = M.n, i = blockIdx.x * kPlaneBlock + threadIdx.x;
  double s[3] = {0.0, 0.0, 0.0};
  if (i < n) {
    float ax[3] = {0.0f, 0.0f, 0.0f}, qe[3] = {0.0f, 0.0f, 0.0f};
    const uint8_t w = S.wall[i];
    const bool fixed = plane == 0 ? w == 2 : w != 0;
    if (!fixed) {
      plane_rows<float>(ax, plane, M.a_rp[i], M.a_rp[i + 1], 1, M.a_ci, M.a, S.x0, n);
      plane_rows<float>(qe, plane, M.q_rp[i], M.q_rp[i + 1], 1, M.q_ci, M.q, C.lv[1].z, M.nc);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (!m.on[j]) continue;
      const int64_t o = (int64_t)plane_comp(plane, j) * n + i;
      double zi = 0.0;
      if (!fixed) {
        zi = (double)(S.x0[o] + M.w[plane == 0 ? j : 3][i] * (S.r32[o] - ax[j]) + qe[j]);
        s[j] = S.r[o] * zi;
      }
      S.z[o] = zi;
    }
  }
  if (!plane_total(s, S.upart + (int64_t)plane * 3 * gridDim.x, S.ctl + kRCntUp0 + plane) || threadIdx.x != 0) return;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int c = plane_comp(plane, j);
    if (!m.on[j]) continue;
    const double old = S.scal[kRRz + c];
    S.scal[kRBeta + c] = first || old == 0.0 ? 0.0 : s[j] / old;
    S.scal[kRRz + c] = s[j];
  }
}

Sys make_sys(const RelaxAmg& G, const RxSystem& A) {
  Sys S;
  S.n = A.n;
  S.nb = (A.n + kPlaneBlock - 1) / kPlaneBlock;
  S.rp = A.rp; S.ci = A.ci; S.wall = A.wall;
  for (int v = 0; v < kRxVar; ++v) S.a[v] = G.lv.empty() ? G.c_v[v] : G.lv[0].a_v[v];
  S.x = A.x; S.r = A.r; S.z = A.z; S.p = A.p; S.q = A.q;
  S.part = A.part; S.upart = G.upart; S.scal = A.scal; S.ctl = A.ctl;
  S.r32 = G.r32;
  S.x0 = G.lv.empty() ? nullptr : G.lv[0].x;
  return S;
}

// The levels for a cluster of `ctas` CTAs that runs the cycle below `first`.
RxCycle make_cycle(const RelaxAmg& G, int first, int ctas) {
  RxCycle C;
  C.L = (int)G.lv.size();
  C.first = first;
  C.nc = G.nc;
  C.cinv = G.cinv;
  for (int l = 0; l < C.L; ++l) {
    const RxLevel& V = G.lv[l];
    CyLevel<float, kRxVar>& D = C.lv[l];
    D.n = V.n; D.nc = V.nc; D.nnz_a = V.nnz_a; D.nnz_q = V.nnz_ap;
    D.a_rp = V.a_rp; D.a_ci = V.a_ci; D.q_rp = V.q_rp; D.q_ci = V.q_ci; D.s_rp = V.s_rp; D.s_ci = V.s_ci;
    for (int v = 0; v < kRxVar; ++v) { D.a[v] = V.a_f[v]; D.q[v] = V.q_f[v]; D.s[v] = V.s_f[v]; D.w[v] = V.w_f[v]; }
    D.b = l == 0 ? G.r32 : V.b;
    D.x = V.x;
    D.z = V.z;
  }
  cy_plan(C, ctas);
  return C;
}

constexpr size_t kLevelBytes = sizeof(float) * kCyShared;

// The level from which one cluster per component runs the cycle (form two).
int first_below(const RelaxAmg& G) {
  int l = 1;
  while (l + 1 < (int)G.lv.size() && G.lv[l].n > kBelowMax) ++l;
  return l;
}

}  // namespace

// The line between the two forms, whole relaxation calls to 1e-12: one
// cluster per component 755 us against 1,090 us at 760 unknowns, 1,120
// against 1,369 at 3,520, 1,684 against 1,759 at 6,930, 2,664 against 2,280
// at 17,820 (with the vectors in global memory).
constexpr int32_t kWholeMax = 8192;

bool relax_mg_whole(int32_t n) { return n <= kWholeMax; }

pdf_status relax_mg_solve(const RelaxAmg& G, const RxSystem& A, int32_t it_end, cudaStream_t st) {
  const int ctas = cy_ctas(A.n);
  CySys<kRxVar> S;
  S.n = A.n;
  S.rp = A.rp; S.ci = A.ci; S.wall = A.wall;
  for (int v = 0; v < kRxVar; ++v) S.a[v] = G.lv.empty() ? G.c_v[v] : G.lv[0].a_v[v];
  S.x = A.x; S.r = A.r; S.p = A.p; S.q = A.q;
  S.rr = A.scal + kRRr; S.rz = A.scal + kRRz; S.tol2 = A.scal + kRTol2;
  S.iters = A.ctl + kRIters; S.state = A.ctl + kRActive;
  S.on = 1; S.off = 0;
  const RxCycle C = make_cycle(G, 0, ctas);
  cudaError_t e = cudaSuccess;
  PDF_KERNEL("k_rx_pcg", st, e = (cy_launch_pcg<kWholeMax, float, kRxVar>(9, ctas, st, S, C, it_end)));
  return e == cudaSuccess ? PDF_OK : cuda_fail(e, "k_rx_pcg");
}

// z = M^-1 r from the FP32 residual and x_0 in place.
static pdf_status relax_mg_cycle(const RelaxAmg& G, const Sys& S, int first, cudaStream_t st) {
  const int lb = first_below(G);
  const RxCycle C = make_cycle(G, lb, kCyMaxCtas);
  auto grid = [&](int64_t rows, int lanes) { return dim3((unsigned)((rows * lanes + kPlaneBlock - 1) / kPlaneBlock), 3); };
  for (int l = 0; l < lb; ++l) {
    const RxLevel& V = G.lv[l];
    // eight lanes per coarse row, a warp where the rows of S are long
    if (V.nnz_ap > 48 * (int64_t)V.nc)
      PDF_KERNEL("k_rx_down", st, k_rx_down<32><<<grid(V.nc, 32), kPlaneBlock, 0, st>>>(S, C, l));
    else
      PDF_KERNEL("k_rx_down", st, k_rx_down<8><<<grid(V.nc, 8), kPlaneBlock, 0, st>>>(S, C, l));
  }
  cudaError_t e = cudaSuccess;
  PDF_KERNEL("k_rx_below", st, e = cy_launch(k_rx_below, 9, kCyMaxCtas, kLevelBytes, st, S, C));
  if (e != cudaSuccess) return cuda_fail(e, "k_rx_below");
  for (int l = lb - 1; l > 0; --l)
    PDF_KERNEL("k_rx_up", st, k_rx_up<8><<<grid(G.lv[l].n, 8), kPlaneBlock, 0, st>>>(S, C, l));
  PDF_KERNEL("k_rx_up0", st, k_rx_up0<<<grid(S.n, 1), kPlaneBlock, 0, st>>>(S, C, first));
  return PDF_OK;
}

pdf_status relax_mg_begin(const RelaxAmg& G, const RxSystem& A, cudaStream_t st) {
  const Sys S = make_sys(G, A);
  PDF_KERNEL("k_rx_begin", st, k_rx_begin<<<dim3(S.nb, 3), kPlaneBlock, 0, st>>>(S, make_cycle(G, 1, kCyMaxCtas)));
  return relax_mg_cycle(G, S, 1, st);
}

pdf_status relax_mg_iterations(const RelaxAmg& G, const RxSystem& A, int k, cudaStream_t st) {
  const Sys S = make_sys(G, A);
  const RxCycle C = make_cycle(G, 1, kCyMaxCtas);
  const dim3 grid(S.nb, 3);
  for (int i = 0; i < k; ++i) {
    PDF_KERNEL("k_rx_spmv", st, k_rx_spmv<<<grid, kPlaneBlock, 0, st>>>(S));
    PDF_KERNEL("k_rx_update", st, k_rx_update<<<grid, kPlaneBlock, 0, st>>>(S, C));
    const pdf_status s = relax_mg_cycle(G, S, 0, st);
    if (s != PDF_OK) return s;
  }
  return PDF_OK;
}

}  // namespace pdfgb
