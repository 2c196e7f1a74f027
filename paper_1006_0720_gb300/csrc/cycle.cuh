// Multigrid V-cycles and sums run by one thread-block cluster.
//
// A conjugate-gradient iteration with a V-cycle is ten or so dependent
// sweeps over a few thousand to a hundred thousand unknowns.  As separate
// kernels each sweep costs a kernel boundary, whatever its size (5-7 us on
// the coarse levels, whose work is well below 1 us).  Here one cluster of
// CTAs runs consecutive sweeps with barriers of its own: cluster barriers
// where a sweep is shared out over the CTAs, and block barriers alone on the
// coarsest levels, which every CTA computes for itself in shared memory
// (redundant work of a few hundred nanoseconds instead of a cluster barrier
// and a trip through L2).
#pragma once
#include "common.cuh"

namespace pdfgb {

constexpr int kCyThreads = 512;    // threads per CTA
constexpr int kCyMaxCtas = 8;      // CTAs per cluster (the portable limit)
constexpr int kCyMaxLv = 12;
constexpr int kCyShared = 6144;    // values of the coarse levels kept in shared memory

// One level with V operator variants: x_l = W b_l, b_{l+1} = S b_l on the way
// down, z_l = x_l + W (b_l - A x_l) + Q z_{l+1} on the way up.
template <typename T, int V>
struct CyLevel {
  int32_t n, nc;
  int32_t gs, gu;  // lanes per row of S (down), of A and Q (up): powers of two
  int64_t nnz_a, nnz_q;
  const int32_t *a_rp, *a_ci, *q_rp, *q_ci, *s_rp, *s_ci;
  const T *a[V], *q[V], *s[V], *w[V];
  T *b, *x, *z;    // [components][n]
};

// Levels first <= l < local are shared out over the CTAs (vectors in global
// memory), levels l >= local are every CTA's own (vectors in shared memory;
// local > first), and so is the coarsest system (nc unknowns, its inverse
// cinv [V][nc][nc]).
template <typename T, int V>
struct Cycle {
  int32_t L, first, local, nc;
  const T* cinv;
  CyLevel<T, V> lv[kCyMaxLv];
};

__device__ __forceinline__ uint32_t cy_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cy_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Barrier over the cluster; orders global and (distributed) shared memory.
// ONE: a cluster of one CTA, whose barrier is the block's.
template <bool ONE>
__device__ __forceinline__ void cy_sync() {
  if (ONE) __syncthreads();
  else asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address of a variable of this CTA's shared memory in the CTA of rank r.
__device__ __forceinline__ uint32_t cy_map(const void* p, uint32_t r) {
  uint32_t dst;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(r));
  return dst;
}
__device__ __forceinline__ void cy_st(uint32_t dst, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(v) : "memory");
}
__device__ __forceinline__ void cy_st(uint32_t dst, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(v) : "memory");
}

// The contiguous rows of a CTA.
struct CyRows {
  int32_t lo, hi;
};
__device__ __forceinline__ CyRows cy_rows(int32_t n, uint32_t rank, uint32_t size) {
  const int32_t per = ((n + (int32_t)size - 1) / (int32_t)size + 31) & ~31;
  const int32_t lo = min(n, per * (int32_t)rank);
  return CyRows{lo, min(n, lo + per)};
}

// A vector entry: shared memory, or global memory that other CTAs write
// (read from L2, past this SM's L1).
template <bool LOCAL, typename T>
__device__ __forceinline__ T cy_ld(const T* p, int32_t i) {
  return LOCAL ? p[i] : __ldcg(p + i);
}

__device__ __forceinline__ int cy_log2(int g) { return 31 - __clz(g); }

// s + sum of v[q] b[ci[q]] over q = q0, q0 + g, ... < e, in order.  Four entries
// at a time: their indices, then their values and vector entries are all in
// flight before the first product (a row's chain of dependent loads, one
// entry after the other, was most of a sweep's time).
template <bool LOCAL, typename TV, typename T>
__device__ __forceinline__ T cy_row(T s, int32_t q0, int32_t e, int g, const int32_t* __restrict__ ci,
                                    const TV* __restrict__ v, const T* b) {
  for (int32_t q = q0; q < e; q += 4 * g) {
    int32_t j[4];
    TV w[4];
    T x[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int32_t k = q + t * g < e ? q + t * g : q;
      j[t] = __ldg(ci + k);
      w[t] = __ldg(v + k);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) x[t] = cy_ld<LOCAL>(b, j[t]);
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (q + t * g < e) s += (T)w[t] * x[t];
  }
  return s;
}

// f(row, sum of v[q] b[ci[q]] over the row's entries) for rows [lo, hi), g lanes
// per row; f runs in the row's first lane.
template <bool LOCAL, typename T, typename F>
__device__ __forceinline__ void cy_sweep(CyRows R, int g, const int32_t* __restrict__ rp,
                                         const int32_t* __restrict__ ci, const T* __restrict__ v, const T* b, F f) {
  const int sh = cy_log2(g), lane = threadIdx.x & (g - 1);
  const int32_t items = (((R.hi - R.lo) << sh) + 31) & ~31;
  for (int32_t k = threadIdx.x; k < items; k += kCyThreads) {
    const int32_t row = R.lo + (k >> sh);
    T s = 0;
    if (row < R.hi) s = cy_row<LOCAL>(s, rp[row] + lane, rp[row + 1], g, ci, v, b);
    for (int o = g >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (row < R.hi && lane == 0) f(row, s);
  }
}

// z = x + W (b - A x) + Q e on rows [lo, hi); LX, LE: where x (with b) and e are.
template <bool LX, bool LE, typename T, int V>
__device__ __forceinline__ void cy_up(const CyLevel<T, V>& M, int v, CyRows R, const T* b, const T* x, const T* e,
                                      T* z) {
  const int g = M.gu, sh = cy_log2(g), lane = threadIdx.x & (g - 1);
  const int32_t items = (((R.hi - R.lo) << sh) + 31) & ~31;
  for (int32_t k = threadIdx.x; k < items; k += kCyThreads) {
    const int32_t row = R.lo + (k >> sh);
    T ax = 0, qe = 0;
    if (row < R.hi) {
      ax = cy_row<LX>(ax, M.a_rp[row] + lane, M.a_rp[row + 1], g, M.a_ci, M.a[v], x);
      qe = cy_row<LE>(qe, M.q_rp[row] + lane, M.q_rp[row + 1], g, M.q_ci, M.q[v], e);
    }
    for (int o = g >> 1; o > 0; o >>= 1) {
      ax += __shfl_xor_sync(0xffffffffu, ax, o);
      qe += __shfl_xor_sync(0xffffffffu, qe, o);
    }
    if (row < R.hi && lane == 0) z[row] = cy_ld<LX>(x, row) + M.w[v][row] * (cy_ld<LX>(b, row) - ax) + qe;
  }
}

// The correction of level `first`: where the cycle of the levels below left it.
template <typename T>
struct CyCorr {
  const T* e;
  bool local;
};

// The V-cycle of the levels below `first` for the right-hand side b0 of level
// `first` (SH: whole in this CTA's shared memory, else in global memory
// and visible to the cluster); component c (offset c n in the vectors of the
// levels below), variant v.  Returns z_{first+1} (the coarsest solution when
// first + 1 == L; the solution of the coarsest system for b0 when first == L).
// sm: kCyShared values.
template <bool ONE, bool SH, typename T, int V>
__device__ CyCorr<T> cy_below(const Cycle<T, V>& C, int v, int c, uint32_t rank, uint32_t size, const T* b0, T* sm) {
  const int L = C.L;
  T* s_b[kCyMaxLv + 1];  // shared b, x, z of the local levels; s_b[L]: the coarsest right-hand side
  T* sp = sm;
  for (int l = C.local; l < L; ++l) {
    s_b[l] = sp;
    sp += 3 * C.lv[l].n;
  }
  T *cb = sp, *cz = sp + C.nc;
  if (C.first == L) {  // nothing but the coarsest system
    for (int32_t i = threadIdx.x; i < C.nc; i += kCyThreads) cb[i] = cy_ld<SH>(b0, i);
    __syncthreads();
  }
  for (int l = C.first; l < L; ++l) {
    const CyLevel<T, V>& M = C.lv[l];
    const bool from_local = l >= C.local;  // (false at l == first)
    const T* b = from_local ? s_b[l] : (l == C.first ? b0 : M.b + (int64_t)c * M.n);
    const bool in_shared = from_local || (SH && l == C.first);
    if (l + 1 >= C.local || l + 1 == L) {  // every CTA for itself
      const bool last = l + 1 == L;
      T* bn = last ? cb : s_b[l + 1];
      T* xn = last ? nullptr : bn + M.nc;
      const T* wn = last ? nullptr : C.lv[l + 1].w[v];
      auto put = [&](int32_t J, T s) {
        bn[J] = s;
        if (!last) xn[J] = wn[J] * s;
      };
      const CyRows R{0, M.nc};
      if (in_shared) cy_sweep<true>(R, M.gs, M.s_rp, M.s_ci, M.s[v], b, put);
      else cy_sweep<false>(R, M.gs, M.s_rp, M.s_ci, M.s[v], b, put);
      __syncthreads();
    } else {
      const CyLevel<T, V>& N = C.lv[l + 1];
      T *bn = N.b + (int64_t)c * N.n, *xn = N.x + (int64_t)c * N.n;
      const T* wn = N.w[v];
      auto put = [&](int32_t J, T s) {
        bn[J] = s;
        xn[J] = wn[J] * s;
      };
      const CyRows R = cy_rows(M.nc, rank, size);
      if (in_shared) cy_sweep<true>(R, M.gs, M.s_rp, M.s_ci, M.s[v], b, put);
      else cy_sweep<false>(R, M.gs, M.s_rp, M.s_ci, M.s[v], b, put);
      cy_sync<ONE>();
    }
  }
  {  // the coarsest system: eight lanes per row of its inverse
    const T* Ci = C.cinv + (int64_t)v * C.nc * C.nc;
    const int lane = threadIdx.x & 7;
    const int32_t items = (C.nc * 8 + 31) & ~31;
    for (int32_t k = threadIdx.x; k < items; k += kCyThreads) {
      const int32_t row = k >> 3;
      T s = 0;
      if (row < C.nc)
        for (int32_t j = lane; j < C.nc; j += 8) s += __ldg(Ci + (int64_t)row * C.nc + j) * cb[j];
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (row < C.nc && lane == 0) cz[row] = s;
    }
    __syncthreads();
  }
  CyCorr<T> e{cz, true};
  for (int l = L - 1; l > C.first; --l) {
    const CyLevel<T, V>& M = C.lv[l];
    if (l >= C.local) {
      T *b = s_b[l], *x = b + M.n, *z = x + M.n;
      cy_up<true, true>(M, v, CyRows{0, M.n}, b, x, e.e, z);
      __syncthreads();
      e = CyCorr<T>{z, true};
    } else {
      const int64_t o = (int64_t)c * M.n;
      const CyRows R = cy_rows(M.n, rank, size);
      if (e.local) cy_up<false, true>(M, v, R, M.b + o, M.x + o, e.e, M.z + o);
      else cy_up<false, false>(M, v, R, M.b + o, M.x + o, e.e, M.z + o);
      cy_sync<ONE>();
      e = CyCorr<T>{M.z + o, false};
    }
  }
  return e;
}

// Sum of v over the cluster, in a fixed order; it is also a
// cluster barrier (what was written to global memory before is visible
// after).  Three consecutive calls take the turns 0, 1, 2 (a buffer is written
// again only after another call's barrier).  The thread values go through
// shared memory and one warp adds them: GB300 adds two FP64 numbers per
// clock and SM, so a shuffle tree in every warp (five adds of 32 lanes each)
// would cost five times the additions.
// Of the threads only the first `used` hold a value.  FP64 scalars that follow
// from the sum are formed by one thread as well, f(total) -> CyOut (a
// division in every thread would cost a microsecond).
struct CyOut {
  double v;   // what the caller wants: a quotient, or the sum itself
  int flag;
};
struct CySum {
  double v[kCyThreads];
  double part[3][kCyMaxCtas];
  CyOut out;
};
template <bool ONE, typename F>
__device__ __forceinline__ CyOut cy_sum(double v, int used, CySum& S, int turn, uint32_t rank, uint32_t size, F f) {
  if ((int)threadIdx.x < used) S.v[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = 0.0, t1 = 0.0;
    for (int k = threadIdx.x; k < used; k += 64) {
      t += S.v[k];
      if (k + 32 < used) t1 += S.v[k + 32];
    }
    t += t1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (ONE) {
      if (threadIdx.x == 0) S.out = f(t);
    } else if (threadIdx.x < size) {
      cy_st(cy_map(&S.part[turn][rank], threadIdx.x), t);  // to every CTA of the cluster
    }
  }
  cy_sync<ONE>();
  if (ONE) return S.out;
  if (threadIdx.x == 0) {
    double t = S.part[turn][0];
    for (uint32_t k = 1; k < size; ++k) t += S.part[turn][k];
    S.out = f(t);
  }
  __syncthreads();
  return S.out;
}

// The operator of a component: the relaxation's nine components use the
// variants 0, 1, 2 (components 0, 4, 8) and 3; a single system has one.
template <int V>
__device__ __forceinline__ int cy_variant(int c) {
  return V == 1 ? 0 : (c == 0 ? 0 : (c == 4 ? 1 : (c == 8 ? 2 : 3)));
}

// Systems to solve: per component c (offset c n) x and r = b - A x, the sums and
// thresholds and the control words.  wall (or NULL) marks fixed unknowns, z = 0
// there: 2 for every component, 1 for the off-diagonal ones (c != 0, 4, 8).
template <int V>
struct CySys {
  int32_t n;
  const int32_t *rp, *ci;
  const double* a[V];
  const uint8_t* wall;
  double *x, *r, *p, *q;
  double *rr, *rz;        // r . r; r . z of the last finished iteration
  const double* tol2;     // stop at r . r <= tol2
  int32_t *iters, *state; // state: `on` while the component is to be solved, then `off`
  int32_t on, off;
};

// Preconditioned conjugate gradients for component blockIdx.x / (cluster size)
// up to iteration it_end (a later launch goes on from iters, rz and the
// vectors): FP64, one V-cycle in T per iteration.  ONE: one CTA per component.
// The vectors live in shared memory, those that are gathered (z and, in T, the
// residual and x_0 = W r) whole in every CTA, each row written to all of
// them by its owner, the others (x, r, p, q) with their rows.
template <bool ONE, typename T, int V>
__global__ void __launch_bounds__(kCyThreads) k_cy_pcg(CySys<V> S, Cycle<T, V> C, int32_t it_end) {
  __shared__ CySum sum;
  extern __shared__ __align__(16) unsigned char dyn[];
  const uint32_t rank = ONE ? 0 : cy_rank(), size = ONE ? 1 : cy_size();
  const int c = blockIdx.x / size, v = cy_variant<V>(c);
  if (S.state[c] != S.on || S.iters[c] >= it_end) return;
  const int32_t n = S.n;
  const int64_t off = (int64_t)c * n;
  const CyRows R = cy_rows(n, rank, size);
  const int32_t per = cy_rows(n, 0, size).hi;
  // shared memory: z [n], x, r, p, q [rows of a CTA], rt and x0 [n]; then the levels
  const int32_t ns = (n + 1) & ~1;
  double* const z = reinterpret_cast<double*>(dyn);
  double* const x = z + ns - R.lo;  // (indexed by row)
  double *const r = x + per, *const p = r + per, *const q = p + per;
  T* const rt = reinterpret_cast<T*>(z + ns + 4 * per);
  T* const x0 = rt + ns;
  T* const sm = x0 + ns;
  auto put_r = [&](int32_t i, T rf, T xf) {
    if (ONE) {
      rt[i] = rf;
      x0[i] = xf;
    } else {
      for (uint32_t k = 0; k < size; ++k) {
        cy_st(cy_map(rt + i, k), rf);
        cy_st(cy_map(x0 + i, k), xf);
      }
    }
  };
  auto fixed = [&](int32_t i) {
    if (V == 1) return false;
    const uint8_t w = S.wall[i];
    return w == 2 || (w == 1 && v == V - 1);
  };
  const CyLevel<T, V>& M = C.lv[0];
  const T* w0 = C.L > 0 ? M.w[v] : nullptr;
  const double tol2 = S.tol2[c];
  int32_t it = S.iters[c];
  double rz_old = S.rz[c], rr = S.rr[c];  // (rz_old: current in thread 0)
  int done = 0;
  const int used = min(R.hi - R.lo, kCyThreads);  // threads with a row
  cy_sync<ONE>();  // every CTA runs (remote stores) and has read the state that the first writes at the end
  for (int32_t i = R.lo + threadIdx.x; i < R.hi; i += kCyThreads) {
    const double ri = S.r[off + i];
    r[i] = ri;
    x[i] = S.x[off + i];
    p[i] = S.p[off + i];
    q[i] = S.q[off + i];
    const T rf = (T)ri;
    put_r(i, rf, w0 ? w0[i] * rf : (T)0);
  }
  cy_sync<ONE>();
  for (;;) {
    // z = M^-1 r, z = 0 on the fixed unknowns, r . z
    const CyCorr<T> e = cy_below<ONE, true, T, V>(C, v, c, rank, size, rt, sm);
    double s = 0.0;
    for (int32_t i = R.lo + threadIdx.x; i < R.hi; i += kCyThreads) {
      double zi = 0.0;
      if (!fixed(i)) {
        if (C.L == 0) {
          zi = (double)e.e[i];
        } else {
          const T ax = cy_row<true>((T)0, M.a_rp[i], M.a_rp[i + 1], 1, M.a_ci, M.a[v], (const T*)x0);
          const T qe = e.local ? cy_row<true>((T)0, M.q_rp[i], M.q_rp[i + 1], 1, M.q_ci, M.q[v], e.e)
                               : cy_row<false>((T)0, M.q_rp[i], M.q_rp[i + 1], 1, M.q_ci, M.q[v], e.e);
          zi = (double)(x0[i] + w0[i] * (rt[i] - ax) + qe);
        }
        s += r[i] * zi;
      }
      if (ONE) z[i] = zi;
      else
        for (uint32_t k = 0; k < size; ++k) cy_st(cy_map(z + i, k), zi);
    }
    const double beta = cy_sum<ONE>(s, used, sum, 0, rank, size, [&](double rz) {
                          const CyOut o{it == 0 || rz_old == 0.0 ? 0.0 : rz / rz_old, 0};
                          rz_old = rz;
                          return o;
                        }).v;
    // p = z + beta p, q = A z + beta q (= A p), p . q
    s = 0.0;
    for (int32_t i = R.lo + threadIdx.x; i < R.hi; i += kCyThreads) {
      const double az = cy_row<true>(0.0, S.rp[i], S.rp[i + 1], 1, S.ci, S.a[v], (const double*)z);
      const double pn = it == 0 ? z[i] : z[i] + beta * p[i], qn = it == 0 ? az : az + beta * q[i];
      p[i] = pn;
      q[i] = qn;
      s += pn * qn;
    }
    // (a single system stops at p . q <= 0, a breakdown)
    const CyOut a = cy_sum<ONE>(s, used, sum, 1, rank, size, [&](double pq) {
      const bool ok = V == 1 ? pq > 0.0 : pq != 0.0;
      return CyOut{ok ? rz_old / pq : 0.0, V == 1 && !ok ? 1 : 0};
    });
    const double alpha = a.v;
    // x += alpha p, r -= alpha q, r . r
    s = 0.0;
    for (int32_t i = R.lo + threadIdx.x; i < R.hi; i += kCyThreads) {
      x[i] += alpha * p[i];
      const double ri = r[i] - alpha * q[i];
      r[i] = ri;
      const T rf = (T)ri;
      put_r(i, rf, w0 ? w0[i] * rf : (T)0);
      s += ri * ri;
    }
    const CyOut o = cy_sum<ONE>(s, used, sum, 2, rank, size, [&](double t) { return CyOut{t, t <= tol2 ? 1 : 0}; });
    rr = o.v;
    done = o.flag | a.flag;
    ++it;
    if (done || it >= it_end) break;
  }
  for (int32_t i = R.lo + threadIdx.x; i < R.hi; i += kCyThreads) {
    S.x[off + i] = x[i];
    S.r[off + i] = r[i];
    S.p[off + i] = p[i];
    S.q[off + i] = q[i];
  }
  if (rank == 0 && threadIdx.x == 0) {
    S.rr[c] = rr;
    S.rz[c] = rz_old;
    S.iters[c] = it;
    S.state[c] = done ? S.off : S.on;
  }
}

// ---- host side

// Lanes per row for `rows` rows of `len` entries on `threads` threads: enough
// that a row's entries are read by consecutive lanes, more while threads
// would be idle.
inline int cy_lanes(int64_t rows, double len, int64_t threads) {
  int g = 1;
  while (g < 32 && 8 * g < len) g *= 2;
  while (g < 32 && 2 * g <= len && rows * 2 * g <= threads) g *= 2;
  return g;
}

// Which levels are every CTA's own, and the lanes per row of each sweep, for
// clusters of `ctas` CTAs.  A level is every CTA's own when the sweep into it
// has at most 6,000 entries (12 per thread: about the time of a cluster
// barrier) and the vectors of all such levels fit into shared memory.
template <typename T, int V>
void cy_plan(Cycle<T, V>& C, int ctas) {
  C.local = C.L;
  int64_t values = 2 * (int64_t)C.nc;
  for (int l = C.L - 1; l > C.first; --l) {
    values += 3 * (int64_t)C.lv[l].n;
    if (C.lv[l - 1].nnz_q > 6000 || values > kCyShared) break;
    C.local = l;
  }
  const int64_t all = (int64_t)kCyThreads * ctas;
  for (int l = 0; l < C.L; ++l) {
    CyLevel<T, V>& D = C.lv[l];
    D.gs = cy_lanes(D.nc, (double)D.nnz_q / D.nc, l + 1 >= C.local ? kCyThreads : all);
    D.gu = cy_lanes(D.n, (double)(D.nnz_a < D.nnz_q ? D.nnz_a : D.nnz_q) / D.n, l >= C.local ? kCyThreads : all);
  }
}

// CTAs per cluster: one per 256 rows, a power of two (128, 512 and 1,024 rows
// per CTA were equal or slower at 760 to 6,930 unknowns).
inline int cy_ctas(int64_t rows) {
  int c = 1;
  while (c < kCyMaxCtas && 256 * (int64_t)c < rows) c *= 2;
  return c;
}

template <typename... Args>
cudaError_t cy_launch(void (*k)(Args...), int clusters, int ctas, size_t shared, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * ctas);
  cfg.blockDim = dim3(kCyThreads);
  cfg.dynamicSmemBytes = shared;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// Dynamic shared memory of k_cy_pcg for n unknowns on clusters of `ctas` CTAs.
template <typename T>
constexpr size_t cy_pcg_shared(int64_t n, int64_t ctas) {
  const size_t per = (size_t)(((n + ctas - 1) / ctas + 31) & ~31), ns = (size_t)((n + 1) & ~1);
  return sizeof(T) * (kCyShared + 2 * ns) + sizeof(double) * (ns + 4 * per);
}

// MAX_N: the most unknowns the caller solves so.  A kernel's limit of dynamic
// shared memory belongs to the kernel, not to the launch, and handles of several
// threads share it: every call sets the same one, that of the largest system
// (a limit per size was lowered by one thread between another's setting and
// its launch).
template <int32_t MAX_N, typename T, int V>
cudaError_t cy_launch_pcg(int comps, int ctas, cudaStream_t st, const CySys<V>& S, const Cycle<T, V>& C,
                          int32_t it_end) {
  // up to 256 unknowns one CTA, 256 per CTA below eight of them
  const size_t limit = ctas == 1 ? cy_pcg_shared<T>(256, 1) : cy_pcg_shared<T>(MAX_N, kCyMaxCtas);
  const size_t bytes = cy_pcg_shared<T>(S.n, ctas);
  if (bytes > limit || 2 * (int64_t)C.nc > kCyShared) return cudaErrorInvalidValue;  // (the latter: see cy_below)
  void (*k)(CySys<V>, Cycle<T, V>, int32_t) = ctas == 1 ? k_cy_pcg<true, T, V> : k_cy_pcg<false, T, V>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
  return e == cudaSuccess ? cy_launch(k, comps, ctas, bytes, st, S, C, it_end) : e;
}

}  // namespace pdfgb
