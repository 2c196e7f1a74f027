// Velocity-conditioned scalar mean for the IECM micromixing model (eq.
// IECM), computed with the sort-and-divide binning of the section on
// conditional statistics and its appendix: the particles of an element are
// sorted by U and divided into parts of equal count (up to one); each part
// is sorted by V and divided, each subpart by W; the conditional mean of a
// particle is the scalar mean of its final part.  A group of n particles is
// divided into k = min(n_c, n / m_min) parts (at least one), part j holding
// the sorted positions i with floor(k i / n) = j; equal velocity components
// are ordered by particle id.
//
// Elements of up to kWarpCap particles take one warp each (k_iecm_warp): the
// entries are sorted by 32-bit keys in registers, one register network per
// level.  Larger elements are listed by it and take one block each
// (k_iecm_cond): their particles in global scratch slices, sorted by rank
// counting inside each group.  Both give the same order: (key, id) is a
// strict total order.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fx.cuh"

namespace pdfgb {

constexpr int kIecmThreads = 128;
constexpr int kWarpCap = 256;

// One copy of the per-particle data in global scratch: the three velocity
// components and the scalar as (high, low) pairs, the particle id and the
// storage slot.  Two copies alternate: every level sorts by moving the data
// into the other copy at the sorted positions, so that the comparisons read
// consecutive entries (no indirection).
struct IecmBuf {
  float* f[8];  // uh ul vh vl wh wl sh sl
  int32_t* id;
  int32_t* slot;
};

struct IecmView {  // the two copies and the group bounds of each position
  IecmBuf a, b;
  int32_t *gs, *ge;
};

__device__ __forceinline__ void load_comp(const fx::df* a, int64_t s, float& h, float& l) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(a) + s);
  h = v.x;
  l = v.y;
}
__device__ __forceinline__ void load_comp(const float* a, int64_t s, float& h, float& l) {
  h = __ldg(a + s);
  l = 0.0f;
}

// (key_j, id_j) < (key_i, id_i) for double-float keys (normalized pairs
// order like their values); evaluated without branches
__device__ __forceinline__ int key_less(float hj, float lj, int32_t ij, float hi, float li, int32_t ii) {
  return (int)((hj < hi) | ((hj == hi) & ((lj < li) | ((lj == li) & (ij < ii)))));
}

// floor(k i / n) and ceil(j n / k) for 0 <= i < n, 0 <= j <= k <= 127: 32-bit
// unsigned arithmetic while the products stay below 2^31 (n < 2^24), 64-bit
// beyond
__device__ __forceinline__ int32_t part_of(int32_t k, int32_t i, int32_t n) {
  if (n < (1 << 24)) return (int32_t)((uint32_t)(k * i) / (uint32_t)n);
  return (int32_t)(((int64_t)k * i) / n);
}
__device__ __forceinline__ int32_t part_start(int32_t j, int32_t n, int32_t k) {
  if (n < (1 << 24)) return (int32_t)(((uint32_t)(j * n) + (uint32_t)(k - 1)) / (uint32_t)k);
  return (int32_t)(((int64_t)j * n + k - 1) / k);
}

// ---------------------------------------------------------------- one warp

constexpr int kIecmWarps = 4;  // elements per block

// The element's entries by their place i in the grouping.
struct WarpEntries {
  float h[3][kWarpCap];    // high parts of U, V, W
  float2 ps[kWarpCap];     // the scalar; later the scalar in sorted order
  int32_t slot[kWarpCap];
  uint16_t ord[kWarpCap];  // tie resolution: entry at each position; bin starts at the end
};

// Ascending bitonic sort of the 32 K keys of a warp, position p = K lane + r in
// register r: one shuffle and one min or max per key and step (steps inside
// a lane need no shuffle).
template <int K>
__device__ __forceinline__ void warp_sort(uint32_t (&x)[K], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * K; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= K) {
        const bool keep_min = ((lane & (j / K)) == 0) == ((lane & (k / K)) == 0);
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const uint32_t y = __shfl_xor_sync(0xffffffffu, x[r], j / K);
          x[r] = keep_min ? min(x[r], y) : max(x[r], y);
        }
      } else {
#pragma unroll
        for (int r = 0; r < K; ++r) {
          if (r & j) continue;
          const bool up = k < K ? (r & k) == 0 : (lane & (k / K)) == 0;
          const uint32_t a = x[r], b = x[r | j];
          x[r] = up ? min(a, b) : max(a, b);
          x[r | j] = up ? max(a, b) : min(a, b);
        }
      }
    }
  }
}

// floor((x + 1/2) / n) = floor(x / n) for integers 0 <= x < 2^15, 1 <= n <= 256 by
// FP32: the quotient stays 1/512 away from the next integer, far more than
// the rounding of 2^-22 times at most 2^8.
__device__ __forceinline__ int32_t small_div(int32_t x, float inv_n) { return (int32_t)(((float)x + 0.5f) * inv_n); }

// One element of 1 to 32 K entries (loaded into S).  Keys: [group start | value |
// entry], the value's place between the element's least and greatest in
// 32 - 2 IB bits (32 - IB on the first level, one group), the entry's number in
// the low IB bits.  The mapping of values to places is monotone, so the order
// is exact except among entries of equal group and place; those (a few
// per thousand groups) are put in the order of (high, low, id) afterwards.
template <int K, typename T>
__device__ __forceinline__ void iecm_element(WarpEntries& S, int32_t N, const T* const (&comp)[3],
                                             const int32_t* __restrict__ pid, const int (&nc)[3], int m_min,
                                             fx::df* __restrict__ cond) {
  constexpr int IB = K == 1 ? 5 : (K == 2 ? 6 : (K == 4 ? 7 : 8));
  constexpr uint32_t kEntry = (1u << IB) - 1;
  const int lane = threadIdx.x & 31;
  const float inv_m = __fdividef(1.0f, (float)m_min);
  // ranges of the three components
  float mn[3], mx[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    mn[c] = __int_as_float(0x7f800000);
    mx[c] = -mn[c];
    for (int i = lane; i < N; i += 32) {
      mn[c] = fminf(mn[c], S.h[c][i]);
      mx[c] = fmaxf(mx[c], S.h[c][i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn[c] = fminf(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], o));
      mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
    }
  }
  int32_t gs[K], gn[K], at[K];  // per position: its group's start and size, the entry there
#pragma unroll
  for (int r = 0; r < K; ++r) {
    gs[r] = 0;
    gn[r] = N;
    at[r] = lane * K + r;
  }
#pragma unroll
  for (int level = 0; level < 3; ++level) {
    const int vb = level == 0 ? 32 - IB : 32 - 2 * IB;  // bits of the value's place
    const float top = (float)((1 << vb) - 2);
    const float range = mx[level] - mn[level];
    const float scale = range > 0.0f ? __fdividef(top, range) : 0.0f;
    uint32_t x[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
      x[r] = 0xffffffffu;  // (past the end; no entry has this key)
      if (lane * K + r < N) {
        const float f = (S.h[level][at[r]] - mn[level]) * scale;
        // (conversion: NaN -> 0, saturating; the clamp also covers a scale of 0 or infinity)
        const uint32_t q = (uint32_t)min(max(__float2int_rz(fminf(f, top)), 0), (1 << vb) - 2);
        x[r] = (level == 0 ? 0u : (uint32_t)gs[r] << (32 - IB)) | (q << IB) | (uint32_t)at[r];
      }
    }
    warp_sort<K>(x, lane);
    // entries of equal group and place next to each other
    const uint32_t next = __shfl_down_sync(0xffffffffu, x[0], 1);
    uint32_t tie = 0;
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const uint32_t y = r + 1 < K ? x[r + 1 < K ? r + 1 : r] : next;
      if (lane * K + r + 1 < N && (x[r] >> IB) == (y >> IB)) tie |= 1u << r;
      at[r] = (int32_t)(x[r] & kEntry);
    }
    if (__any_sync(0xffffffffu, tie != 0)) {
      // exchange neighbours of such runs until their full keys are in order
      const T* a = comp[level];
#pragma unroll
      for (int r = 0; r < K; ++r)
        if (lane * K + r < N) S.ord[lane * K + r] = (uint16_t)(at[r] | ((tie >> r & 1u) << 15));
      __syncwarp();
      for (int quiet = 0, par = 0; quiet < 2; par ^= 1) {
        bool moved = false;
        for (int p = 2 * lane + par; p + 1 < N; p += 64) {
          const uint32_t oi = S.ord[p], oj = S.ord[p + 1];
          if (!(oi & 0x8000u)) continue;
          const int32_t si = S.slot[oi & 0x7fffu], sj = S.slot[oj & 0x7fffu];
          float hi, li, hj, lj;
          load_comp(a, si, hi, li);
          load_comp(a, sj, hj, lj);
          if (key_less(hj, lj, __ldg(pid + sj), hi, li, __ldg(pid + si))) {
            S.ord[p] = (uint16_t)((oj & 0x7fffu) | 0x8000u);
            S.ord[p + 1] = (uint16_t)((oi & 0x7fffu) | (oj & 0x8000u));
            moved = true;
          }
        }
        __syncwarp();
        quiet = __any_sync(0xffffffffu, moved) ? 0 : quiet + 1;
      }
#pragma unroll
      for (int r = 0; r < K; ++r)
        if (lane * K + r < N) at[r] = S.ord[lane * K + r] & 0x7fff;
      __syncwarp();
    }
    // divide each group into k parts of equal count
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const int32_t n = gn[r], p = lane * K + r - gs[r];
      const int32_t k = max(1, min(nc[level], small_div(n, inv_m)));
      const int32_t j = small_div(k * p, __fdividef(1.0f, (float)n));
      const float inv_k = __fdividef(1.0f, (float)k);
      const int32_t b = small_div(j * n + k - 1, inv_k), e = small_div(j * n + n + k - 1, inv_k);
      gs[r] += b;
      gn[r] = e - b;
    }
  }
  // bin means in double-float, each bin added in sorted order by one lane; the
  // mean is left at the bin's first position
  float2 v[K];
#pragma unroll
  for (int r = 0; r < K; ++r) v[r] = S.ps[at[r] & (kWarpCap - 1)];
  __syncwarp();
  int bins = 0;
#pragma unroll
  for (int r = 0; r < K; ++r) {
    const int p = lane * K + r;
    if (p < N) S.ps[p] = v[r];
    const bool first = p < N && gs[r] == p;
    const uint32_t m = __ballot_sync(0xffffffffu, first);
    if (first) S.ord[bins + __popc(m & ((1u << lane) - 1))] = (uint16_t)p;
    bins += __popc(m);
  }
  // (register r of the lanes: the starts are not in order across r, each
  // bin's end comes from its size, kept beside the start)
  __syncwarp();
#pragma unroll
  for (int r = 0; r < K; ++r)
    if (lane * K + r < N && gs[r] == lane * K + r) S.h[0][gs[r]] = __int_as_float(gn[r]);
  __syncwarp();
  for (int t = lane; t < bins; t += 32) {
    const int a = S.ord[t], n = __float_as_int(S.h[0][a]);
    const float2 f = S.ps[a];
    fx::acc s;
    s.init(fx::df{f.x, f.y});
    for (int q = a + 1; q < a + n; ++q) s.add(fx::df{S.ps[q].x, S.ps[q].y});
    const fx::df mean = fx::df_norm(fx::mul(s.value(), fx::recip_df(n)));
    S.ps[a] = make_float2(mean.h, mean.l);
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < K; ++r)
    if (lane * K + r < N) reinterpret_cast<float2*>(cond)[S.slot[at[r]]] = S.ps[gs[r]];
}

// One warp per element of at most kWarpCap particles; the larger ones are
// appended to big[1 ..], their number in big[0].  Instruction issue bounds it, at
// well under half of the instructions of one block per element with the entries
// moved through shared memory level by level (39,402 elements of 100 particles:
// 376 -> 131 us).
template <typename T>
__global__ void __launch_bounds__(32 * kIecmWarps) k_iecm_warp(const int32_t* __restrict__ seg,
                                                               const int32_t* __restrict__ order, int32_t n_tri,
                                                               const T* __restrict__ u, const T* __restrict__ v,
                                                               const T* __restrict__ w, const T* __restrict__ ps,
                                                               const int32_t* __restrict__ pid, int nc0, int nc1,
                                                               int nc2, int m_min, int32_t* __restrict__ big,
                                                               fx::df* __restrict__ cond) {
  __shared__ WarpEntries sh[kIecmWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int32_t e = blockIdx.x * kIecmWarps + wid;
  if (e >= n_tri) return;
  const int32_t beg = seg[e], N = seg[e + 1] - beg;
  if (N == 0) return;
  if (N > kWarpCap) {
    if (lane == 0) big[1 + atomicAdd(big, 1)] = e;
    return;
  }
  WarpEntries& S = sh[wid];
  for (int i = lane; i < N; i += 32) {
    const int32_t s = order ? __ldg(order + beg + i) : beg + i;
    float l;
    S.slot[i] = s;
    load_comp(u, s, S.h[0][i], l);
    load_comp(v, s, S.h[1][i], l);
    load_comp(w, s, S.h[2][i], l);
    float2 f;
    load_comp(ps, s, f.x, f.y);
    S.ps[i] = f;
  }
  __syncwarp();
  const T* const comp[3] = {u, v, w};
  const int nc[3] = {nc0, nc1, nc2};
  if (N <= 32) iecm_element<1>(S, N, comp, pid, nc, m_min, cond);
  else if (N <= 64) iecm_element<2>(S, N, comp, pid, nc, m_min, cond);
  else if (N <= 128) iecm_element<4>(S, N, comp, pid, nc, m_min, cond);
  else iecm_element<8>(S, N, comp, pid, nc, m_min, cond);
}

// --------------------------------------------------------------- one block

// One block per listed element (list[0] of them).
template <typename T>
__global__ void __launch_bounds__(kIecmThreads) k_iecm_cond(const int32_t* __restrict__ seg,
                                                            const int32_t* __restrict__ order,
                                                            const int32_t* __restrict__ list,
                                                            const T* __restrict__ u, const T* __restrict__ v,
                                                            const T* __restrict__ w, const T* __restrict__ ps,
                                                            const int32_t* __restrict__ pid, int nc0, int nc1,
                                                            int nc2, int m_min, IecmView big,
                                                            fx::df* __restrict__ cond) {
  const int tid = threadIdx.x;
  const int32_t count = list[0];
  for (int32_t t = blockIdx.x; t < count; t += gridDim.x) {
    const int32_t e = list[1 + t];
    const int32_t beg = seg[e], N = seg[e + 1] - beg;
    // the element's slices of the global scratch
    IecmView V = big;
    for (int c = 0; c < 2; ++c) {
      IecmBuf& B = c == 0 ? V.a : V.b;
      for (int q = 0; q < 8; ++q) B.f[q] += beg;
      B.id += beg;
      B.slot += beg;
    }
    V.gs += beg;
    V.ge += beg;
    for (int i = tid; i < N; i += kIecmThreads) {
      const int64_t s = order ? (int64_t)order[beg + i] : (int64_t)(beg + i);
      V.a.slot[i] = (int32_t)s;
      V.a.id[i] = pid[s];
      load_comp(u, s, V.a.f[0][i], V.a.f[1][i]);
      load_comp(v, s, V.a.f[2][i], V.a.f[3][i]);
      load_comp(w, s, V.a.f[4][i], V.a.f[5][i]);
      load_comp(ps, s, V.a.f[6][i], V.a.f[7][i]);
      V.gs[i] = 0;
      V.ge[i] = N;
    }
    __syncthreads();
    const int ncs[3] = {nc0, nc1, nc2};
#pragma unroll  // static indices into the copies' pointer arrays
    for (int level = 0; level < 3; ++level) {
      const float* kh = V.a.f[2 * level];
      const float* kl = V.a.f[2 * level + 1];
      // sort each group [gs, ge) by rank counting; every entry moves to its
      // sorted position in the other copy
      for (int pos = tid; pos < N; pos += kIecmThreads) {
        const int32_t a = V.gs[pos], b = V.ge[pos];
        const float hi = kh[pos], li = kl[pos];
        const int32_t ii = V.a.id[pos];
        int32_t r = 0;
#pragma unroll 4
        for (int32_t q = a; q < b; ++q) r += key_less(kh[q], kl[q], V.a.id[q], hi, li, ii);
        const int32_t to = a + r;
#pragma unroll
        for (int c = 0; c < 8; ++c) V.b.f[c][to] = V.a.f[c][pos];
        V.b.id[to] = ii;
        V.b.slot[to] = V.a.slot[pos];
      }
      __syncthreads();
      // divide each group into k parts of equal count
      for (int pos = tid; pos < N; pos += kIecmThreads) {
        const int32_t a = V.gs[pos], n = V.ge[pos] - a;
        int32_t k = (int32_t)((uint32_t)n / (uint32_t)m_min);
        if (k > ncs[level]) k = ncs[level];
        if (k < 1) k = 1;
        const int32_t j = part_of(k, pos - a, n);
        V.gs[pos] = a + part_start(j, n, k);
        V.ge[pos] = a + part_start(j + 1, n, k);
      }
      const IecmBuf t = V.a;
      V.a = V.b;
      V.b = t;
      __syncthreads();
    }
    // bin means: the first position of each bin adds its bin in sorted order
    // (double-float) and leaves the mean at that position of the spare copy
    for (int pos = tid; pos < N; pos += kIecmThreads) {
      const int32_t a = V.gs[pos], b = V.ge[pos];
      if (pos != a) continue;
      fx::acc s;
      s.init(fx::df{V.a.f[6][a], V.a.f[7][a]});
      for (int32_t q = a + 1; q < b; ++q) s.add(fx::df{V.a.f[6][q], V.a.f[7][q]});
      const fx::df mean = fx::df_norm(fx::mul(s.value(), fx::recip_df(b - a)));
      V.b.f[0][a] = mean.h;
      V.b.f[1][a] = mean.l;
    }
    __syncthreads();
    for (int pos = tid; pos < N; pos += kIecmThreads) {
      const int32_t a = V.gs[pos];
      reinterpret_cast<float2*>(cond)[V.a.slot[pos]] = make_float2(V.b.f[0][a], V.b.f[1][a]);
    }
  }
}

// Grid of the block kernel: an element above kWarpCap has more than that many
// particles, so n / kWarpCap blocks are enough; at most 16 per SM.
static int iecm_blocks(int64_t n) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (int)std::max<int64_t>(1, std::min<int64_t>(n / kWarpCap, (int64_t)sms * 16));
}

// Conditional means of every particle from the grouping in seg / order
// (order: storage slot of each grouped position, NULL for the identity).
pdf_status iecm_cond(pdf_particles* P, const int32_t* seg, const int32_t* order, cudaStream_t st) {
  if (P->iecm_bins[0] <= 0) return PDF_OK;
  const MeshDev& M = P->mesh->d;
  IecmView big;
  float* f = P->iecm_scratch_f;
  int32_t* g = P->iecm_scratch_i;
  const int64_t n = P->n;
  for (int c = 0; c < 2; ++c) {
    IecmBuf& B = c == 0 ? big.a : big.b;
    for (int q = 0; q < 8; ++q) B.f[q] = f + (8 * c + q) * n;
    B.id = g + (2 * c) * n;
    B.slot = g + (2 * c + 1) * n;
  }
  big.gs = g + 4 * n;
  big.ge = g + 5 * n;
  const int nb = iecm_blocks(n);
  const unsigned nw = (unsigned)((M.n_tri + kIecmWarps - 1) / kIecmWarps);
  int32_t* list = P->iecm_big;
  PDF_CUDA(cudaMemsetAsync(list, 0, sizeof(int32_t), st));
  auto run = [&](auto* u, auto* v, auto* w, auto* ps) -> pdf_status {
    using T = std::remove_reference_t<decltype(*u)>;
    PDF_KERNEL("k_iecm_cond", st, k_iecm_warp<T><<<nw, 32 * kIecmWarps, 0, st>>>(
                                      seg, order, M.n_tri, u, v, w, ps, P->pid, P->iecm_bins[0], P->iecm_bins[1],
                                      P->iecm_bins[2], P->iecm_min, list, P->cond));
    PDF_KERNEL("k_iecm_block", st, k_iecm_cond<T><<<nb, kIecmThreads, 0, st>>>(
                                      seg, order, list, u, v, w, ps, P->pid, P->iecm_bins[0], P->iecm_bins[1],
                                      P->iecm_bins[2], P->iecm_min, big, P->cond));
    return PDF_OK;
  };
  const pdf_status s = P->precision == PDF_FP64 ? run(P->u, P->v, P->w, P->ps) : run(P->uf, P->vf, P->wf, P->psf);
  if (s != PDF_OK) return s;
  P->have_cond = true;
  return PDF_OK;
}

__global__ void k_cond_to_f64(const fx::df* __restrict__ a, const int32_t* __restrict__ pid,
                              double* __restrict__ b, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[pid[i]] = __longlong_as_double((long long)fx::df2d_rn(a[i]));
}

}  // namespace pdfgb

using namespace pdfgb;

extern "C" pdf_status pdf_particles_set_iecm(pdf_particles* p, int32_t nu, int32_t nv, int32_t nw,
                                             int32_t m_min) {
  if (!p) return fail(PDF_EINVAL, "pdf_particles_set_iecm: NULL handle");
  if (nu == 0 && nv == 0 && nw == 0) {
    p->iecm_bins[0] = p->iecm_bins[1] = p->iecm_bins[2] = 0;
    p->have_cond = false;
    return PDF_OK;
  }
  if (nu < 1 || nv < 1 || nw < 1 || m_min < 1 || nu > 127 || nv > 127 || nw > 127)
    return fail(PDF_EINVAL, "pdf_particles_set_iecm: bins must be in [1, 127] and m_min >= 1 (or all bins 0 to disable)");
  if (!p->cond) {
    const size_t n = (size_t)p->n;
    PDF_CUDA(cudaMalloc((void**)&p->cond, sizeof(fx::df) * n));
    PDF_CUDA(cudaMalloc((void**)&p->iecm_scratch_f, sizeof(float) * 16 * n));
    PDF_CUDA(cudaMalloc((void**)&p->iecm_scratch_i, sizeof(int32_t) * 6 * n));
    PDF_CUDA(cudaMalloc((void**)&p->iecm_big, sizeof(int32_t) * ((size_t)p->mesh->d.n_tri + 1)));
  }
  p->iecm_bins[0] = nu;
  p->iecm_bins[1] = nv;
  p->iecm_bins[2] = nw;
  p->iecm_min = m_min;
  p->have_cond = false;
  return PDF_OK;
}

extern "C" pdf_status pdf_iecm_cond(const pdf_particles* p, double* cond, void* stream) {
  if (!p || !cond) return fail(PDF_EINVAL, "pdf_iecm_cond: NULL argument");
  if (!p->have_cond) return fail(PDF_ESTATE, "pdf_iecm_cond: enable IECM and call pdf_estimate_stats first");
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t n = p->n;
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096));
  PDF_KERNEL("k_cond_to_f64", st, k_cond_to_f64<<<g, 256, 0, st>>>(p->cond, p->pid, cond, n));
  return PDF_OK;
}
