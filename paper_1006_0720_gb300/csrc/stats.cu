// Particle-in-cell statistics (sec. 3.3) and derivatives (sec. 3.4).
//
// Grouping: a stable least-significant-digit radix sort of (element id,
// storage slot) pairs in place of the paper's per-element linked lists.
// Stability makes the particle order inside every element ascending in
// storage slot, so the segmented reductions below always add the same
// numbers in the same order: the statistics are deterministic without
// floating-point atomics.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fx.cuh"

namespace pdfgb {

// How a sort of n keys below 2^key_bits is done.  As few passes as digits of
// up to 11 bits allow, the digits as narrow as that number of passes leaves
// them: 2,048 elements take one pass, 2^20 (the 535,720-triangle obstacle
// mesh) two of 10 bits instead of three of 9, and a mesh of 11,000 elements
// two of 7, whose counters are cheaper to clear and to scan.  Tiles of
// 2,048 keys instead of 4,096 up to 131,072 keys, so that a small set still
// spreads over the GPU.  With at most kFusedTiles tiles every scatter block
// sums the tile counts itself instead of a scan kernel doing so.  Above 8,192
// tiles, four consecutive tiles share one histogram (a block takes them in
// turn): the tile counts of 68.6 million keys and 1,024 digits shrink from 68
// to 17 MB (the scan of them from 42 to 16 us); at 15.9 million keys two tiles
// per block made the scatter 71 instead of 68 us.
constexpr int kSortThreads = 256;   // of the histogram
constexpr int kScatterThreads = 512;
constexpr int kTileLarge = 4096, kTileSmall = 2048;
constexpr int kMaxBits = 11, kMinBits = 6;
constexpr int kFusedTiles = 128;
struct RadixPlan {
  int passes, bits, tile;
  int sub;        // tiles per histogram
  int64_t tiles;  // histograms
  bool fused;
};
static RadixPlan radix_plan(int64_t n, int key_bits, int max_bits) {
  RadixPlan R;
  R.passes = std::max(1, (key_bits + max_bits - 1) / max_bits);
  R.bits = std::max(kMinBits, (key_bits + R.passes - 1) / R.passes);
  R.tile = n <= 131072 ? kTileSmall : kTileLarge;
  R.tiles = (n + R.tile - 1) / R.tile;
  R.sub = R.tiles > 8192 ? 4 : 1;
  R.tiles = (R.tiles + R.sub - 1) / R.sub;
  R.fused = R.tiles <= kFusedTiles;
  return R;
}
static int key_bits_of(int64_t n_keys) {
  int bits = 1;
  while ((1LL << bits) < n_keys) ++bits;
  return bits;
}

// Entries of the tile histogram for n keys below 2^key_bits, and of the digit
// totals and chunk sums of the scan (any sort; to be zeroed once, every pass
// that scans leaves the sums at zero again).
int64_t radix_hist_len(int64_t n, int key_bits) {
  const RadixPlan R = radix_plan(n, key_bits, kMaxBits);
  return R.tiles << R.bits;
}
constexpr int kScanChunks = 64;  // of tiles
int32_t radix_part_len() { return (1 + kScanChunks) << kMaxBits; }  // and the chunk sums of the scan

// The chunk of a tile: chunk c holds the tiles [n_tiles c / 64, n_tiles (c + 1) / 64).
__device__ __forceinline__ int64_t scan_chunk(int64_t n_tiles, int64_t tile) {
  return (kScanChunks * (tile + 1) - 1) / n_tiles;
}

// Per-tile digit histogram, tile by tile: hist[tile * bins + digit].  (Digit by
// digit, every count went to a sector of its own: with 10-bit digits the
// 32-byte sectors of a tile's counts were twice the bytes of its keys, here
// and again in the scatter.)  Thread t counts the tile's keys PER t ... PER (t + 1) - 1
// (16-byte loads when the keys are 16-byte aligned) as runs of equal digits,
// one shared atomic per run: the element ids arrive nearly sorted (the state
// is reordered by element every few steps, and the second pass reads the first
// pass's output), so a thread's keys are mostly one or two runs.  sums (zero
// before, or NULL): the counts of each chunk of tiles, [kScanChunks][bins], for
// k_scan_bins.
template <int BITS, int TILE>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const int32_t* keys, int64_t n,
                                                             int shift, int sub, int32_t* __restrict__ hist,
                                                             int32_t* __restrict__ sums) {
  overlap_begin();
  constexpr int kBins = 1 << BITS, kPer = TILE / kSortThreads;
  __shared__ int32_t h[kBins];
  for (int b = threadIdx.x; b < kBins; b += kSortThreads) h[b] = 0;
  __syncthreads();
  for (int t = 0; t < sub; ++t) {
    const int64_t i0 = ((int64_t)blockIdx.x * sub + t) * TILE + (int64_t)threadIdx.x * kPer;
    int32_t k[kPer];
    if (i0 + kPer <= n && (reinterpret_cast<uintptr_t>(keys + i0) & 15) == 0) {
      const int4* q = reinterpret_cast<const int4*>(keys + i0);
#pragma unroll
      for (int j = 0; j < kPer / 4; ++j) {
        const int4 v = q[j];
        k[4 * j] = v.x; k[4 * j + 1] = v.y; k[4 * j + 2] = v.z; k[4 * j + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int r = 0; r < kPer; ++r) k[r] = (i0 + r < n) ? keys[i0 + r] : 0;
    }
    const int m = (int)max((int64_t)0, min((int64_t)kPer, n - i0));  // keys of this thread
    int run_d = -1, run_c = 0;
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      if (r >= m) break;
      const int d = (k[r] >> shift) & (kBins - 1);
      if (d != run_d) {
        if (run_c) atomicAdd(&h[run_d], run_c);
        run_d = d;
        run_c = 0;
      }
      ++run_c;
    }
    if (run_c) atomicAdd(&h[run_d], run_c);
  }
  __syncthreads();
  if (sums) sums += scan_chunk(gridDim.x, blockIdx.x) * kBins;
  for (int b = threadIdx.x; b < kBins; b += kSortThreads) {
    const int32_t c = h[b];
    hist[(int64_t)blockIdx.x * kBins + b] = c;
    if (sums && c) atomicAdd(sums + b, c);
  }
}

// Exclusive block-wide prefix sum (blockDim a multiple of 32, at most
// 1024); *total receives the block's sum.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t* total) {
  __shared__ int32_t warp_sums[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_sums[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    int32_t s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane < nw) warp_sums[lane] = s;
  }
  __syncthreads();
  const int32_t warp_base = wid > 0 ? warp_sums[wid - 1] : 0;
  if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
  const int32_t r = warp_base + inc - v;
  __syncthreads();
  return r;
}

// The exclusive prefix of every digit's counts over the tiles, in place, and
// the digits' totals in part, by blocks of a chunk of tiles (blockIdx.x) and a
// group of 32 digits (blockIdx.y), from the sums of the earlier chunks.
// Thread (x, y) takes digit x of the group and the y-th of the chunk's eight
// runs of tiles, so that a warp reads 128 consecutive bytes.
__global__ void __launch_bounds__(256) k_scan_bins(int32_t* hist, int64_t n_tiles, int bins,
                                                   const int32_t* sums, int32_t* __restrict__ part) {
  overlap_begin();
  __shared__ int32_t before[8][32], own[8][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, b = blockIdx.y * 32 + x;
  const int64_t c0 = n_tiles * blockIdx.x / kScanChunks, c1 = n_tiles * (blockIdx.x + 1) / kScanChunks;
  const int64_t lo = c0 + (c1 - c0) * y / 8, hi = c0 + (c1 - c0) * (y + 1) / 8;
  int32_t t = 0, p = 0;
#pragma unroll
  for (int c = y; c < kScanChunks; c += 8) {  // the chunks before this one, and all
    const int32_t v = sums[c * bins + b];
    if (c < (int)blockIdx.x) p += v;
    t += v;
  }
  before[y][x] = p;
  own[y][x] = t;
  __syncthreads();
  if (blockIdx.x == 0 && y == 0) {
    int32_t total = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) total += own[k][x];
    part[b] = total;
  }
  __syncthreads();
  t = 0;
#pragma unroll 4
  for (int64_t i = lo; i < hi; ++i) t += hist[i * bins + b];
  own[y][x] = t;
  __syncthreads();
  int32_t acc = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) acc += before[k][x] + (k < y ? own[k][x] : 0);
#pragma unroll 4
  for (int64_t i = lo; i < hi; ++i) {
    const int32_t v = hist[i * bins + b];
    hist[i * bins + b] = acc;
    acc += v;
  }
}

// Stable scatter of `sub` consecutive tiles, one after the other, by 512
// threads.  Warp w owns the tile's items
// [TILE / 16 w, TILE / 16 (w + 1)) and ranks them in rounds of 32 in
// index order (match.any groups equal digits, one lane of each group
// advances the warp's own row of shared digit counters, so no block barrier
// between rounds); one pass over the (warp, digit) counts then gives every
// warp and digit its output offset, so items with equal digits keep their
// index order.  The digits' bases come from the scanned histogram (hist, part)
// or (FUSED) from the unscanned one.  seg (a single-pass sort by
// element): block 0 also writes the segment offsets, which are the digit
// bases.  Tiles of 4,096 keys and digits of 9 bits: 64 registers, two blocks
// per SM; the ranking waits on the MIO queue, and more warps (512 threads of 8
// items instead of 256 of 16) cover it.
template <int BITS>
constexpr size_t scatter_shared() {
  return sizeof(int32_t) * ((size_t)(kScatterThreads / 32) * ((1 << BITS) + 1) + (1 << BITS));
}
template <int BITS, int TILE, bool FUSED>
__global__ void __launch_bounds__(kScatterThreads, BITS <= 10 ? 2 : 1) k_radix_scatter(
    const int32_t* keys_in, const int32_t* vals_in, int64_t n, int shift,
    int sub, int64_t n_tiles, const int32_t* hist, int32_t* part,
    int32_t* __restrict__ keys_out, int32_t* __restrict__ vals_out, int32_t* __restrict__ seg, int32_t n_seg) {
  overlap_begin();
  constexpr int kBins = 1 << BITS;
  constexpr int kWarps = kScatterThreads / 32;       // 16
  constexpr int kPerWarp = TILE / kWarps;            // 256 or 128 items
  constexpr int kItems = kPerWarp / 32;              // 8 or 4 rounds
  constexpr int kDig = kBins > kScatterThreads ? kBins / kScatterThreads : 1;  // digits per thread
  extern __shared__ __align__(16) int32_t smem[];
  int32_t* wcnt = smem;                              // [kWarps][kBins + 1]; the extra bin takes the tile's padding
  int32_t* dbase = smem + kWarps * (kBins + 1);      // [kBins] next output position of each digit
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int64_t w0 = (int64_t)blockIdx.x * sub * TILE + (int64_t)wid * kPerWarp;
  int32_t key[kItems], val[kItems], off[kItems];
  auto load = [&]() {
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
      const int64_t i = w0 + r * 32 + lane;
      const bool valid = i < n;
      key[r] = valid ? keys_in[i] : 0;
      val[r] = valid ? (vals_in ? vals_in[i] : (int32_t)i) : 0;
    }
  };
  load();
  // the counts of the thread's digits in the earlier tiles and in all tiles
  const int b0 = threadIdx.x * kDig;
  int32_t mine[kDig], total[kDig];
#pragma unroll
  for (int q = 0; q < kDig; ++q) mine[q] = total[q] = 0;
  if (FUSED) {
    // 512 / bins threads share a digit below 512 bins, each every so many tiles
    constexpr int kShare = kBins < kScatterThreads ? kScatterThreads / kBins : 1;
    const int d0 = kShare > 1 ? threadIdx.x % kBins : b0;
    const int t0 = kShare > 1 ? threadIdx.x / kBins : 0;
#pragma unroll 8
    for (int t = t0; t < (int)n_tiles; t += kShare) {
      int32_t c[kDig];
      const int32_t* h = hist + (int64_t)t * kBins + d0;
      if (kDig == 4) {
        const int4 v = *reinterpret_cast<const int4*>(h);
        c[0] = v.x; c[kDig - 3] = v.y; c[kDig - 2] = v.z; c[kDig - 1] = v.w;
      } else {
#pragma unroll
        for (int q = 0; q < kDig; ++q) c[q] = h[q];
      }
#pragma unroll
      for (int q = 0; q < kDig; ++q) {
        total[q] += c[q];
        if (t < (int)blockIdx.x) mine[q] += c[q];
      }
    }
    if (kShare > 1) {  // (kDig == 1; the counters' space for the shares)
      wcnt[threadIdx.x] = mine[0];
      wcnt[kScatterThreads + threadIdx.x] = total[0];
      __syncthreads();
      mine[0] = total[0] = 0;
      if (b0 < kBins) {
#pragma unroll
        for (int k = 0; k < kShare; ++k) {
          mine[0] += wcnt[k * kBins + b0];
          total[0] += wcnt[kScatterThreads + k * kBins + b0];
        }
      }
      __syncthreads();
    }
  } else if (b0 < kBins) {
#pragma unroll
    for (int q = 0; q < kDig; ++q) {
      total[q] = part[b0 + q];
      mine[q] = hist[(int64_t)blockIdx.x * kBins + b0 + q];
    }
    // the chunk sums behind part go back to zero for the next pass
    if (blockIdx.x < kScanChunks) {
#pragma unroll
      for (int q = 0; q < kDig; ++q) part[(1 + blockIdx.x) * kBins + b0 + q] = 0;
    }
  }
  for (int i = threadIdx.x; i < kWarps * (kBins + 1); i += kScatterThreads) wcnt[i] = 0;
  {
    int32_t sum = 0;
#pragma unroll
    for (int q = 0; q < kDig; ++q) sum += total[q];
    int32_t all;
    int32_t base = block_exclusive_scan(sum, &all);
#pragma unroll
    for (int q = 0; q < kDig; ++q) {
      if (b0 < kBins) {
        dbase[b0 + q] = base + mine[q];
        if (seg && blockIdx.x == 0 && b0 + q < n_seg) seg[b0 + q] = base;
      }
      base += total[q];
    }
    if (seg && blockIdx.x == 0 && threadIdx.x == 0) seg[n_seg] = (int32_t)n;
  }
  __syncthreads();
  const uint32_t lt_mask = (1u << lane) - 1u;
  int32_t* row = wcnt + wid * (kBins + 1);
  for (int t = 0;;) {
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int64_t i = w0 + r * 32 + lane;
    const int d = (i < n) ? ((key[r] >> shift) & (kBins - 1)) : kBins;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const int rank = __popc(peers & lt_mask);
    const int32_t before = row[d];
    __syncwarp();
    if (rank == 0) row[d] = before + __popc(peers);
    __syncwarp();
    off[r] = before + rank;
  }
  __syncthreads();
  // (warp, digit) offsets: the digit's next position and the earlier warps' counts
#pragma unroll
  for (int q = 0; q < kDig; ++q) {
    const int b = b0 + q;
    if (b >= kBins) break;
    int32_t acc = dbase[b];
#pragma unroll
    for (int k = 0; k < kWarps; ++k) {
      const int32_t c = wcnt[k * (kBins + 1) + b];
      wcnt[k * (kBins + 1) + b] = acc;
      acc += c;
    }
    dbase[b] = acc;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int64_t i = w0 + r * 32 + lane;
    if (i < n) {
      const int d = (key[r] >> shift) & (kBins - 1);
      const int32_t pos = row[d] + off[r];
      keys_out[pos] = key[r];
      vals_out[pos] = val[r];
    }
  }
  if (++t == sub) break;
  // the block's next tile
  w0 += TILE;
  load();
  __syncthreads();
  for (int i = threadIdx.x; i < kWarps * (kBins + 1); i += kScatterThreads) wcnt[i] = 0;
  __syncthreads();
  }
}

// seg[e] = first sorted position whose key >= e; seg[n_tri] = n.  Thread t
// takes positions 16t .. 16t + 15 (four 16-byte loads when the keys are
// 16-byte aligned) and position n counts as key n_tri; the key before the
// thread's first comes from the lane below (lane 0 loads it).  One thread
// per 16 positions, n / 16 + 1 threads in all.
constexpr int kSegPer = 16;
int64_t seg_offsets_threads(int64_t n) { return n / kSegPer + 1; }
__global__ void __launch_bounds__(256) k_seg_offsets(const int32_t* keys, int64_t n, int32_t n_tri,
                                                     int32_t* __restrict__ seg) {
  overlap_begin();
  const int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * kSegPer;
  int32_t k[kSegPer];
  if (i0 + kSegPer <= n && (reinterpret_cast<uintptr_t>(keys + i0) & 15) == 0) {
    const int4* q = reinterpret_cast<const int4*>(keys + i0);
#pragma unroll
    for (int j = 0; j < kSegPer / 4; ++j) {
      const int4 v = q[j];
      k[4 * j] = v.x; k[4 * j + 1] = v.y; k[4 * j + 2] = v.z; k[4 * j + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kSegPer; ++j) k[j] = (i0 + j < n) ? keys[i0 + j] : n_tri;
  }
  int32_t prev = __shfl_up_sync(0xffffffffu, k[kSegPer - 1], 1);
  if ((threadIdx.x & 31) == 0) prev = (i0 == 0) ? -1 : ((i0 - 1 < n) ? keys[i0 - 1] : n_tri);
  if (i0 > n) return;
#pragma unroll
  for (int j = 0; j < kSegPer; ++j) {
    const int64_t i = i0 + j;
    if (i > n) break;
    const int32_t cur = k[j];  // n_tri at i == n
    for (int32_t e = prev + 1; e <= cur; ++e) seg[e] = (int32_t)i;
    prev = cur;
  }
}

// A stored state value as a double-float (exact for both storage forms).
template <bool OVER>
__device__ __forceinline__ fx::df ld_df(const fx::df* a, int64_t i) {
  const float2 v = ld_result<OVER>(reinterpret_cast<const float2*>(a) + i);
  return fx::df{v.x, v.y};
}
template <bool OVER>
__device__ __forceinline__ fx::df ld_df(const float* a, int64_t i) {
  return fx::df{ld_result<OVER>(a + i), 0.f};
}

// Eight lanes per element (four elements per warp), one pass over the
// element's particles in the grouping's order (sec. 3.3: N, means, central
// moments with 1/N).  Lane j of a group takes sorted positions j, j + 8, ...
// (eight consecutive positions per load across the group).  Every value
// enters as its deviation d = x - x_0 from the element's first particle, a
// double-float with an absolute error of about 2^-48 |x| (the resolution of
// the stored forms); each lane sums the deviations and their pairwise
// products in double-float in its order, the eight lane sums are combined
// by a fixed butterfly, and
//   mean = x_0 + S_a / N,   moment_ab = (S_ab - S_a S_b / N) / N.
// The shift keeps the cancellation in the moments to a factor of about two
// (the deviations are of the size of the fluctuations).  The order of every
// addition is fixed by the stable grouping, so the results are
// deterministic; a reordering of the storage changes them by rounding only.
// Only FP32 additions and fused multiply-adds per particle (no conversions),
// two values per instruction: the same sums in the same order in two thirds
// of the instructions.  15.9M particles 206 -> 201 us (its reads, 0.7 GB,
// take 105 us), 5.1M in FP32 form 75 -> 64 us.
constexpr int kStatLanes = 8;

__device__ __forceinline__ void prefetch_l2(const void* a) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}

__device__ __forceinline__ void acc_xor(fx::acc2& a, int o) {
  fx::df2 b;
  b.h.x = __shfl_xor_sync(0xffffffffu, a.h.x, o);
  b.h.y = __shfl_xor_sync(0xffffffffu, a.h.y, o);
  b.l.x = __shfl_xor_sync(0xffffffffu, a.l.x, o);
  b.l.y = __shfl_xor_sync(0xffffffffu, a.l.y, o);
  a.add(b);
}

// x - k for stored double-floats, normalized: fx::sub with the final
// renormalization by Fast2Sum instead of TwoSum.  Stored values satisfy
// |l| <= ulp(h)/2, so after the exact TwoSum of the high parts (s, e) the
// low part t = x.l + (e - k.l) never has a larger exponent than s (equal
// exponents: x.h - k.h is exact and a nonzero multiple of the ulp, and
// |t| <= one ulp; across a power of two |t| <= 1.5 ulps of the smaller;
// otherwise |t| is far below |s|; s = 0 gives (t, 0)): under that condition
// Fast2Sum returns the same pair as TwoSum, three instructions fewer.
__device__ __forceinline__ fx::df deviation(fx::df x, fx::df k) {
  const fx::df s = fx::two_sum(x.h, -k.h);
  const float t = __fadd_rn(x.l, __fadd_rn(s.l, -k.l));
  return fx::fast_two_sum(s.h, t);
}
// The same for two values at once.  FP32 values (T = float) have no low parts
// and TwoSum's pair is the exact, normalized difference already.
template <typename T>
__device__ __forceinline__ fx::df deviation_of(fx::df x, fx::df k) {
  if constexpr (std::is_same<T, float>::value) return fx::two_sum(x.h, -k.h);
  return deviation(x, k);
}
template <typename T>
__device__ __forceinline__ fx::df2 deviation2(fx::df2 x, fx::df2 k) {
  const fx::df2 s = fx::two_sum2(x.h, fx::neg2(k.h));
  if constexpr (std::is_same<T, float>::value) return s;
  const fx::f2 t = fx::add2(x.l, fx::sub2(s.l, k.l));
  const fx::f2 h = fx::add2(s.h, t);
  return fx::df2{h, fx::sub2(t, fx::sub2(h, s.h))};
}

// a[i] for a lane-dependent i, by selects (no local-memory array)
template <int N>
__device__ __forceinline__ fx::df pick(const fx::df (&a)[N], int i) {
  fx::df r = a[0];
#pragma unroll
  for (int q = 1; q < N; ++q)
    if (i == q) r = a[q];
  return r;
}
template <int N>
__device__ __forceinline__ fx::df pick_acc(const fx::acc (&a)[N], int i) {
  fx::df r = fx::df{a[0].h, a[0].l};
#pragma unroll
  for (int q = 1; q < N; ++q)
    if (i == q) r = fx::df{a[q].h, a[q].l};
  return fx::df_norm(r);
}

// Central moment m (pairs uu, vv, ww, uv, uw, vw, psi psi) from the sums of
// the deviations (s1) and of their products (s2): (S_ab - S_a S_b / N) / N.
__device__ __forceinline__ double moment(const fx::acc (&s1)[5], const fx::acc (&s2)[7], int m, fx::df invN) {
  const int a = m == 6 ? 4 : (m < 3 ? m : (m == 5 ? 1 : 0));
  const int b = m == 6 ? 4 : (m < 3 ? m : (m == 3 ? 1 : 2));
  const fx::df Sa = pick_acc(s1, a), Sb = pick_acc(s1, b);
  const fx::df corr = fx::df_norm(fx::mul(fx::df_norm(fx::mul(Sa, Sb)), invN));
  return __longlong_as_double((long long)fx::df2d(fx::df_norm(fx::mul(fx::sub(pick_acc(s2, m), corr), invN))));
}

template <typename T, bool OVER>
__global__ void __launch_bounds__(256, 3) k_elem_stats_grp(const int32_t* seg,
                                                       const int32_t* pid, int32_t n_tri, const T* u, const T* v,
                                                       const T* w, const T* om, const T* ps,
                                                       double* __restrict__ es) {
  overlap_begin();
  const int lane = threadIdx.x & 31, j = lane & (kStatLanes - 1);
  const int64_t group = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kStatLanes;
  const int64_t n_groups = ((int64_t)gridDim.x * blockDim.x) / kStatLanes;
  // every lane of a warp runs the same number of rounds (the butterfly
  // below needs all 32 lanes)
  const int64_t rounds = (n_tri + n_groups - 1) / n_groups;
  int64_t e = group;
  for (int64_t r = 0; r < rounds; ++r, e += n_groups) {
    const bool live = e < n_tri;
    const int32_t beg = live ? seg[e] : 0, end = live ? seg[e + 1] : 0;
    const int32_t N = end - beg;
    {  // the next element of this group on its way to L2 (after a
       // reordering of the state its particles sit near their positions in
       // the grouped order)
      const int64_t en = e + n_groups;
      if (en < n_tri) {
        const int32_t nb = seg[en], ne = seg[en + 1];
        for (int32_t i = nb + 16 * j; i < ne; i += 16 * kStatLanes) {
          prefetch_l2(u + i); prefetch_l2(v + i); prefetch_l2(w + i); prefetch_l2(om + i); prefetch_l2(ps + i);
          if (pid) prefetch_l2(pid + i);
        }
      }
    }
    // values in pairs (u, v) and (w, psi), omega by itself
    fx::df2 Kuv{}, Kwp{};
    fx::df Km{0.f, 0.f};
    if (N > 0) {
      const int32_t p0 = pid ? ld_result<OVER>(pid + beg) : beg;
      Kuv = fx::pair(ld_df<OVER>(u, p0), ld_df<OVER>(v, p0));
      Kwp = fx::pair(ld_df<OVER>(w, p0), ld_df<OVER>(ps, p0));
      Km = ld_df<OVER>(om, p0);
    }
    // sums of the deviations (u, v), (w, psi) and of their products (uu, vv),
    // (ww, psi psi), (uw, vw); (uv, the deviations of omega)
    fx::acc2 suv, swp, quv, qwp, qw, qx;
    {
      const fx::df2 z{};
      suv.init(z); swp.init(z); quv.init(z); qwp.init(z); qw.init(z); qx.init(z);
    }
    // two particles per lane and iteration (positions i and i + 8), their
    // slots loaded one iteration ahead, so that ten state loads are in
    // flight before the first is needed; the sums still take the particles
    // in the lane's order i, i + 8, i + 16, ...
    auto slot = [&](int32_t i) { return pid ? ld_result<OVER>(pid + i) : i; };
    int32_t qa = beg + j < end ? slot(beg + j) : 0;
    int32_t qb = beg + j + kStatLanes < end ? slot(beg + j + kStatLanes) : 0;
    auto acc1 = [&](fx::df xu, fx::df xv, fx::df xw, fx::df xm, fx::df xp) {
      // normalized, so that the dropped product of the low parts is below
      // 2^-48 of the product even when the deviation is far below the value
      const fx::df2 duv = deviation2<T>(fx::pair(xu, xv), Kuv);
      const fx::df2 dwp = deviation2<T>(fx::pair(xw, xp), Kwp);
      const fx::df dm = deviation_of<T>(xm, Km);
      suv.add(duv);
      swp.add(dwp);
      quv.add(fx::mul_df2(duv, duv));
      qwp.add(fx::mul_df2(dwp, dwp));
      qw.add(fx::mul_df2(duv, fx::pair(dwp.lane0(), dwp.lane0())));
      qx.add(fx::pair(fx::mul(duv.lane0(), duv.lane1()), dm));
    };
    for (int32_t i = beg + j; i < end; i += 2 * kStatLanes) {
      const int32_t pa = qa, pb = qb;
      const bool hb = i + kStatLanes < end;
      qa = i + 2 * kStatLanes < end ? slot(i + 2 * kStatLanes) : 0;
      qb = i + 3 * kStatLanes < end ? slot(i + 3 * kStatLanes) : 0;
      const fx::df au = ld_df<OVER>(u, pa), av = ld_df<OVER>(v, pa), aw = ld_df<OVER>(w, pa), am = ld_df<OVER>(om, pa), ap = ld_df<OVER>(ps, pa);
      fx::df bu = au, bv = av, bw = aw, bm = am, bp = ap;
      if (hb) { bu = ld_df<OVER>(u, pb); bv = ld_df<OVER>(v, pb); bw = ld_df<OVER>(w, pb); bm = ld_df<OVER>(om, pb); bp = ld_df<OVER>(ps, pb); }
      acc1(au, av, aw, am, ap);
      if (hb) acc1(bu, bv, bw, bm, bp);
    }
    // butterfly within the group of eight: every lane ends with the totals
#pragma unroll
    for (int o = kStatLanes / 2; o > 0; o >>= 1) {
      acc_xor(suv, o);
      acc_xor(swp, o);
      acc_xor(quv, o);
      acc_xor(qwp, o);
      acc_xor(qw, o);
      acc_xor(qx, o);
    }
    auto one = [](float h, float l) { return fx::acc{h, l}; };
    const fx::df K[5] = {Kuv.lane0(), Kuv.lane1(), Kwp.lane0(), Km, Kwp.lane1()};
    const fx::acc s1[5] = {one(suv.h.x, suv.l.x), one(suv.h.y, suv.l.y), one(swp.h.x, swp.l.x), one(qx.h.y, qx.l.y),
                           one(swp.h.y, swp.l.y)};
    const fx::acc s2[7] = {one(quv.h.x, quv.l.x), one(quv.h.y, quv.l.y), one(qwp.h.x, qwp.l.x), one(qx.h.x, qx.l.x),
                           one(qw.h.x, qw.l.x),   one(qw.h.y, qw.l.y),   one(qwp.h.y, qwp.l.y)};
    if (!live) continue;
    double* out = es + e * PDF_NES;
    if (N == 0) {
#pragma unroll
      for (int q = 0; q < PDF_NES; ++q)
        if ((q & (kStatLanes - 1)) == j) out[q] = 0.0;
      continue;
    }
    // the 13 outputs (N, the five means, the seven central moments) are
    // shared out: lane j forms and writes outputs j and j + 8
    // (lanes 1-5 a mean, lanes 0-4 and 6-7 one moment each: one pass of
    // each formula per warp)
    const fx::df invN = fx::recip_df(N);
    if (j == 0) out[0] = (double)N;
    if (j >= 1 && j <= 5) {
      const fx::df Kq = pick(K, j - 1);
      const fx::df Sq = pick_acc(s1, j - 1);
      out[j] = __longlong_as_double((long long)fx::df2d(fx::add(Kq, fx::df_norm(fx::mul(Sq, invN)))));
    }
    const int m = j < 5 ? j + 2 : j - 6;  // output 6 + m; lane 5 has none
    if (j != 5) out[6 + m] = moment(s1, s2, m, invN);
  }
}

// 1 / c for the element counts of a node (the correctly rounded quotients,
// as the division gives them): GB300's FP64 pipe bounds the node passes,
// and a division costs it more than a dozen instructions.
constexpr int kRecipMax = 64;
struct RecipTable {
  double v[kRecipMax + 1];
  constexpr RecipTable() : v() {
    v[0] = 0.0;
    for (int c = 1; c <= kRecipMax; ++c) v[c] = 1.0 / (double)c;
  }
};
__device__ const RecipTable kRecip;
__device__ __forceinline__ double recip_count(int32_t c) {
  return c <= kRecipMax ? __ldg(&kRecip.v[c]) : 1.0 / (double)c;
}

// Node pass: mean over the non-empty surrounding elements (twins merged);
// a node with none keeps its previous value.
__global__ void k_node_stats(const int32_t* __restrict__ nse_off, const int32_t* __restrict__ nse,
                             int32_t n_nodes, const double* es, double* ns,
                             long long* __restrict__ kept) {
  overlap_begin();
  for (int32_t n = blockIdx.x * blockDim.x + threadIdx.x; n < n_nodes; n += gridDim.x * blockDim.x) {
    double acc[PDF_NNS];
#pragma unroll
    for (int q = 0; q < PDF_NNS; ++q) acc[q] = 0.0;
    // empty elements hold zeros and are added like the others: without a
    // branch on N the loads of several elements are in flight together
    // (79,600 nodes: 35 -> 29 us, 39,900: 23.6 -> 18.1 us)
    int c = 0;
    const int32_t end = nse_off[n + 1];
#pragma unroll 3
    for (int32_t i = nse_off[n]; i < end; ++i) {
      const double* s = es + (int64_t)nse[i] * PDF_NES;
      // s[0] = N >= 0: the bits of +0.0 (and -0.0) are not positive, those of
      // any N > 0 are (an integer test instead of an FP64 compare)
      c += __double_as_longlong(s[0]) > 0 ? 1 : 0;
#pragma unroll
      for (int q = 0; q < PDF_NNS; ++q) acc[q] += s[1 + q];
    }
    if (c == 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(kept), 1ULL);
      continue;
    }
    const double inv = recip_count(c);
#pragma unroll
    for (int q = 0; q < PDF_NNS; ++q) ns[(int64_t)n * PDF_NNS + q] = acc[q] * inv;
  }
}

// Element gradients of nodal <U>, <V>, <W>, <vv> (eq. gradient with the
// analytic shape-function derivatives): eg[e] = Ux Uy Vx Vy Wx Wy vvx vvy.
__global__ void k_elem_grad1(const int32_t* __restrict__ tri, const double* __restrict__ dN,
                             int32_t n_tri, const double* ns, double* __restrict__ eg) {
  overlap_begin();
  for (int32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n_tri; e += gridDim.x * blockDim.x) {
    const double* d = dN + (int64_t)e * 6;
    double g[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int fld[4] = {0, 1, 2, 6};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double* S = ns + (int64_t)tri[3 * e + j] * PDF_NNS;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        g[2 * f] += d[j] * S[fld[f]];
        g[2 * f + 1] += d[3 + j] * S[fld[f]];
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) eg[(int64_t)e * 8 + q] = g[q];
  }
}

__global__ void k_node_grad1(const int32_t* __restrict__ nse_off, const int32_t* __restrict__ nse,
                             int32_t n_nodes, const double* eg, double* __restrict__ nd) {
  overlap_begin();
  for (int32_t n = blockIdx.x * blockDim.x + threadIdx.x; n < n_nodes; n += gridDim.x * blockDim.x) {
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    const int32_t b = nse_off[n], c = nse_off[n + 1] - b;
    for (int32_t i = b; i < b + c; ++i) {
      const double* g = eg + (int64_t)nse[i] * 8;
#pragma unroll
      for (int q = 0; q < 6; ++q) acc[q] += g[q];
      acc[6] += g[7];
    }
    double* D = nd + (int64_t)n * PDF_NND;
    const double inv = recip_count(c > 0 ? c : 1);
#pragma unroll
    for (int q = 0; q < 6; ++q) D[q] = acc[q] * inv;
    D[9] = acc[6] * inv;
  }
}

// Second pass: d/dx of the node dU_i/dx plus d/dy of the node dU_i/dy.
__global__ void k_elem_grad2(const int32_t* __restrict__ tri, const double* __restrict__ dN,
                             int32_t n_tri, const double* nd, double* __restrict__ eg) {
  overlap_begin();
  for (int32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n_tri; e += gridDim.x * blockDim.x) {
    const double* d = dN + (int64_t)e * 6;
    double l[3] = {0, 0, 0};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double* D = nd + (int64_t)tri[3 * e + j] * PDF_NND;
#pragma unroll
      for (int i = 0; i < 3; ++i) l[i] += d[j] * D[2 * i] + d[3 + j] * D[2 * i + 1];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) eg[(int64_t)e * 8 + i] = l[i];
  }
}

__global__ void k_node_grad2(const int32_t* __restrict__ nse_off, const int32_t* __restrict__ nse,
                             int32_t n_nodes, const double* eg, double* __restrict__ nd) {
  overlap_begin();
  for (int32_t n = blockIdx.x * blockDim.x + threadIdx.x; n < n_nodes; n += gridDim.x * blockDim.x) {
    double acc[3] = {0, 0, 0};
    const int32_t b = nse_off[n], c = nse_off[n + 1] - b;
    for (int32_t i = b; i < b + c; ++i) {
      const double* g = eg + (int64_t)nse[i] * 8;
      acc[0] += g[0]; acc[1] += g[1]; acc[2] += g[2];
    }
    const double inv = recip_count(c > 0 ? c : 1);
    double* D = nd + (int64_t)n * PDF_NND;
    D[6] = acc[0] * inv; D[7] = acc[1] * inv; D[8] = acc[2] * inv;
  }
}

static int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

static int blocks_for(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)sm_count() * 32));
}

// Threads per block of a pass over n nodes or elements: 128, fewer while that
// leaves less than four blocks per SM.  The FP64 pipe, two operations per
// clock for a whole SM, bounds these passes, so a small mesh wants its warps
// on as many SMs as there are (node coefficients, 39,900 nodes: 26.2 -> 23.3 us;
// element rows, 1,482 elements: 14.1 -> 11.7 us).
int pass_threads(int64_t n) {
  int t = 128;
  while (t > 32 && (n + t - 1) / t < 4 * (int64_t)sm_count()) t /= 2;
  return t;
}
int pass_blocks(int64_t n) { return blocks_for(n, pass_threads(n)); }

// Whether a pass over n nodes or elements overlaps its predecessor (see
// launch_over): blocks of one warp, at most two or three on an SM.
static bool small_pass(int64_t n) { return pass_threads(n) == 32; }

// One stable pass of the radix sort on the digit at `shift` (see RadixPlan).
template <int BITS, int TILE, bool FUSED>
static pdf_status radix_pass_t(const RadixPlan& R, const int32_t* kin, const int32_t* vin, int64_t n, int shift,
                               int32_t* hist, int32_t* part, int32_t* kout, int32_t* vout, int32_t* seg,
                               int32_t n_seg, cudaStream_t st) {
  const unsigned nt = (unsigned)R.tiles;
  constexpr size_t bytes = scatter_shared<BITS>();
  if (bytes > 48 * 1024)
    PDF_CUDA(cudaFuncSetAttribute(k_radix_scatter<BITS, TILE, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)bytes));
  constexpr int kBins = 1 << BITS;
  int32_t* sums = FUSED ? nullptr : part + kBins;
  PDF_KERNEL("k_radix_hist", st, launch_over(overlap(n), k_radix_hist<BITS, TILE>, nt, kSortThreads, 0, st, kin, n, shift,
             R.sub, hist, sums););
  if (!FUSED)
    PDF_KERNEL("k_scan_bins", st, launch_over(overlap(n), k_scan_bins, dim3(kScanChunks, kBins / 32), 256, 0, st, hist,
               R.tiles, kBins, sums, part););
  PDF_KERNEL("k_radix_scatter", st, launch_over(overlap(n), k_radix_scatter<BITS, TILE, FUSED>, nt, kScatterThreads, bytes,
             st, kin, vin, n, shift, R.sub, R.tiles, hist, part, kout, vout, seg, n_seg););
  return PDF_OK;
}
template <int BITS>
static pdf_status radix_pass_b(const RadixPlan& R, const int32_t* kin, const int32_t* vin, int64_t n, int shift,
                               int32_t* hist, int32_t* part, int32_t* kout, int32_t* vout, int32_t* seg,
                               int32_t n_seg, cudaStream_t st) {
  if (R.tile == kTileSmall)  // (at most 64 tiles: always fused)
    return radix_pass_t<BITS, kTileSmall, true>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
  if (R.fused)
    return radix_pass_t<BITS, kTileLarge, true>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
  return radix_pass_t<BITS, kTileLarge, false>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
}
static pdf_status radix_pass(const RadixPlan& R, const int32_t* kin, const int32_t* vin, int64_t n, int shift,
                             int32_t* hist, int32_t* part, int32_t* kout, int32_t* vout, int32_t* seg,
                             int32_t n_seg, cudaStream_t st) {
  switch (R.bits) {
    case 6: return radix_pass_b<6>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
    case 7: return radix_pass_b<7>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
    case 8: return radix_pass_b<8>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
    case 9: return radix_pass_b<9>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
    case 10: return radix_pass_b<10>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
    default: return radix_pass_b<11>(R, kin, vin, n, shift, hist, part, kout, vout, seg, n_seg, st);
  }
}

// Stable grouping by element of n keys into the last of the passes' buffers
// (kout[pass], vout[pass]) with the segment offsets in seg.
static pdf_status group_keys(const RadixPlan& R, const int32_t* elem, int64_t n, int32_t n_tri, int32_t* hist,
                             int32_t* part, int32_t* const* kout, int32_t* const* vout, int32_t* seg,
                             cudaStream_t st) {
  const int32_t* kin = elem;
  const int32_t* vin = nullptr;  // first pass: the values are the indices
  const bool one = R.passes == 1;
  for (int pass = 0; pass < R.passes; ++pass) {
    const pdf_status s = radix_pass(R, kin, vin, n, pass * R.bits, hist, part, kout[pass], vout[pass],
                                    one ? seg : nullptr, n_tri, st);
    if (s != PDF_OK) return s;
    kin = kout[pass];
    vin = vout[pass];
  }
  if (!one)
    PDF_KERNEL("k_seg_offsets", st, launch_over(overlap(n), k_seg_offsets,
               (unsigned)((seg_offsets_threads(n) + 255) / 256), 256, 0, st, kin, n, n_tri, seg););
  return PDF_OK;
}

// Stable grouping of particles by element.  Leaves sorted element ids in
// keys[out], particle ids in vals[out] and segment offsets in seg.
pdf_status group_by_element(pdf_particles* P, cudaStream_t st) {
  const int32_t n_tri = P->mesh->d.n_tri;
  const RadixPlan R = radix_plan(P->n, key_bits_of(n_tri), kMaxBits);
  int32_t* const kout[3] = {P->keys[0], P->keys[1], P->keys[0]};
  int32_t* const vout[3] = {P->vals[0], P->vals[1], P->vals[0]};
  const pdf_status s = group_keys(R, P->elem, P->n, n_tri, P->hist, P->hist_part, kout, vout, P->seg, st);
  if (s != PDF_OK) return s;
  P->sorted_key_slot = (R.passes - 1) & 1;
  P->sorted_pid = P->vals[P->sorted_key_slot];
  return PDF_OK;
}

// Copy of every state array into the grouping's order (slot i <- slot idx[i]).
struct ReorderArgs {
  const int32_t* idx;
  int64_t n;
  const long long* src8[7];
  long long* dst8[7];
  const int32_t* src4[6];
  int32_t* dst4[6];
  int n8, n4;
};

__global__ void k_reorder(ReorderArgs R) {
  overlap_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < R.n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t j = R.idx[i];
#pragma unroll
    for (int k = 0; k < 7; ++k)
      if (k < R.n8) R.dst8[k][i] = __ldg(R.src8[k] + j);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < R.n4) R.dst4[k][i] = __ldg(R.src4[k] + j);
  }
}

// Copies the state into the grouping's order, into the second set of state
// arrays (adopt_reorder then makes them the state).
static pdf_status launch_reorder(pdf_particles* P, cudaStream_t st) {
  ReorderArgs R;
  R.idx = P->sorted_pid;
  R.n = P->n;
  R.n8 = R.n4 = 0;
  auto add8 = [&](void* src, void* dst) {
    R.src8[R.n8] = static_cast<const long long*>(src);
    R.dst8[R.n8++] = static_cast<long long*>(dst);
  };
  auto add4 = [&](void* src, void* dst) {
    R.src4[R.n4] = static_cast<const int32_t*>(src);
    R.dst4[R.n4++] = static_cast<int32_t*>(dst);
  };
  add8(P->x, P->x2);
  add8(P->y, P->y2);
  if (P->precision == PDF_FP64) {
    add8(P->u, P->u2); add8(P->v, P->v2); add8(P->w, P->w2); add8(P->om, P->om2); add8(P->ps, P->ps2);
  } else {
    add4(P->uf, P->uf2); add4(P->vf, P->vf2); add4(P->wf, P->wf2); add4(P->omf, P->omf2); add4(P->psf, P->psf2);
  }
  add4(P->pid, P->pid2);
  // one thread per particle (0.31 ms at 15.9M particles against 0.46 ms
  // for a grid of 32 blocks per SM striding over them)
  PDF_KERNEL("k_reorder", st, launch_over(overlap(P->n), k_reorder, (unsigned)((P->n + 255) / 256), 256, 0, st, R););
  return PDF_OK;
}

// Adopts the copy (host pointers only; work issued afterwards sees it): the
// sorted order becomes the storage order (sorted_pid = NULL) and the element
// ids are the sorted keys.
static void adopt_reorder(pdf_particles* P) {
  std::swap(P->x, P->x2);
  std::swap(P->y, P->y2);
  std::swap(P->u, P->u2); std::swap(P->v, P->v2); std::swap(P->w, P->w2);
  std::swap(P->om, P->om2); std::swap(P->ps, P->ps2);
  std::swap(P->uf, P->uf2); std::swap(P->vf, P->vf2); std::swap(P->wf, P->wf2);
  std::swap(P->omf, P->omf2); std::swap(P->psf, P->psf2);
  std::swap(P->pid, P->pid2);
  std::swap(P->elem, P->keys[P->sorted_key_slot]);
  P->sorted_pid = nullptr;
}

pdf_status iecm_cond(pdf_particles* P, const int32_t* seg, const int32_t* order, cudaStream_t st);

// Element statistics of the grouped particles (seg, order) into P->es.
static pdf_status elem_stats(pdf_particles* P, const int32_t* seg, const int32_t* order, cudaStream_t st) {
  const MeshDev& M = P->mesh->d;
  // one element per group of eight lanes up to 48 blocks of 256 per SM
  // (three resident at 80 registers); beyond that each group walks several
  // elements and prefetches the next one.  At 15.9M particles on 158,802
  // elements 3, 12, 24 and 48 blocks per SM took 0.29, 0.27, 0.25 and
  // 0.22 ms: with one element per group no group waits for a long one.
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)M.n_tri * kStatLanes + 255) / 256,
                                                           (int64_t)sm_count() * 48));
  auto run = [&](auto* u, auto* v, auto* w, auto* om, auto* ps) -> pdf_status {
    using T = std::remove_reference_t<decltype(*u)>;
    if (overlap(P->n) && P->n <= kOverlapPpe * M.n_tri)
      PDF_KERNEL("k_elem_stats", st, launch_over(true, k_elem_stats_grp<T, true>, nb, 256, 0, st, seg, order, M.n_tri, u,
                 v, w, om, ps, P->es));
    else
      PDF_KERNEL("k_elem_stats", st, launch_over(false, k_elem_stats_grp<T, false>, nb, 256, 0, st, seg, order, M.n_tri,
                 u, v, w, om, ps, P->es));
    return PDF_OK;
  };
  return P->precision == PDF_FP64 ? run(P->u, P->v, P->w, P->om, P->ps) : run(P->uf, P->vf, P->wf, P->omf, P->psf);
}

// Node statistics and node derivatives from the element statistics P->es
// (sec. 3.3 second pass, sec. 3.4).
pdf_status node_stats_from_elements(pdf_particles* P, cudaStream_t st) {
  const MeshDev& M = P->mesh->d;
  PDF_KERNEL("k_node_stats", st, launch_over(small_pass(M.n_nodes), k_node_stats, pass_blocks(M.n_nodes),
             pass_threads(M.n_nodes), 0, st, M.nse_off, M.nse, M.n_nodes, P->es, P->ns, P->counters + 8););
  return node_derivs_from_node_stats(P, st);
}

pdf_status node_derivs_from_node_stats(pdf_particles* P, cudaStream_t st) {
  const MeshDev& M = P->mesh->d;
  PDF_KERNEL("k_elem_grad1", st, launch_over(small_pass(M.n_tri), k_elem_grad1, pass_blocks(M.n_tri),
             pass_threads(M.n_tri), 0, st, M.tri, M.dN, M.n_tri, P->ns, P->eg););
  PDF_KERNEL("k_node_grad1", st, launch_over(small_pass(M.n_nodes), k_node_grad1, pass_blocks(M.n_nodes),
             pass_threads(M.n_nodes), 0, st, M.nse_off, M.nse, M.n_nodes, P->eg, P->nd););
  PDF_KERNEL("k_elem_grad2", st, launch_over(small_pass(M.n_tri), k_elem_grad2, pass_blocks(M.n_tri),
             pass_threads(M.n_tri), 0, st, M.tri, M.dN, M.n_tri, P->nd, P->eg););
  PDF_KERNEL("k_node_grad2", st, launch_over(small_pass(M.n_nodes), k_node_grad2, pass_blocks(M.n_nodes),
             pass_threads(M.n_nodes), 0, st, M.nse_off, M.nse, M.n_nodes, P->eg, P->nd););
  return PDF_OK;
}

pdf_status estimate_stats(pdf_particles* P, cudaStream_t st) {
  pdf_status s = group_by_element(P, st);
  if (s != PDF_OK) return s;
  if (P->reorder_every > 0 && ++P->since_reorder >= P->reorder_every) {
    // (the copy beside the statistics on a second stream gained nothing:
    // both are limited by the same gathers)
    s = launch_reorder(P, st);
    if (s != PDF_OK) return s;
    adopt_reorder(P);
    P->since_reorder = 0;
  }
  s = elem_stats(P, P->seg, P->sorted_pid, st);
  if (s != PDF_OK) return s;
  s = node_stats_from_elements(P, st);
  if (s != PDF_OK) return s;
  P->have_stats = true;
  return iecm_cond(P, P->seg, P->sorted_pid, st);
}

}  // namespace pdfgb

using namespace pdfgb;

extern "C" pdf_status pdf_estimate_stats(pdf_particles* p, const pdf_mesh* m, double* elem_stats,
                                         double* node_stats, double* node_derivs, void* stream) {
  if (!p || !m || p->mesh != m) return fail(PDF_EINVAL, "pdf_estimate_stats: NULL or mismatched handles");
  cudaStream_t st = (cudaStream_t)stream;
  pdf_status s = estimate_stats(p, st);
  if (s != PDF_OK) return s;
  const MeshDev& M = m->d;
  if (elem_stats)
    PDF_CUDA(cudaMemcpyAsync(elem_stats, p->es, sizeof(double) * M.n_tri * PDF_NES, cudaMemcpyDefault, st));
  if (node_stats)
    PDF_CUDA(cudaMemcpyAsync(node_stats, p->ns, sizeof(double) * M.n_nodes * PDF_NNS, cudaMemcpyDefault, st));
  if (node_derivs)
    PDF_CUDA(cudaMemcpyAsync(node_derivs, p->nd, sizeof(double) * M.n_nodes * PDF_NND, cudaMemcpyDefault, st));
  return PDF_OK;
}

namespace pdfgb {

// Statistics with caller-chosen grouping buffers (used by the
// allocation-free entry point in noalloc.cu).  keys_b/vals_b receive the
// result; at most two passes of 9-bit digits, so n_tri <= 2^18, and at most
// kFusedTiles tiles, so that no pass scans (there is no space for a scan's
// sums); hist holds hist_len entries.
static_assert((PDF_NOALLOC_MAX_PARTICLES + kTileLarge - 1) / kTileLarge <= kFusedTiles,
              "the largest set without allocations is grouped without a scan");
static_assert(PDF_NOALLOC_MAX_ELEMENTS <= 1 << 18, "two digits of 9 bits");
pdf_status estimate_stats_with_buffers(pdf_particles* P, int32_t* keys_a, int32_t* vals_a,
                                       int32_t* keys_b, int32_t* vals_b, int32_t* hist,
                                       int64_t hist_len, int32_t* seg, cudaStream_t st) {
  const MeshDev& M = P->mesh->d;
  const RadixPlan R = radix_plan(P->n, key_bits_of(M.n_tri), 9);
  if (R.passes > 2 || !R.fused || (R.tiles << R.bits) > hist_len)
    return fail(PDF_EINVAL, "estimate_stats_with_buffers: the grouping's plan does not fit the buffers");
  int32_t* const kout[2] = {R.passes == 2 ? keys_a : keys_b, keys_b};
  int32_t* const vout[2] = {R.passes == 2 ? vals_a : vals_b, vals_b};
  pdf_status s = group_keys(R, P->elem, P->n, M.n_tri, hist, nullptr, kout, vout, seg, st);
  if (s != PDF_OK) return s;
  const int32_t* vin = vals_b;
  s = elem_stats(P, seg, vin, st);
  if (s != PDF_OK) return s;
  s = node_stats_from_elements(P, st);
  if (s != PDF_OK) return s;
  P->have_stats = true;
  return iecm_cond(P, seg, vin, st);
}

// Stable LSD radix sort of n non-negative int32 keys below 2^bits, the
// values the original indices; ping-pong buffers k0/v0, k1/v1 of n entries,
// hist of radix_hist_len(n, bits) and hist_part of radix_part_len() entries,
// zeroed once.
// *keys_out / *vals_out receive the sorted buffers.
pdf_status radix_sort_index(const int32_t* keys, int64_t n, int bits, int32_t* k0, int32_t* v0, int32_t* k1,
                            int32_t* v1, int32_t* hist, int32_t* hist_part, const int32_t** keys_out,
                            const int32_t** vals_out, cudaStream_t st) {
  const RadixPlan R = radix_plan(n, bits, kMaxBits);
  const int32_t* kin = keys;
  const int32_t* vin = nullptr;
  int32_t* kout[2] = {k0, k1};
  int32_t* vout[2] = {v0, v1};
  for (int pass = 0; pass < R.passes; ++pass) {
    int32_t* ko = kout[pass & 1];
    int32_t* vo = vout[pass & 1];
    const pdf_status s = radix_pass(R, kin, vin, n, pass * R.bits, hist, hist_part, ko, vo, nullptr, 0, st);
    if (s != PDF_OK) return s;
    kin = ko;
    vin = vo;
  }
  *keys_out = kin;
  *vals_out = vin;
  return PDF_OK;
}

}  // namespace pdfgb
