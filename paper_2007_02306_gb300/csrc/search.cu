// Clutter-resistant search on sm_103a (Section 3.2: Listing 1, Eq. distanceFunctionExpression;
// ranking of Section 4.1 with the tie rule of Section 4.2).
//
// d(i, j) = sum over r in [0,N), c in [1,N) with a != 0 of (a - b)^2, a and b the needle's and
// haystack's column deltas.  rank_i = #{j : d(i,j) < d(i,match_i)}, top1_i = smallest j with
// minimal d(i,j).  Everything is integer arithmetic, so results are exact.
//
// Stages:
//   k_encode_needles, k_encode_groups   per image: int8 column deltas (delta of column 0 := 0);
//                   for needles also a byte mask of the non-zero deltas and per-row sums of
//                   squared deltas, for the haystack groups of 32 images, piece-major; images
//                   with any |delta| > 127 are "wide" and listed apart.
//   k_true_distance d(i, match_i) in int64 straight from the uint16 images.
//   k_dense         narrow x narrow pairs on CUDA cores.  Per row, sum m(a-b)^2 =
//                   sum a^2 + sum (mb)^2 - 2 sum ab with sum a^2 precomputed and the other two
//                   as dp4a over 4 packed deltas (plus one AND for mb); each row's sum is >= 0,
//                   so partial sums are monotone and a pair stops once it exceeds
//                   d(i, match_i) (the early exit of Section 4.4, which never changes a rank).
//                   A block keeps 4 needles in shared memory and sweeps a band of haystack
//                   tiles (1,024 images each, four per thread at N <= 64), rows heaviest
//                   first; each broadcast needle word serves all of a thread's images.
//   k_wide          pairs with a wide side: Listing 1 over the needle's non-zero deltas in
//                   int64, reading the uint16 images.
//   k_finalize      combines counts and top-1 candidates.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"

namespace rici {
namespace {

constexpr int kDenseThreads = 256;     // threads of a dense block
constexpr int64_t kBandMax = 8;        // haystack tiles per band of the dense work order
constexpr int kWideThreads = 256;
constexpr unsigned long long kNoBest = ~0ull;

__device__ __forceinline__ int delta_at(const uint16_t *img, int N, int r, int c) {
  return c == 0 ? 0 : (int)img[r * N + c] - (int)img[r * N + c - 1];
}

// Four deltas clamped to [-127, 127] as the bytes of a word.
__device__ __forceinline__ uint32_t pack_deltas(int a, int b, int c, int d) {
  a = min(max(a, -127), 127);
  b = min(max(b, -127), 127);
  c = min(max(c, -127), 127);
  d = min(max(d, -127), 127);
  return __byte_perm(__byte_perm((uint32_t)a, (uint32_t)b, 0x0040),
                     __byte_perm((uint32_t)c, (uint32_t)d, 0x0040), 0x5410);
}
// 0xff in every byte of w that is not zero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t w) {
  const uint32_t t = (w | ((w & 0x7f7f7f7fu) + 0x7f7f7f7fu)) & 0x80808080u;  // bit 7: not zero
  return (t >> 7) * 0xffu;
}
// The 8 pixels at flat position k0 (a multiple of 8) of an image; vec: one 16-byte load.
__device__ __forceinline__ uint4 load_pixels8(const uint16_t *img, int k0, bool vec) {
  if (vec) return *reinterpret_cast<const uint4 *>(img + k0);
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e)
    w[e] = (uint32_t)img[k0 + 2 * e] | ((uint32_t)img[k0 + 2 * e + 1] << 16);
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Needle side of the CUDA-core forms, one warp per image, 256 pixels per pass (rows_of_8(N)):
// image-major int8 deltas, byte masks of the non-zero ones and, with row_sq, the sum of each
// row's squared (clamped) deltas, [n][N].
__global__ void k_encode_needles(const uint16_t *__restrict__ imgs, int64_t n, int N,
                                 int8_t *__restrict__ delta, int8_t *__restrict__ mask,
                                 int *__restrict__ wide_flag, int *__restrict__ wide_list,
                                 int *__restrict__ wide_count, int *__restrict__ row_sq) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int K = N * N, rl = N / 8;  // rl: lanes of a row (a power of two, at most 16)
  const bool vec = aligned16(imgs);
  for (int64_t i = w; i < n; i += nw) {
    const uint16_t *img = imgs + i * K;
    int wide = 0;
#pragma unroll 4
    for (int base = 0; base < K; base += 256) {
      const int k0 = base + lane * 8;
      const bool in = k0 < K;
      int d[8];
      deltas8(in ? load_pixels8(img, k0, vec) : make_uint4(0, 0, 0, 0), lane, N, d);
#pragma unroll
      for (int e = 0; e < 8; ++e) wide |= d[e] > 127 || d[e] < -127;
      const uint2 a = make_uint2(pack_deltas(d[0], d[1], d[2], d[3]),
                                 pack_deltas(d[4], d[5], d[6], d[7]));
      if (in) {
        *reinterpret_cast<uint2 *>(delta + i * K + k0) = a;
        // from the deltas themselves: a wide delta is not zero
        *reinterpret_cast<uint2 *>(mask + i * K + k0) =
            make_uint2(nonzero_bytes(a.x), nonzero_bytes(a.y));
      }
      if (row_sq) {
        int sq = __dp4a((int)a.x, (int)a.x, __dp4a((int)a.y, (int)a.y, 0));
        for (int k = 1; k < rl; k <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, k);
        if (in && (lane & (rl - 1)) == 0) row_sq[i * N + k0 / N] = sq;
      }
    }
    wide = __any_sync(0xffffffffu, wide);
    if (lane == 0) {
      wide_flag[i] = wide;
      if (wide) wide_list[atomicAdd(wide_count, 1)] = (int)i;
    }
  }
}

// Haystack side of the CUDA-core forms: int8 deltas of groups of 32 consecutive images, so that the
// 32 lanes of a warp (one image each) read the same piece of their images with one contiguous
// access.  Within a group the 32-bit words (4 deltas) of an image are cut into pieces of CW words,
// piece-major: piece v of image l is at word (v * 32 + l) * CW.
//   CW = min(4, N / 4)  k_dense: pieces of 16 bytes within a row (a warp reads 512 bytes)
//   CW = 1              k_sparse: any word of the 32 images is one 128-byte line
// list (optional): encode images list[0 .. *list_count) of imgs as images 0, 1, ... (a compacted
// subset, count read on the device; n is then an upper bound).  Images past the last are zero.
// wide_flag and narrow (bit l of word g: image 32 g + l exists and is not wide; zero words up to
// a multiple of four groups) are optional.
// One block per group; 256 pixels of its images at a time cross through shared memory, so that
// both the reads (512 bytes of an image) and the writes are contiguous.  Writing from one warp
// per image instead left 1 or 16 bytes in every 128-byte line (262,144 images of 64 x 64:
// 2.2 ms with CW = 1, 1.5 ms per 90,000 with CW = 4).
constexpr int kGroupWarps = 8;
template <int CW>
__global__ void __launch_bounds__(kGroupWarps * 32) k_encode_groups(
    const uint16_t *__restrict__ imgs, int64_t n, int N, int8_t *__restrict__ delta,
    int *__restrict__ wide_flag, int *__restrict__ wide_list, int *__restrict__ wide_count,
    const int *__restrict__ list, const int *__restrict__ list_count,
    uint32_t *__restrict__ narrow) {
  __shared__ uint32_t group_wide;
  constexpr int kPerW = 32 / kGroupWarps;  // images of a warp
  __shared__ uint32_t tile[64][33];        // [word of the 256 pixels][image]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int K = N * N;
  if (list) n = *list_count < n ? *list_count : n;
  const bool vec = aligned16(imgs);
  for (int64_t g = blockIdx.x; g * 32 < n; g += gridDim.x) {
    int wide[kPerW];
    const uint16_t *img[kPerW];
    if (threadIdx.x == 0) group_wide = 0;  // (read by nobody before the barriers below)
#pragma unroll
    for (int q = 0; q < kPerW; ++q) {
      const int64_t i = g * 32 + warp * kPerW + q;
      wide[q] = 0;
      img[q] = i < n ? imgs + (list ? (int64_t)list[i] : i) * K : nullptr;
    }
    uint32_t *out = reinterpret_cast<uint32_t *>(delta) + g * (int64_t)(K / 4) * 32;
    for (int base = 0; base < K; base += 256) {
      const int k0 = base + lane * 8;
      uint4 px[kPerW];
#pragma unroll
      for (int q = 0; q < kPerW; ++q)
        px[q] = k0 < K && img[q] ? load_pixels8(img[q], k0, vec) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int q = 0; q < kPerW; ++q) {
        int d[8];
        deltas8(px[q], lane, N, d);
#pragma unroll
        for (int e = 0; e < 8; ++e) wide[q] |= d[e] > 127 || d[e] < -127;
        tile[2 * lane][warp * kPerW + q] = pack_deltas(d[0], d[1], d[2], d[3]);
        tile[2 * lane + 1][warp * kPerW + q] = pack_deltas(d[4], d[5], d[6], d[7]);
      }
      __syncthreads();
      const int nv = min(64, (K - base) / 4) / CW;  // pieces of these pixels
      for (int v = warp; v < nv; v += kGroupWarps) {
        uint32_t *dst = out + ((int64_t)(base / 4 / CW + v) * 32 + lane) * CW;
        if constexpr (CW == 4)
          *reinterpret_cast<uint4 *>(dst) = make_uint4(tile[4 * v][lane], tile[4 * v + 1][lane],
                                                       tile[4 * v + 2][lane], tile[4 * v + 3][lane]);
        else if constexpr (CW == 2)
          *reinterpret_cast<uint2 *>(dst) = make_uint2(tile[2 * v][lane], tile[2 * v + 1][lane]);
        else
          *dst = tile[v][lane];
      }
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kPerW; ++q) {
      const int any = __any_sync(0xffffffffu, wide[q]);
      const int64_t i = g * 32 + warp * kPerW + q;
      if (lane == 0 && i < n) {
        if (wide_flag) wide_flag[i] = any;
        if (any) {
          wide_list[atomicAdd(wide_count, 1)] = (int)i;
          atomicOr(&group_wide, 1u << (warp * kPerW + q));
        }
      }
    }
    if (narrow) {
      __syncthreads();
      if (threadIdx.x == 0) {
        const int64_t left = n - g * 32;
        narrow[g] = ~group_wide & (left >= 32 ? 0xffffffffu : (1u << left) - 1u);
        if (left <= 32)
          for (int64_t e = g + 1; e & 3; ++e) narrow[e] = 0;
      }
      __syncthreads();
    }
  }
}

// Exact int64 distance of one pair, one warp.  kRows (rows_of_8(N), both images 16-byte aligned): 256
// pixels per pass, else 32.  Two instantiations, so that the kernels of the second form keep the few
// registers of its loop (k_distances 31 against 42: 2,000 x 3,000 distances of 33 x 33 11.1 against
// 14.8 ms with both in one).
template <bool kRows>
__device__ int64_t warp_crss(const uint16_t *n, const uint16_t *h, int N) {
  const int lane = threadIdx.x & 31;
  const int K = N * N;
  unsigned long long s = 0;
  if constexpr (kRows) {
#pragma unroll 4
    for (int base = 0; base < K; base += 256) {
      const int k0 = base + lane * 8;
      const bool in = k0 < K;
      int a[8], b[8];
      deltas8(in ? load_pixels8(n, k0, true) : make_uint4(0, 0, 0, 0), lane, N, a);
      deltas8(in ? load_pixels8(h, k0, true) : make_uint4(0, 0, 0, 0), lane, N, b);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const unsigned x = a[e] != 0 ? (unsigned)abs(a[e] - b[e]) : 0u;  // at most 131,070
        s += (unsigned long long)x * x;
      }
    }
  } else {
    for (int k = lane; k < K; k += 32) {
      int r = k / N, c = k - r * N;
      if (c == 0) continue;
      int a = delta_at(n, N, r, c);
      if (a != 0) {
        long long d = (long long)a - (long long)delta_at(h, N, r, c);
        s += (unsigned long long)(d * d);
      }
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  return (int64_t)__shfl_sync(0xffffffffu, s, 0);
}

// Also sets up each needle's rank, minimum and flags.
template <bool kRows>
__global__ void k_true_distance(const SearchScene *__restrict__ tab, const int *__restrict__ qscene,
                                int64_t Qtot, int N, int64_t *__restrict__ dtrue,
                                int *__restrict__ rank, unsigned long long *__restrict__ best,
                                int *__restrict__ flags, int *__restrict__ top1_flag, int *status) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t K = (int64_t)N * N;
  for (int64_t i = w; i < Qtot; i += nw) {
    const SearchScene &sc = tab[scene_at(qscene, i)];
    const int64_t il = i - sc.qoff;
    const int64_t m = sc.match ? sc.match[il] : il;
    if (lane == 0) top1_flag[i] = 0;
    if (m < 0 || m >= sc.H) {
      if (lane == 0) {
        set_status(status, RICI_ERR_INDEX_OUT_OF_RANGE);
        dtrue[i] = -1;
        rank[i] = -1;
        best[i] = kNoBest;
        flags[i] = 2;  // invalid: no search for this needle
      }
      continue;
    }
    int64_t d = warp_crss<kRows>(sc.needles + il * K, sc.haystack + m * K, N);
    if (lane == 0) {
      dtrue[i] = d;
      rank[i] = 0;
      best[i] = kNoBest;
      flags[i] = 0;
    }
  }
}

// Scene of every launch-wide needle and haystack image.
__global__ void k_scene_index(const SearchScene *__restrict__ tab, int ns, int64_t Qtot,
                              int64_t Htot, int *__restrict__ qscene, int *__restrict__ hscene) {
  const int64_t n = Qtot > Htot ? Qtot : Htot;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x) {
    if (x < Qtot) {
      int lo = 0, hi = ns - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab[mid].qoff <= x) lo = mid; else hi = mid - 1;
      }
      qscene[x] = lo;
    }
    if (x < Htot) {
      int lo = 0, hi = ns - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab[mid].hoff <= x) lo = mid; else hi = mid - 1;
      }
      hscene[x] = lo;
    }
  }
}

constexpr int kCounts = 16;  // list lengths of a call, zeroed with its scene table
constexpr int kFillChunk = 150;
struct SearchFill {
  SearchScene e[kFillChunk];
  int n;
};
__global__ void k_fill_search_table(SearchScene *dst, SearchFill f, int *counts, int ncounts) {
  if (threadIdx.x < ncounts) counts[threadIdx.x] = 0;
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) dst[i] = f.e[i];
}

__device__ __forceinline__ unsigned long long pack_best(int64_t d, int64_t j) {
  unsigned long long dd = d >= 0xffffffffll ? 0xffffffffull : (unsigned long long)d;
  return (dd << 32) | (unsigned long long)(uint32_t)j;
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    unsigned long long o = __shfl_down_sync(0xffffffffu, v, d);
    v = o < v ? o : v;
  }
  return v;
}

// Narrow x narrow pairs.  Block: kTQ needles (deltas + masks in shared memory) x
// kDenseThreads * kImg haystack images (kImg per thread, in consecutive groups of 32).
template <int N, int kTQ, int kImg, bool kCount, bool kCounted>
__global__ void __launch_bounds__(kDenseThreads, (N * kImg <= 64 ? 4 : 2) * 256 / kDenseThreads)
    k_dense(
    const int8_t *__restrict__ ndelta, const int8_t *__restrict__ nmask,
    const int *__restrict__ nrowsq, const int *__restrict__ nwide, int64_t Q,
    const int8_t *__restrict__ hdelta,
    const int *__restrict__ hwide, int64_t H, const int64_t *__restrict__ dtrue,
    const int *__restrict__ nflags, int *__restrict__ rank, unsigned long long *__restrict__ best,
    unsigned long long *__restrict__ counters, int64_t tile0, int64_t tiles_q, int64_t tiles_h,
    int64_t band_h, int64_t blocks, const int *__restrict__ hcount,
    const int *__restrict__ hmap, const int *__restrict__ gate) {
  // kCounted: the haystack holds *hcount images (H is an upper bound), usually far fewer, so the grid
  // is bounded and its blocks step through the `blocks` work items (a grid for H took 0.1-0.2 ms to
  // find nothing to do in 131,072 blocks); otherwise one block per item.
  // hmap (optional): haystack image j is image hmap[j] of the caller's haystack (a compacted subset)
  // gate (optional): *gate == 0 means no needle is ranked here, and every block returns at once
  constexpr int WPR = N / 4;  // 32-bit words per row
  constexpr int K = N * N;
  extern __shared__ int2 am_raw[];  // [kTQ][K/4] (needle delta word, mask word)
  auto am = reinterpret_cast<int2(*)[K / 4]>(am_raw);
  __shared__ int thr_s[kTQ];
  __shared__ int act_s[kTQ];
  __shared__ int wrow[kTQ][N];     // sum of squared needle deltas per (needle, row)
  __shared__ int ord[N];           // rows by decreasing tile weight
  __shared__ unsigned rmask[N];    // needles of the tile with a non-zero delta in the row
  __shared__ int nrows_s;
  const int tid = threadIdx.x, lane = tid & 31;
  // Work order: bands of band_h haystack tiles.  A block holds one needle tile and sweeps the
  // haystack tiles of one band; consecutive blocks take consecutive needle tiles of the same band,
  // so a band's haystack images are read from DRAM once and reused from L2 by every needle tile,
  // and the needle tile's set-up (shared-memory fill, row order) is paid once per band.
  if (gate && *gate == 0) return;  // uniform over the grid
  if (kCounted) H = *hcount < H ? *hcount : H;
  int64_t L = tile0 + blockIdx.x;
  do {
    const int64_t band = L / tiles_q, qt = L - band * tiles_q;
    const int64_t h0 = band * band_h;
    const int64_t h1 = tiles_h - h0 < band_h ? tiles_h : h0 + band_h;
    const int64_t q0 = qt * kTQ;
    if (kCounted) {
      // bands ascend: nothing is left for this block (uniform over the block)
      if (h0 * (int64_t)(kDenseThreads * kImg) >= H) return;
      __syncthreads();  // the item before is done with the shared arrays
    }

    bool act = false;
    if (tid < kTQ) {
      const int64_t q = q0 + tid;
      act = q < Q && nflags[q] == 0 && !nwide[q];
      int64_t t = act ? dtrue[q] : -1;
      thr_s[tid] = t > 0x7fffffffll ? 0x7fffffff : (int)t;
      act_s[tid] = act;
    }
    if (!__syncthreads_or(act)) continue;  // no needle of this tile is ranked here
    for (int x = tid; x < kTQ * (K / 4); x += kDenseThreads) {
      int q = x / (K / 4), wd = x - q * (K / 4);
      int a = 0, m = 0;
      if (q0 + q < Q) {
        a = reinterpret_cast<const int *>(ndelta + (q0 + q) * K)[wd];
        m = reinterpret_cast<const int *>(nmask + (q0 + q) * K)[wd];
      }
      am[q][wd] = make_int2(a, m);
    }
    __syncthreads();
    // Rows are visited heaviest first so that distances pass the early-exit threshold sooner;
    // the sum is order independent, so the result is unchanged.  Rows where no needle of the
    // tile has a non-zero delta contribute nothing and are skipped.
    for (int x = tid; x < kTQ * N; x += kDenseThreads) {
      int q = x / N, r = x - q * N;
      wrow[q][r] = act_s[q] ? nrowsq[(q0 + q) * N + r] : 0;
    }
    __syncthreads();
    __shared__ int tile_w[N];
    if (tid < N) {
      int W = 0;
      unsigned msk = 0;
#pragma unroll
      for (int q = 0; q < kTQ; ++q) {
        W += wrow[q][tid];
        if (wrow[q][tid] > 0) msk |= 1u << q;
      }
      rmask[tid] = msk;
      tile_w[tid] = W;
    }
    __syncthreads();
    if (tid < N) {
      const int W = tile_w[tid];
      int rk = 0, nz = 0;
      for (int r2 = 0; r2 < N; ++r2) {
        const int W2 = tile_w[r2];
        rk += (W2 > W) || (W2 == W && r2 < tid);
        nz += W2 > 0;
      }
      ord[rk] = tid;
      if (tid == 0) nrows_s = nz;
    }
    __syncthreads();
    const int nrows = nrows_s;

    constexpr int kTile = kDenseThreads * kImg;  // haystack images per tile
    constexpr int CW = WPR < 4 ? WPR : 4;
    constexpr int64_t kGroupWords = (int64_t)N * WPR * 32;  // one group of 32 interleaved images
    const int warp = tid >> 5;
    for (int64_t ht = h0; ht < h1; ++ht) {
      // this thread's images: j0 + 32 k, k < kImg (a warp owns kImg consecutive groups of 32)
      const int64_t j0 = ht * kTile + (int64_t)warp * (32 * kImg) + lane;
      int acc[kImg][kTQ];  // partial distance minus the needle's true distance (exit once > 0)
      unsigned alive[kImg];
      unsigned inrange = 0;  // images of this thread inside the haystack (their rows are loaded)
#pragma unroll
      for (int k = 0; k < kImg; ++k) {
        const int64_t j = j0 + 32 * k;
        const bool valid = j < H && !hwide[j];
        if (j < H) inrange |= 1u << k;
        alive[k] = 0;
#pragma unroll
        for (int q = 0; q < kTQ; ++q) {
          acc[k][q] = -thr_s[q];
          if (valid && act_s[q]) alive[k] |= 1u << q;
        }
      }
      const int *hgrp = reinterpret_cast<const int *>(hdelta) + (j0 >> 5) * kGroupWords + lane * CW;
      unsigned long long pair_rows = 0, lane_slots = 0;
      int hw[kImg][WPR];
#pragma unroll
      for (int k = 0; k < kImg; ++k)
#pragma unroll
        for (int v = 0; v < WPR; ++v) hw[k][v] = 0;
      for (int i = 0; i < nrows; ++i) {
        unsigned any = 0;
#pragma unroll
        for (int k = 0; k < kImg; ++k) any |= alive[k];
        if (__ballot_sync(0xffffffffu, any != 0) == 0) break;
        const int r = ord[i];
        const unsigned rm = rmask[r];
        unsigned use[kImg], uor = 0;
#pragma unroll
        for (int k = 0; k < kImg; ++k) {
          use[k] = alive[k] & rm;
          uor |= use[k];
          if (kCount) pair_rows += __popc(use[k]);
        }
        const unsigned wuse = __reduce_or_sync(0xffffffffu, uor);  // needles any lane still needs
#pragma unroll
        for (int k = 0; k < kImg; ++k) {
          // every row of an image inside the haystack is loaded, even once its pairs have all
          // exited: a uniform load is cheaper than the divergent branch that would skip it
          if ((inrange >> k) & 1u) {
            const int *src = hgrp + k * kGroupWords + r * (WPR * 32);
#pragma unroll
            for (int v = 0; v < WPR / CW; ++v) {
              if constexpr (CW == 4) {
                const int4 x = *reinterpret_cast<const int4 *>(src + v * 32 * CW);
                hw[k][4 * v] = x.x;
                hw[k][4 * v + 1] = x.y;
                hw[k][4 * v + 2] = x.z;
                hw[k][4 * v + 3] = x.w;
              } else {
                const int2 x = *reinterpret_cast<const int2 *>(src + v * 32 * CW);
                hw[k][2 * v] = x.x;
                hw[k][2 * v + 1] = x.y;
              }
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kTQ; ++q) {
          if (((wuse >> q) & 1u) == 0) continue;
          if (kCount) lane_slots += kImg;  // kImg warp-wide needle-row iterations (32 lane slots each)
          // row sum of m (a - b)^2 = sum a^2 + sum (m b)^2 - 2 sum a b, with sum a^2 precomputed;
          // the (m b)^2 chain starts from the running value, and one chain per term and image
          // suffices because the warps of the block hide the dp4a latency
          const int w = wrow[q][r];
          int sb[kImg], sa[kImg];
#pragma unroll
          for (int k = 0; k < kImg; ++k) {
            sb[k] = acc[k][q] + w;
            sa[k] = 0;
          }
          const int4 *amq = reinterpret_cast<const int4 *>(&am[q][r * WPR]);
#pragma unroll
          for (int v = 0; v < WPR; v += 2) {
            const int4 x = amq[v >> 1];  // (a_v, m_v, a_v+1, m_v+1)
#pragma unroll
            for (int k = 0; k < kImg; ++k) {
              const int b0 = hw[k][v], b1 = hw[k][v + 1];
              const int bm0 = b0 & x.y, bm1 = b1 & x.w;
              sb[k] = __dp4a(bm0, bm0, sb[k]);
              sa[k] = __dp4a(x.x, b0, sa[k]);
              sb[k] = __dp4a(bm1, bm1, sb[k]);
              sa[k] = __dp4a(x.z, b1, sa[k]);
            }
          }
#pragma unroll
          for (int k = 0; k < kImg; ++k) {
            // an image whose pair has exited keeps computing with stale deltas; its value is
            // never read again, since only pairs still alive are counted
            acc[k][q] = sb[k] - 2 * sa[k];
            if (acc[k][q] > 0) alive[k] &= ~(1u << q);
          }
        }
      }
      // count and top-1 candidates (pairs that never exceeded the threshold hold exact values)
#pragma unroll
      for (int q = 0; q < kTQ; ++q) {
        if (!act_s[q]) continue;
        int c = 0;
        unsigned long long b = kNoBest;
#pragma unroll
        for (int k = 0; k < kImg; ++k) {
          const bool fin = (alive[k] >> q) & 1u;
          c += fin && acc[k][q] < 0;
          const int64_t jj = j0 + 32 * k;
          const unsigned long long bk =
              fin ? pack_best(acc[k][q] + thr_s[q], hmap ? (int64_t)hmap[jj] : jj) : kNoBest;
          b = bk < b ? bk : b;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) c += __shfl_down_sync(0xffffffffu, c, d);
        b = warp_min_u64(b);
        if (lane == 0) {
          if (c) atomicAdd(&rank[q0 + q], c);
          if (b != kNoBest) atomicMin(&best[q0 + q], b);
        }
      }
      if (kCount) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) pair_rows += __shfl_down_sync(0xffffffffu, pair_rows, d);
        if (lane == 0 && pair_rows) atomicAdd(counters, pair_rows);
        if (lane == 0 && lane_slots) atomicAdd(counters + 3, 32ull * lane_slots);
      }
    }
  } while (kCounted && (L += gridDim.x) < blocks);
}

// Sparse-needle form.  Listing 1 only touches positions where the needle's delta is non-zero, so
// each needle is reduced to the list of its 32-bit words (4 deltas) holding a non-zero delta:
// entry = (a word, mask word, byte offset of the word in the word-major haystack group,
// sum of the word's squared deltas).  Each word adds m(a-b)^2 >= 0 over its 4 positions, so the
// partial sum may be compared with d(i, match_i) after any word; words are listed heaviest
// first (descending sum a^2, in 64 logarithmic classes) so that pairs pass the threshold sooner.
// The order decides only when a pair stops, never its result.
constexpr int kSparseWarps = 8;   // needles per block, one per warp
constexpr int kSparseImg = 4;     // haystack images per lane
constexpr int kSparseStepLong = 2;  // needle words per step after the first two (loads of a step are
                                    // in flight together; four spill the sweep's registers: 16,384
                                    // sparse needles x 262,144 5.4 against 4.3 ms)
constexpr int64_t kSparseBandMax = 64;  // haystack tiles per band of the sparse work order

__device__ __forceinline__ int sparse_class(int wsq) {  // 0 = heaviest
  const int lg = 31 - __clz(wsq);
  const int frac = lg >= 2 ? (wsq >> (lg - 2)) & 3 : (wsq << (2 - lg)) & 3;
  return 63 - (4 * lg + frac);
}

// One warp per needle: the needle's non-zero words as sparse entries, heaviest class first
// (order inside a class is arbitrary).  ent: [Q][K/4] int4 slabs; ecount[i] = entries of i.
__global__ void __launch_bounds__(256) k_sparse_needles(const int8_t *__restrict__ nd,
                                                        const int8_t *__restrict__ nm, int64_t Q,
                                                        int N, int4 *__restrict__ ent,
                                                        int *__restrict__ ecount) {
  __shared__ int cls_n[8][64];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int KW = N * N / 4;
  int *cnt = cls_n[wib];
  for (int64_t i = w0; i < Q; i += nw) {
    const int *a32 = reinterpret_cast<const int *>(nd + i * (int64_t)N * N);
    const int *m32 = reinterpret_cast<const int *>(nm + i * (int64_t)N * N);
    cnt[lane] = 0;
    cnt[lane + 32] = 0;
    __syncwarp();
    for (int w = lane; w < KW; w += 32) {
      const int a = a32[w];
      if (a != 0) atomicAdd(&cnt[sparse_class(__dp4a(a, a, 0))], 1);
    }
    __syncwarp();
    // exclusive scan of the 64 class sizes (two per lane)
    const int c0 = cnt[2 * lane], c1 = cnt[2 * lane + 1];
    int incl = c0 + c1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    cnt[2 * lane] = incl - c0 - c1;
    cnt[2 * lane + 1] = incl - c1;
    __syncwarp();
    int4 *e = ent + i * (int64_t)KW;
    for (int w = lane; w < KW; w += 32) {
      const int a = a32[w];
      if (a != 0) {
        const int wsq = __dp4a(a, a, 0);
        const int pos = atomicAdd(&cnt[sparse_class(wsq)], 1);
        e[pos] = make_int4(a, m32[w], w * 128, wsq);
      }
    }
    if (lane == 0) ecount[i] = total;
    __syncwarp();
  }
}

// Narrow needles x narrow haystack images over the needles' sparse entries.  Block: kSparseWarps
// needles (one per warp) sweeping a band of haystack tiles of 32 * kSparseImg images; lane l of a
// warp holds images j0 + l + 32 k.  Most pairs of sparse needles stop within a word or two, so a tile
// is decided by the needle's first two words where it can be: both stay in registers for the band,
// their words of the next tile are loaded (one coalesced 128-byte access per entry and 32 images, at
// constant distances from one running address) before the current tile is summed, and where every
// image is narrow and none is left the tile ends at one vote.  104 instructions per needle and tile; half of
// the issue slots are used, the gathers' latency is the first stall (2,048 needles x 65,536 images), and
// with a quarter of the words (32 x 32 images) it is as fast.  16,384 sparse needles x 262,144 images of 64 x
// 64, whole calls: 7.8 ms with early loads alone, 4.4 ms with the constant distances and the single vote (64
// registers, four blocks per SM; three 5.2 ms).  Groups held in shared memory instead of gathers
// were slower (+0.8 ms), as was deciding by one word (+0.65 ms).
// The images of a tile that the needle's first two words leave: the further entries, 32 at a time
// through shared memory (`stage`, one per lane; registers would hold a step's four), kSparseStepLong
// per step with their loads in flight together, then the count and the minimum.  Warp collective;
// returns the words this lane evaluated.  (Inlined: as a call it spilled the sweep's registers.)
template <int N, bool kCount>
__device__ __forceinline__ unsigned long long sparse_rest(const int8_t *tile, const int4 *e, int ne,
                                                          int (&acc)[kSparseImg], unsigned alive,
                                                          int thr, int j0, int4 *stage, int *rank,
                                                          unsigned long long *best,
                                                          unsigned long long &lane_slots) {
  constexpr int kGroup = N * N / 4 * 128;
  const int lane = threadIdx.x & 31;
  unsigned long long pair_words = 0;
  for (int i = 2; i < ne; i += kSparseStepLong) {
    if (__ballot_sync(0xffffffffu, alive != 0) == 0) return pair_words;
    if (((i - 2) & 31) == 0) {
      __syncwarp();
      stage[lane] = i + lane < ne ? e[i + lane] : make_int4(0, 0, 0, 0);
      __syncwarp();
    }
    const int4 *E = stage + ((i - 2) & 31);
    if (kCount) {
      const int n = ne - i < kSparseStepLong ? ne - i : kSparseStepLong;
      pair_words += (unsigned long long)__popc(alive) * n;
      lane_slots += (unsigned long long)kSparseImg * n;
    }
    int w[kSparseStepLong][kSparseImg];
#pragma unroll
    for (int u = 0; u < kSparseStepLong; ++u) {
      const int8_t *p = tile + E[u].z;
#pragma unroll
      for (int k = 0; k < kSparseImg; ++k)
        w[u][k] = (alive >> k) & 1u ? *reinterpret_cast<const int *>(p + k * kGroup) : 0;
    }
#pragma unroll
    for (int u = 0; u < kSparseStepLong; ++u) {
      const int4 x = E[u];
#pragma unroll
      for (int k = 0; k < kSparseImg; ++k) {
        const int bm = w[u][k] & x.y;
        acc[k] = __dp4a(bm, bm, acc[k] + x.w) - 2 * __dp4a(x.x, w[u][k], 0);
      }
    }
#pragma unroll
    for (int k = 0; k < kSparseImg; ++k)
      if (acc[k] > 0) alive &= ~(1u << k);  // images that have exited keep stale sums
  }
  if (__ballot_sync(0xffffffffu, alive != 0) == 0) return pair_words;
  int c = 0;
  unsigned long long bb = kNoBest;
#pragma unroll
  for (int k = 0; k < kSparseImg; ++k) {
    const bool fin = (alive >> k) & 1u;
    c += fin && acc[k] < 0;
    const unsigned long long bk = fin ? pack_best(acc[k] + thr, j0 + 32 * k) : kNoBest;
    bb = bk < bb ? bk : bb;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) c += __shfl_down_sync(0xffffffffu, c, d);
  bb = warp_min_u64(bb);
  if (lane == 0) {
    if (c) atomicAdd(rank, c);
    if (bb != kNoBest) atomicMin(best, bb);
  }
  return pair_words;
}

template <int N, bool kCount>
__global__ void __launch_bounds__(kSparseWarps * 32, 4) k_sparse(
    const int4 *__restrict__ ent, const int *__restrict__ ecount,
    const int *__restrict__ nwide, int64_t Q, const int8_t *__restrict__ hword,
    const uint4 *__restrict__ narrow, int64_t H, const int64_t *__restrict__ dtrue,
    const int *__restrict__ nflags, int *__restrict__ rank, unsigned long long *__restrict__ best,
    unsigned long long *__restrict__ counters, int64_t tile0, int64_t tiles_q, int64_t tiles_h,
    int64_t band_h) {
  constexpr int kTile = 32 * kSparseImg;
  static_assert(kSparseImg == 4, "one uint4 of image bits per tile");
  __shared__ int4 stage[kSparseWarps][32];
  constexpr int KW = N * N / 4;
  constexpr int kGroup = KW * 128;  // bytes of a group of 32 images
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t L = tile0 + blockIdx.x;
  const int64_t band = L / tiles_q, qt = L - band * tiles_q;
  const int64_t h0 = band * band_h;
  const int64_t h1 = tiles_h - h0 < band_h ? tiles_h : h0 + band_h;
  const int64_t q = qt * kSparseWarps + warp;
  if (q >= Q || nflags[q] != 0 || nwide[q]) return;  // the whole warp leaves; no block barrier follows
  const int64_t tq = dtrue[q];
  const int thr = tq > 0x7fffffffll ? 0x7fffffff : (int)tq;
  const int ne = ecount[q];
  const int4 *e = ent + q * (int64_t)KW;
  const int4 zero = make_int4(0, 0, 0, 0);  // a zero entry adds nothing
  const int4 e0 = ne > 0 ? e[0] : zero, e1 = ne > 1 ? e[1] : zero;
  const int start = e0.w + e1.w - thr;
  unsigned long long pair_words = 0, lane_slots = 0;
  // words of the first two entries of the next tile's images; the haystack is padded to whole tiles
  const int8_t *at = hword + h0 * (int64_t)(kSparseImg * kGroup) + lane * 4;
  int n0[kSparseImg], n1[kSparseImg];
  auto fetch = [&]() {
    const int8_t *p0 = at + e0.z, *p1 = at + e1.z;
#pragma unroll
    for (int k = 0; k < kSparseImg; ++k) {
      n0[k] = *reinterpret_cast<const int *>(p0 + k * kGroup);
      n1[k] = *reinterpret_cast<const int *>(p1 + k * kGroup);
    }
  };
  fetch();
  uint4 nbits = narrow[h0];
#pragma unroll 2
  for (int64_t ht = h0; ht < h1; ++ht) {
    const uint4 bits = nbits;
    int b0[kSparseImg], b1[kSparseImg];
#pragma unroll
    for (int k = 0; k < kSparseImg; ++k) {
      b0[k] = n0[k];
      b1[k] = n1[k];
    }
    const int8_t *tile = at;
    if (ht + 1 < h1) {
      at += kSparseImg * kGroup;
      fetch();
      nbits = narrow[ht + 1];
    }
    // partial distance minus the needle's true distance (exit once > 0); per word m (a - b)^2 =
    // sum a^2 + sum (m b)^2 - 2 sum a b
    int acc[kSparseImg];
#pragma unroll
    for (int k = 0; k < kSparseImg; ++k) {
      const int m0 = b0[k] & e0.y, m1 = b1[k] & e1.y;
      acc[k] = __dp4a(m1, m1, __dp4a(m0, m0, start)) -
               2 * __dp4a(e1.x, b1[k], __dp4a(e0.x, b0[k], 0));
    }
    const bool some = min(min(acc[0], acc[1]), min(acc[2], acc[3])) <= 0;
    if (kCount) {
      const int n = ne < 2 ? ne : 2;
      pair_words += (unsigned long long)n * (((bits.x >> lane) & 1u) + ((bits.y >> lane) & 1u) +
                                             ((bits.z >> lane) & 1u) + ((bits.w >> lane) & 1u));
      lane_slots += (unsigned long long)n * kSparseImg;
    }
    if (__ballot_sync(0xffffffffu, some) == 0) continue;
    unsigned alive = 0;
#pragma unroll
    for (int k = 0; k < kSparseImg; ++k) {
      const unsigned w = k == 0 ? bits.x : (k == 1 ? bits.y : (k == 2 ? bits.z : bits.w));
      if (acc[k] <= 0) alive |= ((w >> lane) & 1u) << k;
    }
    const unsigned long long more =
        sparse_rest<N, kCount>(tile, e, ne, acc, alive, thr, (int)(ht * kTile) + lane, stage[warp],
                               rank + q, best + q, lane_slots);
    if (kCount) pair_words += more;
  }
  if (kCount) {  // lane_slots is the same in every lane of the warp
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) pair_words += __shfl_down_sync(0xffffffffu, pair_words, d);
    if (lane == 0 && pair_words) atomicAdd(counters, pair_words);
    if (lane == 0 && lane_slots) atomicAdd(counters + 3, 32ull * lane_slots);
  }
}

// Pairs with a wide side, exact int64 (launch-wide indices; haystack restricted to the needle's
// scene).  List mode:
//   pass 0: needles = wide needle list, haystack = the needle's whole scene.
//   pass 1: needles = all needles that are not wide, haystack = wide images of the same scene.
//   pass 2: needles = all needles, haystack = the whole scene (reference path).
// mode 0 runs passes 0 and 1 (in one launch), mode 2 pass 2.  kRows: rows_of_8(N), 40 registers and six
// blocks per SM (at 32 they spill); else eight.  The items' costs differ widely, so the first form's
// grid is twice what is resident: 1,000 x 2,000 images of noise of 32 x 32 17.9 ms with one and a third
// times as many blocks, 13.3 ms with just as many, 13.2 ms so; 300 x 3,000 of 64 x 64 39.3, 28.5,
// 27.5 ms; the images outside int8 of 16,384 x 262,144 sparse ones 122, 120, 111 us.
template <bool kRows>
__global__ void __launch_bounds__(kWideThreads, kRows ? 6 : 8) k_wide(
    const SearchScene *__restrict__ tab, const int *__restrict__ qscene,
    const int *__restrict__ hscene, int64_t Qtot, int64_t Hmax, int N, int mode,
    const int *__restrict__ nwide, const int *__restrict__ wide_n_list,
    const int *__restrict__ wide_n_count, const int *__restrict__ wide_h_list,
    const int *__restrict__ wide_h_count, const int64_t *__restrict__ dtrue,
    const int *__restrict__ nflags, int *__restrict__ rank, unsigned long long *__restrict__ best,
    int *__restrict__ top1_flag, unsigned long long *__restrict__ counters,
    const int *__restrict__ sub_list, const int *__restrict__ sub_count) {
  // sub_list (optional, pass 1): iterate entries sub_list[0 .. *sub_count) of the wide haystack
  // list only (the images of that list outside the int8 class)
  extern __shared__ int2 nz[];  // (flat position, needle delta) of non-zero needle deltas
  __shared__ int nnz_s;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t K = (int64_t)N * N;
  const int64_t chunks_all = (Hmax + kWideThreads - 1) / kWideThreads;
  const int64_t nh = mode == 0 ? (sub_list ? *sub_count : *wide_h_count) : 0;  // pass 1
  const int64_t chunks_list = (nh + kWideThreads - 1) / kWideThreads;
  const int64_t items0 = (mode == 0 ? *wide_n_count : Qtot) * chunks_all;
  const int64_t items = items0 + (mode == 0 ? Qtot * chunks_list : 0);
  for (int64_t it0 = blockIdx.x; it0 < items; it0 += gridDim.x) {
    const int pass = mode == 2 ? 2 : (it0 < items0 ? 0 : 1);
    const int64_t it = pass == 1 ? it0 - items0 : it0, chunks = pass == 1 ? chunks_list : chunks_all;
    const int64_t qi = it / chunks, ch = it - qi * chunks;
    const int64_t i = pass == 0 ? wide_n_list[qi] : qi;
    if (nflags[i] != 0 || (pass == 1 && nwide[i])) continue;  // uniform over the block
    const int si = scene_at(qscene, i);
    const SearchScene &sc = tab[si];
    if (pass != 1 && ch * kWideThreads >= sc.H) continue;     // uniform over the block
    const int64_t il = i - sc.qoff;
    const uint16_t *n = sc.needles + il * K;
    // compact the needle's non-zero deltas (any order: the sum is exact)
    __syncthreads();
    if (tid == 0) nnz_s = 0;
    __syncthreads();
    if constexpr (kRows) {  // 256 pixels per warp and pass
      const bool vec = aligned16(n);
      for (int base = (tid >> 5) * 256; base < K; base += kWideThreads * 8) {
        const int k0 = base + lane * 8;
        int d[8];
        deltas8(k0 < K ? load_pixels8(n, k0, vec) : make_uint4(0, 0, 0, 0), lane, N, d);
        int c = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) c += d[e] != 0;
        int at = c;  // entries of the lanes up to this one
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, at, m);
          if (lane >= m) at += y;
        }
        int wbase = 0;
        if (lane == 31) wbase = atomicAdd(&nnz_s, at);
        at += __shfl_sync(0xffffffffu, wbase, 31) - c;
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (d[e] != 0) nz[at++] = make_int2(k0 + e, d[e]);
      }
    }
    for (int64_t base = kRows ? K : 0; base < K; base += kWideThreads) {
      int k = (int)(base + tid);
      int a = 0;
      if (k < K) {
        int r = k / N, c = k - r * N;
        a = delta_at(n, N, r, c);
      }
      unsigned bal = __ballot_sync(0xffffffffu, a != 0);
      int wbase = 0;
      if (lane == 0) wbase = atomicAdd(&nnz_s, __popc(bal));
      wbase = __shfl_sync(0xffffffffu, wbase, 0);
      if (a != 0) nz[wbase + __popc(bal & ((1u << lane) - 1u))] = make_int2(k, a);
    }
    __syncthreads();
    const int nnz = nnz_s;
    const int64_t thr = dtrue[i];
    const int64_t hj = ch * kWideThreads + tid;
    int64_t jl = -1;  // scene-local haystack index
    if (pass == 1) {
      if (hj < nh) {
        const int64_t jg = wide_h_list[sub_list ? sub_list[hj] : hj];
        if (scene_at(hscene, jg) == si) jl = jg - sc.hoff;
      }
    } else if (hj < sc.H) {
      jl = hj;
    }
    int cnt = 0;
    unsigned long long b = kNoBest;
    unsigned long long npairs = 0, nterms = 0;
    if (jl >= 0) {
      const uint16_t *h = sc.haystack + jl * K;
      long long acc = 0;
      int e = 0;
      for (; e < nnz && acc <= thr; ++e) {
        int2 p = nz[e];
        long long d = (long long)p.y - ((long long)h[p.x] - (long long)h[p.x - 1]);
        acc += d * d;
      }
      npairs = 1;
      nterms = e;
      if (acc <= thr) {
        cnt = acc < thr;
        b = pack_best(acc, jl);
        if (acc >= 0xffffffffll) atomicOr(&top1_flag[i], 1);
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, d);
    b = warp_min_u64(b);
    if (counters) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        npairs += __shfl_down_sync(0xffffffffu, npairs, d);
        nterms += __shfl_down_sync(0xffffffffu, nterms, d);
      }
    }
    if (lane == 0) {
      if (cnt) atomicAdd(&rank[i], cnt);
      if (b != kNoBest) atomicMin(&best[i], b);
      if (counters && npairs) {
        atomicAdd(counters + 1, npairs);
        atomicAdd(counters + 2, nterms);
      }
    }
  }
}

// Per-needle choice of form (RICI_SEARCH_AUTO): a needle whose non-zero delta words are at most
// 1/kAutoSparseShare of its words goes to the sparse-needle form, every other int8-class needle
// to the fp16 tensor cores.  Writes the tensor-core skip flags (sparse_of), the exclusions of the
// dense middle pass (the sparse needles and those outside int8) and of the sparse kernel (the
// tensor-core needles and those outside int8).
constexpr int kAutoSparseShare = 4;

__global__ void k_auto_assign(const int *__restrict__ ecount, const int *__restrict__ n8wide,
                              int64_t Q, int KW, int *__restrict__ sparse_of,
                              int *__restrict__ excl_dense, int *__restrict__ excl_sparse) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Q;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int wide = n8wide[i];
    const int sp = !wide && (int64_t)ecount[i] * kAutoSparseShare <= KW;
    sparse_of[i] = sp;
    excl_dense[i] = wide || sp;
    excl_sparse[i] = wide || !sp;
  }
}

// skip_tile[m] = 1 when no needle of tensor-core needle tile m (128 needles) is ranked there;
// *any_tile (zeroed before) becomes 1 when some tile is left.
__global__ void k_auto_tiles(const int *__restrict__ excl_dense, int64_t Q, int64_t tiles_m,
                             int *__restrict__ skip_tile, int *__restrict__ any_tile) {
  const int lane = threadIdx.x & 31;
  for (int64_t m = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; m < tiles_m;
       m += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    int any = 0;
    for (int k = lane; k < 128; k += 32) {
      const int64_t i = m * 128 + k;
      any |= i < Q && !excl_dense[i];
    }
    any = __any_sync(0xffffffffu, any);
    if (lane == 0) {
      skip_tile[m] = !any;
      if (any) atomicOr(any_tile, 1);
    }
  }
}

// Scene-local outputs: rank, true distance and top-1 (smallest index among minimal distances).  The
// packed minimum holds distances below 2^32 - 1 exactly; where it is at that limit (top1_flag: some
// pair's distance reached it) the top-1 is the exact (distance, index) minimum over the scene instead.
// Each such needle takes a pass over its haystack by one block, so the needles are dealt out to all
// blocks of the grid one by one: 300 such needles x 3,000 images of 32 x 32 took 96.7 ms with 256
// consecutive needles to a block.  Four blocks of 16 warps per SM: 1.29 ms for 1,000 needles x 2,000, 1.71
// ms for 300 x 3,000 of 64 x 64, 4.6 us where there is no such needle (eight of 8 warps 1.16, 2.58 ms,
// 4.7 us; two of 32 1.10, 1.66 ms, 5.4 us).
constexpr int kFinalizeBlocks = 152 * 4, kFinalizeWarps = 16;
template <bool kRows>
__global__ void __launch_bounds__(kFinalizeWarps * 32, 4)
    k_finalize(const SearchScene *__restrict__ tab, const int *__restrict__ qscene, int64_t Qtot,
               int N, const int *__restrict__ rank, const int64_t *__restrict__ dtrue,
               const unsigned long long *__restrict__ best, const int *__restrict__ nflags,
               const int *__restrict__ top1_flag) {
  __shared__ int64_t exact_s[kFinalizeWarps * 32];
  __shared__ int nexact;
  __shared__ long long bd[kFinalizeWarps];
  __shared__ long long bj[kFinalizeWarps];
  const int64_t K = (int64_t)N * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // (loads side by side: a chain of them is this kernel's time)
  auto is_exact = [&](int64_t i, int flags, unsigned long long bv) -> bool {
    const int t1 = top1_flag[i];
    return (t1 != 0) & (flags == 0) & ((bv >> 32) == 0xffffffffull) & (bv != kNoBest);
  };
  // needles blockIdx.x + k gridDim.x, one per thread at a time (the first look at them before the
  // outputs below, whose latency covers it)
  auto mine = [&](int64_t k0) { return blockIdx.x + (k0 + threadIdx.x) * gridDim.x; };
  bool ex = mine(0) < Qtot && is_exact(mine(0), nflags[mine(0)], best[mine(0)]);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Qtot;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int flags = nflags[i], r = rank[i];
    const unsigned long long bv = best[i];
    const int64_t dt = dtrue[i];
    const bool e = is_exact(i, flags, bv);
    const SearchScene &sc = tab[scene_at(qscene, i)];
    const int64_t il = i - sc.qoff;
    sc.rank[il] = r;
    if (sc.dtrue) sc.dtrue[il] = dt;
    if (sc.top1 && !e)
      sc.top1[il] = (flags != 0 || bv == kNoBest) ? -1 : (int32_t)(uint32_t)(bv & 0xffffffffull);
  }
  for (int64_t k0 = 0; blockIdx.x + k0 * gridDim.x < Qtot; k0 += kFinalizeWarps * 32) {
    const int64_t i = mine(k0);
    if (k0) ex = i < Qtot && is_exact(i, nflags[i], best[i]);
    if (threadIdx.x == 0) nexact = 0;
    if (!__syncthreads_or(ex)) continue;  // (uniform over the block)
    if (ex) exact_s[atomicAdd(&nexact, 1)] = i;
    __syncthreads();
    for (int x = 0; x < nexact; ++x) {
      const int64_t ie = exact_s[x];
      const SearchScene &sc = tab[scene_at(qscene, ie)];
      if (!sc.top1) continue;  // (uniform over the block)
      const int64_t il = ie - sc.qoff;
      long long md = 0x7fffffffffffffffll, mj = -1;
      for (int64_t j = warp; j < sc.H; j += kFinalizeWarps) {
        long long d = warp_crss<kRows>(sc.needles + il * K, sc.haystack + j * K, N);
        if (d < md) {
          md = d;
          mj = j;
        }
      }
      if (lane == 0) {
        bd[warp] = md;
        bj[warp] = mj;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        long long d0 = bd[0], j0 = bj[0];
        for (int w = 1; w < kFinalizeWarps; ++w)
          if (bd[w] < d0 || (bd[w] == d0 && bj[w] < j0)) {
            d0 = bd[w];
            j0 = bj[w];
          }
        sc.top1[il] = (int32_t)j0;
      }
      __syncthreads();
    }
  }
}

// Full distance matrix (exact int64), one warp per pair.
template <bool kRows>
__global__ void k_distances(const uint16_t *__restrict__ nimg, int64_t Q,
                            const uint16_t *__restrict__ himg, int64_t H, int N,
                            int64_t *__restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t K = (int64_t)N * N;
  for (int64_t p = w; p < Q * H; p += nw) {
    const int64_t i = p / H, j = p - i * H;
    int64_t d = warp_crss<kRows>(nimg + i * K, himg + j * K, N);
    if (lane == 0) out[p] = d;
  }
}

// Distances of one needle to kMany images, one warp: the needle's deltas once for all, sums in 32 bits
// (all images 16-byte aligned with rows_of_8(N)).  Returns false where a sum could pass 2^31: K
// (largest difference)^2 bounds it.
constexpr int kMany = 4;
__device__ __forceinline__ bool warp_crss_many(const uint16_t *n, const uint16_t *const (&h)[kMany],
                                               int N, int64_t (&out)[kMany]) {
  const int lane = threadIdx.x & 31, K = N * N;
  unsigned s[kMany] = {}, bits = 0;
  for (int base = 0; base < K; base += 256) {
    const int k0 = base + lane * 8;
    const bool in = k0 < K;
    uint4 px[kMany];
#pragma unroll
    for (int m = 0; m < kMany; ++m)
      px[m] = in ? load_pixels8(h[m], k0, true) : make_uint4(0, 0, 0, 0);
    int a[8];
    deltas8(in ? load_pixels8(n, k0, true) : make_uint4(0, 0, 0, 0), lane, N, a);
#pragma unroll
    for (int m = 0; m < kMany; ++m) {
      int b[8];
      deltas8(px[m], lane, N, b);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const unsigned x = a[e] != 0 ? (unsigned)abs(a[e] - b[e]) : 0u;
        s[m] += x * x;
        bits |= x;
      }
    }
  }
  bits = __reduce_or_sync(0xffffffffu, bits);
#pragma unroll
  for (int m = 0; m < kMany; ++m) out[m] = (int64_t)__reduce_add_sync(0xffffffffu, s[m]);
  return (unsigned long long)bits * bits * (unsigned)K < (1ull << 31);
}

// A whole small search of one scene in one launch: block i ranks needle i, one warp per pair, every
// distance exact in int64 (so no classes, lists or fallbacks).
constexpr int kSmallWarps = 16;
template <bool kRows>
__global__ void __launch_bounds__(kSmallWarps * 32) k_search_small(SearchScene sc, int N,
                                                                   int64_t *__restrict__ distances,
                                                                   int *status) {
  __shared__ int64_t dt_s;
  __shared__ int cnt_s[kSmallWarps];
  __shared__ int64_t bd_s[kSmallWarps], bj_s[kSmallWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t K = (int64_t)N * N, i = blockIdx.x;
  const uint16_t *needle = sc.needles + i * K;
  const int64_t m = sc.match ? sc.match[i] : i;
  const bool valid = m >= 0 && m < sc.H;
  if (warp == 0) {
    const int64_t d = valid ? warp_crss<kRows>(needle, sc.haystack + m * K, N) : -1;
    if (lane == 0) {
      dt_s = d;
      if (!valid) set_status(status, RICI_ERR_INDEX_OUT_OF_RANGE);
    }
  }
  __syncthreads();
  const int64_t dt = dt_s;
  int cnt = 0;
  int64_t bd = INT64_MAX, bj = -1;
  if (valid || distances) {
    for (int64_t j0 = warp; j0 < sc.H; j0 += kMany * kSmallWarps) {
      int64_t d[kMany];
      const uint16_t *h[kMany];
#pragma unroll
      for (int m = 0; m < kMany; ++m) {  // (past the end: the last image again)
        const int64_t j = j0 + m * kSmallWarps;
        h[m] = sc.haystack + (j < sc.H ? j : sc.H - 1) * K;
      }
      if (!kRows || !warp_crss_many(needle, h, N, d)) {
#pragma unroll 1
        for (int m = 0; m < kMany; ++m) {
          const int64_t j = j0 + m * kSmallWarps;
          const int64_t x = warp_crss<kRows>(needle, sc.haystack + (j < sc.H ? j : sc.H - 1) * K, N);
#pragma unroll
          for (int o = 0; o < kMany; ++o)
            if (o == m) d[o] = x;
        }
      }
#pragma unroll
      for (int m = 0; m < kMany; ++m) {
        const int64_t j = j0 + m * kSmallWarps;
        if (j >= sc.H) continue;
        cnt += d[m] < dt;
        if (d[m] < bd) {  // j ascends: the smallest index of a minimum stays
          bd = d[m];
          bj = j;
        }
        if (distances && lane == 0) distances[i * sc.H + j] = d[m];
      }
    }
  }
  if (lane == 0) {
    cnt_s[warp] = cnt;
    bd_s[warp] = bd;
    bj_s[warp] = bj;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kSmallWarps; ++w) {
      cnt += cnt_s[w];
      if (bj_s[w] >= 0 && (bd_s[w] < bd || (bd_s[w] == bd && bj_s[w] < bj))) {
        bd = bd_s[w];
        bj = bj_s[w];
      }
    }
    sc.rank[i] = valid ? cnt : -1;
    if (sc.dtrue) sc.dtrue[i] = dt;
    if (sc.top1) sc.top1[i] = valid ? (int32_t)bj : -1;
  }
}

// Whether a call takes k_search_small: the forms that leave the choice to the library (DEFAULT, AUTO),
// no work counters, and so little work that launches decide.  The haystack is limited (256 images of
// up to 32 x 32, 64 of 64 x 64, 16 of 128 x 128), and with it the work in all: past that the general
// sequence wins (64 x 512 images of 32 x 32 80 against 93 us, 512 x 512 95 against 190 us).  Within:
//   8 pixels per lane (rows): on top of what both sides pay, the blocks (one per needle) take about 5 ns
//     each, and 0.35 ns per 256 pixels of a pair, where a warp takes four pairs at a time, there or not;
//     the general sequence's further launches take 25 us and 4.5 us per 256 pixels.  162 x 162 images
//     of 32 x 32 114 us in 19 launches, 23 us here; 4,000 x 4 75 and 54 us, 4,000 x 16 75 and 126 us;
//     16,000 x 1 of 8 x 8 61 and 109 us; 600 x 16 of 64 x 64 109 and 64 us, 1,000 x 16 108 and 111 us.
//   1 pixel per lane (other resolutions, unaligned images): `serial` steps one after another in a warp,
//     0.3 us each, so it wins up to 72 of them (1 x 64 images of 20 x 20 32 and 27 us, 1 x 32 of 33 x 33 50
//     and 54 us, 64 x 240 52 and 186 us) while the needles' blocks are resident together (300 x 4 of
//     33 x 33 52 and 47 us, 1,000 x 1 of 24 x 24 35 and 60 us).  Unaligned images that the general
//     sequence would take on tensor cores up to 256 steps (64 x 64 of 32 x 32 78 and 60 us, 64 x 256
//     89 and 179 us; 1 x 16 of 64 x 64 156 and 148 us).
bool small_search(const SearchBatch &b, bool rows) {
  const int64_t Q = b.Qtot, H = b.Htot, K = (int64_t)b.N * b.N, K1 = K < 1024 ? 1024 : K;
  if (!((b.mode == RICI_SEARCH_DEFAULT || b.mode == RICI_SEARCH_AUTO) && b.num_scenes == 1 &&
        !b.counters && H * K1 <= (1 << 18) && Q * H * K1 <= (1 << 26)))
    return false;
  if (rows) {
    const int64_t passes = (K + 255) / 256;
    const int64_t work = Q * (H < 16 ? H : 16) * ((H + 63) / 64) * passes;
    return 7 * work + 100 * Q <= 500000 + 90000 * passes;
  }
  const int64_t serial = (K + 31) / 32 * (1 + (H + 15) / 16);
  return rows_of_8(b.N) ? serial <= 256 && Q * (serial + 16) <= (1 << 16)
                        : serial <= 72 && Q * (serial + 16) <= (1 << 15);
}

bool dense_supported(int N) { return N == 8 || N == 16 || N == 32 || N == 64 || N == 128; }

template <int N>
cudaError_t launch_dense(const int8_t *nd, const int8_t *nm, const int *nrs, const int *nw, int64_t Q,
                         const int8_t *hd, const int *hw, int64_t H, const int64_t *dt,
                         const int *nf, int *rank, unsigned long long *best,
                         unsigned long long *counters, cudaStream_t st,
                         const int *hcount = nullptr, const int *hmap = nullptr,
                         const int *gate = nullptr) {
  // 4 needles x 4 haystack images per thread (N <= 64; 120 registers, two blocks of 256 threads
  // per SM) is the fastest measured shape: each broadcast needle word serves four images, and
  // the per-row bookkeeping is shared by 16 (needle, image) pairs
  constexpr int kTQ = N <= 64 ? 4 : 2;  // N = 128: 64 KB of needle tile, two blocks per SM
  constexpr int kImg = N <= 64 ? 4 : 1;
  const size_t smem = sizeof(int2) * kTQ * (N * N / 4);
  auto kern = hcount ? (counters ? k_dense<N, kTQ, kImg, true, true>
                                 : k_dense<N, kTQ, kImg, false, true>)
                     : (counters ? k_dense<N, kTQ, kImg, true, false>
                                 : k_dense<N, kTQ, kImg, false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t th = (H + kDenseThreads * kImg - 1) / (kDenseThreads * kImg);
  const int64_t tq = (Q + kTQ - 1) / kTQ;
  // bands as long as possible while the grid still gives every SM a few waves of blocks
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t band_h = th * tq / ((int64_t)sms * 2 * 4);
  band_h = band_h < 1 ? 1 : (band_h > kBandMax ? kBandMax : band_h);
  const int64_t total = (th + band_h - 1) / band_h * tq;
  const int64_t kMaxGrid = hcount ? (int64_t)sms * 32 : 0x7fffffffll;
  for (int64_t t0 = 0; t0 < total; t0 += hcount ? total : kMaxGrid) {
    const int64_t n = total - t0 < kMaxGrid ? total - t0 : kMaxGrid;
    kern<<<(unsigned)n, kDenseThreads, smem, st>>>(nd, nm, nrs, nw, Q, hd, hw, H, dt, nf, rank,
                                                   best, counters, t0, tq, th, band_h, total, hcount,
                                                   hmap, gate);
    count_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_sparse(const int4 *ent, const int *ecount, const int *nw, int64_t Q,
                          const int8_t *hd, const uint32_t *narrow, int64_t H, int N,
                          const int64_t *dt, const int *nf, int *rank, unsigned long long *best,
                          unsigned long long *counters, cudaStream_t st) {
  auto pick = [&](auto n) {
    return counters ? k_sparse<decltype(n)::value, true> : k_sparse<decltype(n)::value, false>;
  };
  auto kern = N == 8    ? pick(std::integral_constant<int, 8>())
              : N == 16 ? pick(std::integral_constant<int, 16>())
              : N == 32 ? pick(std::integral_constant<int, 32>())
              : N == 64 ? pick(std::integral_constant<int, 64>())
                        : pick(std::integral_constant<int, 128>());
  const int64_t th = (H + 32 * kSparseImg - 1) / (32 * kSparseImg);
  const int64_t tq = (Q + kSparseWarps - 1) / kSparseWarps;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // bands as long as possible while the grid still gives every SM several waves of blocks
  int64_t band_h = th * tq / ((int64_t)sms * 8 * 4);
  band_h = band_h < 1 ? 1 : (band_h > kSparseBandMax ? kSparseBandMax : band_h);
  const int64_t total = (th + band_h - 1) / band_h * tq;
  constexpr int64_t kMaxGrid = 0x7fffffffll;
  for (int64_t t0 = 0; t0 < total; t0 += kMaxGrid) {
    const int64_t n = total - t0 < kMaxGrid ? total - t0 : kMaxGrid;
    kern<<<(unsigned)n, kSparseWarps * 32, 0, st>>>(ent, ecount, nw, Q, hd,
                                                    reinterpret_cast<const uint4 *>(narrow), H, dt,
                                                    nf, rank,
                                                    best, counters, t0, tq, th, band_h);
    count_launches(1);
  }
  return cudaGetLastError();
}

}  // namespace

void search_tiles(int64_t Q, int64_t H, int32_t *tiles_m, int32_t *tiles_n) {
  *tiles_m = (int32_t)((Q + 127) / 128);
  *tiles_n = (int32_t)((H + 255) / 256);
}

// Bytes of the haystack's int8 deltas (groups of 32 images).  In a tensor-core search the rows of its
// split-square images lie there before: their GEMM is done when the images of neither class are
// encoded, and from 6,144 images on they take no more room.
static int64_t haystack_delta_bytes(int64_t H, int N, bool split_rows) {
  const int64_t deltas = (H + 127) / 128 * 128 * N * N;
  const int64_t rows = split_rows ? tc_split_bytes(H, N) : 0;
  return deltas > rows ? deltas : rows;
}

int64_t search_batch_workspace_bytes(int num_scenes, int64_t Q, int64_t H, int N, int mode) {
  const int64_t K = (int64_t)N * N;
  mode &= 0xff;
  const bool autom = mode == RICI_SEARCH_AUTO && num_scenes == 1 && tc_supported(N) &&
                     dense_supported(N);
  const bool tensor = (mode == RICI_SEARCH_TENSOR || mode == RICI_SEARCH_DEFAULT ||
                       mode == RICI_SEARCH_AUTO) && tc_supported(N);
  const bool i8 = mode == RICI_SEARCH_INT8_TC && i8_supported(N);
  const bool packed = !tensor && !i8 && mode != RICI_SEARCH_EXACT_SLOW && dense_supported(N);
  const bool sparse = packed && mode == RICI_SEARCH_SPARSE;
  const bool mid = tensor && num_scenes == 1 && dense_supported(N);
  Carver c(nullptr);
  c.take<SearchScene>(num_scenes);
  c.take<int>(num_scenes == 1 ? 0 : Q);  // scene of each needle
  c.take<int>(num_scenes == 1 ? 0 : H);  // scene of each haystack image
  c.take<int8_t>(packed || mid ? Q * K : 0);  // needle deltas (CUDA-core forms)
  c.take<int8_t>(packed || mid ? Q * K : 0);  // needle masks
  c.take<int>((packed && !sparse) || mid ? Q * N : 0);  // needle row sums of squared deltas
  c.take<int8_t>(packed || mid ? haystack_delta_bytes(H, N, mid) : 0);  // haystack deltas
  c.take<int>(Q);                        // needle wide flags
  c.take<int>(H + 4);                    // haystack wide flags (or, sparse form, a bit per image)
  c.take<int>(Q);                        // wide needle list
  c.take<int>(H);                        // wide haystack list
  c.take<int>(kCounts);                  // list lengths
  c.take<int>(Q);                        // per-needle state flags
  c.take<int>(Q);                        // top-1 exact fallback flags
  c.take<unsigned long long>(Q);         // packed best (distance, index)
  c.take<int64_t>(Q);                    // true distances
  c.take<int>(Q);                        // ranks
  c.take<int4>(sparse || autom ? Q * (K / 4) : 0);  // sparse needle entries (a slab per needle)
  c.take<int>(sparse || autom ? Q : 0);  // sparse entries per needle
  c.take<char>(tensor ? tc_workspace_bytes(Q, H, N, num_scenes == 1) : 0);
  c.take<char>(i8 ? i8_workspace_bytes(Q, H, N) : 0);
  c.take<int>(mid ? Q : 0);      // int8 class flags of the needles (dense middle pass)
  c.take<int>(mid ? H : 0);      // int8 class flags of the compacted haystack images
  c.take<int>(mid ? Q + H : 0);  // lists written by its encodes
  c.take<int>(mid ? H : 0);      // images of neither tensor-core class
  c.take<int8_t>(autom ? (H + 127) / 128 * 128 * K : 0);  // word-major haystack of the sparse form
  c.take<uint32_t>(autom ? (H + 127) / 128 * 4 : 0);  // its int8 class, a bit per image
  c.take<int>(autom ? H : 0);      // the images outside it
  c.take<int>(autom ? 3 * Q : 0);  // per-needle choice and the two exclusions
  c.take<int>(autom ? Q / 128 + 2 : 0);  // tensor-core needle tiles to skip
  return c.off + 256;
}

int64_t search_workspace_bytes(int64_t Q, int64_t H, int32_t N, int32_t mode) {
  return search_batch_workspace_bytes(1, Q, H, N, mode);
}

cudaError_t launch_search_batch(const SearchScene *scenes, const SearchBatch &b, void *ws,
                                cudaStream_t st, int64_t *out_distances) {
  const int64_t Q = b.Qtot, H = b.Htot;
  const int N = b.N;
  const int64_t K = (int64_t)N * N;
  if (Q == 0) return cudaSuccess;
  // rows: images that a warp reads 8 pixels at a time; pairs: and that fill its 256 pixels (8 x 8 ones
  // leave three lanes of four idle: 1,000 x 20,000 distances 4.38 ms so, 4.06 ms 32 pixels at a time)
  bool rows = rows_of_8(N);
  for (int i = 0; i < b.num_scenes; ++i)
    rows = rows && aligned16(scenes[i].needles) && aligned16(scenes[i].haystack);
  const bool pairs = rows && K >= 256;
  if (small_search(b, rows)) {
    const auto small_kernel = rows ? k_search_small<true> : k_search_small<false>;
    small_kernel<<<(unsigned)Q, kSmallWarps * 32, 0, st>>>(scenes[0], N, out_distances, b.status);
    count_launches(1);
    return cudaGetLastError();
  }
  const int withhold = (b.mode & RICI_SEARCH_TEST_WITHHOLD_LOAD) ? 1 : 0;
  const int mode = b.mode & 0xff;
  // RICI_SEARCH_AUTO (single scene): each needle ranked by the fp16 tensor cores or by the
  // sparse-needle form, chosen from its share of non-zero delta words (k_auto_assign)
  const bool autom = mode == RICI_SEARCH_AUTO && b.num_scenes == 1 && tc_supported(N) &&
                     dense_supported(N);
  const bool tensor = (mode == RICI_SEARCH_TENSOR || mode == RICI_SEARCH_DEFAULT ||
                       mode == RICI_SEARCH_AUTO) && tc_supported(N);
  const bool i8 = mode == RICI_SEARCH_INT8_TC && i8_supported(N);
  const bool packed = !tensor && !i8 && mode != RICI_SEARCH_EXACT_SLOW && dense_supported(N) &&
                      b.num_scenes == 1;
  const bool sparse = packed && mode == RICI_SEARCH_SPARSE;
  const bool dense = packed && !sparse;
  // single-scene tensor-core calls: pairs of a narrow needle with a haystack image outside both
  // tensor-core classes but inside int8 run on the dense CUDA-core kernel over a compacted haystack
  // instead of the int64 kernel
  const bool mid = tensor && b.num_scenes == 1 && dense_supported(N);
  Carver c(ws);
  SearchScene *tab = c.take<SearchScene>(b.num_scenes);
  const bool single = b.num_scenes == 1;  // every image is of scene 0: no index arrays
  int *qscene = single ? nullptr : c.take<int>(Q);
  int *hscene = single ? nullptr : c.take<int>(H);
  int8_t *nd = c.take<int8_t>(packed || mid ? Q * K : 0);
  int8_t *nm = c.take<int8_t>(packed || mid ? Q * K : 0);
  int *nrs = c.take<int>(dense || mid ? Q * N : 0);
  int8_t *hd = c.take<int8_t>(packed || mid ? haystack_delta_bytes(H, N, mid) : 0);
  int *nwide = c.take<int>(Q);
  int *hwide = c.take<int>(H + 4);
  int *wn_list = c.take<int>(Q);
  int *wh_list = c.take<int>(H);
  int *counts = c.take<int>(kCounts);
  int *nflags = c.take<int>(Q);
  int *t1flag = c.take<int>(Q);
  unsigned long long *best = c.take<unsigned long long>(Q);
  int64_t *dt = c.take<int64_t>(Q);
  int *rank = c.take<int>(Q);
  int4 *sent = c.take<int4>(sparse || autom ? Q * (K / 4) : 0);
  int *scount = c.take<int>(sparse || autom ? Q : 0);
  char *tc_ws = tensor ? c.take<char>(tc_workspace_bytes(Q, H, N, b.num_scenes == 1)) : nullptr;
  char *i8_ws = i8 ? c.take<char>(i8_workspace_bytes(Q, H, N)) : nullptr;
  int *mid_nflag = c.take<int>(mid ? Q : 0);
  int *mid_hflag = c.take<int>(mid ? H : 0);
  int *mid_list = c.take<int>(mid ? Q + H : 0);
  // the images of neither tensor-core class; in small searches of images below 32 x 32 all outside
  // the fp16 class: the second GEMM's two launches cost more than the CUDA cores take for them there.
  // With it against without, 8 x 8: 600 x 20,000 84 against 77 us, 2,000 x 60,000 182 against 196,
  // 8,000 x 200,000 614 against 683; 16 x 16: 83 against 75, 193 against 184, 652 against 645
  const bool split = mid && (N >= 32 || Q * H >= (1ll << 26));
  int *left_list = c.take<int>(mid ? H : 0);
  if (!split) left_list = wh_list;
  int *const left_count = counts + (split ? 6 : 1);
  int8_t *hword = c.take<int8_t>(autom ? (H + 127) / 128 * 128 * K : 0);
  uint32_t *auto_narrow = c.take<uint32_t>(autom ? (H + 127) / 128 * 4 : 0);
  int *auto_list = c.take<int>(autom ? H : 0);
  int *auto_n = c.take<int>(autom ? 3 * Q : 0);
  int *skip_tile = c.take<int>(autom ? Q / 128 + 2 : 0);
  int *sparse_of = autom ? auto_n : nullptr;
  int *excl_dense = autom ? auto_n + Q : nullptr;
  int *excl_sparse = autom ? auto_n + 2 * Q : nullptr;

  cudaError_t e;
  for (int s0 = 0; s0 < b.num_scenes; s0 += kFillChunk) {
    SearchFill f;
    f.n = b.num_scenes - s0 < kFillChunk ? b.num_scenes - s0 : kFillChunk;
    for (int i = 0; i < f.n; ++i) f.e[i] = scenes[s0 + i];
    k_fill_search_table<<<1, 256, 0, st>>>(tab + s0, f, counts, kCounts);
    count_launches(1);
  }
  const int wpb = 8;
  auto blocks_for = [&](int64_t items) {
    int64_t nb = (items + wpb - 1) / wpb;
    return (int)(nb < 152 * 64 ? (nb > 0 ? nb : 1) : 152 * 64);
  };
  if (!single) {
    k_scene_index<<<blocks_for((Q > H ? Q : H) / 32 + 1), 256, 0, st>>>(tab, b.num_scenes, Q, H,
                                                                        qscene, hscene);
    count_launches(1);
  }
  const auto true_kernel = pairs ? k_true_distance<true> : k_true_distance<false>;
  true_kernel<<<blocks_for(Q), 32 * wpb, 0, st>>>(tab, qscene, Q, N, dt, rank, best, nflags, t1flag,
                                                  b.status);
  count_launches(1);
  unsigned long long *cnt = reinterpret_cast<unsigned long long *>(b.counters);
  const size_t wide_smem = sizeof(int2) * (size_t)K;
  const auto wide_kernel = rows_of_8(N) ? k_wide<true> : k_wide<false>;
  const int wide_blocks = 152 * (rows_of_8(N) ? 12 : 8);
  if ((e = cudaFuncSetAttribute(wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)wide_smem)) != cudaSuccess)
    return e;
  // int64 pairs: needles outside the class against everything and the others against the images
  // outside it (mode 0), or every pair (mode 2)
  auto wide = [&](int mode, const int *sub_list = nullptr, const int *sub_count = nullptr,
                  const int *list = nullptr, const int *list_count = nullptr) {
    wide_kernel<<<wide_blocks, kWideThreads, wide_smem, st>>>(
        tab, qscene, hscene, Q, b.Hmax, N, mode, nwide, wn_list, counts + 0, list ? list : wh_list,
        list_count ? list_count : counts + 1, dt, nflags, rank, best, t1flag, cnt, sub_list,
        sub_count);
    count_launches(1);
  };
  auto run_dense = [&](const int *nexcl, const int *hexcl, const int *hcount, const int *hmap,
                       const int *gate = nullptr) {
    switch (N) {
      case 8: return launch_dense<8>(nd, nm, nrs, nexcl, Q, hd, hexcl, H, dt, nflags, rank, best, cnt, st, hcount, hmap, gate);
      case 16: return launch_dense<16>(nd, nm, nrs, nexcl, Q, hd, hexcl, H, dt, nflags, rank, best, cnt, st, hcount, hmap, gate);
      case 32: return launch_dense<32>(nd, nm, nrs, nexcl, Q, hd, hexcl, H, dt, nflags, rank, best, cnt, st, hcount, hmap, gate);
      case 64: return launch_dense<64>(nd, nm, nrs, nexcl, Q, hd, hexcl, H, dt, nflags, rank, best, cnt, st, hcount, hmap, gate);
      default: return launch_dense<128>(nd, nm, nrs, nexcl, Q, hd, hexcl, H, dt, nflags, rank, best, cnt, st, hcount, hmap, gate);
    }
  };
  // the haystack of a single scene (or its images list[0 .. *count)) for k_dense, for k_sparse
  const int group_blocks = (int)((H + 31) / 32 < 152 * 32 ? (H + 31) / 32 : 152 * 32);
  auto encode_rows = [&](int8_t *out, int *flag, int *wlist, int *wcount, const int *list,
                         const int *count) {
    auto kern = N == 8 ? k_encode_groups<2> : k_encode_groups<4>;
    kern<<<group_blocks, kGroupWarps * 32, 0, st>>>(scenes[0].haystack, H, N, out, flag, wlist,
                                                    wcount, list, count, nullptr);
    count_launches(1);
  };
  auto encode_words = [&](int8_t *out, uint32_t *narrow, int *wlist, int *wcount) {
    k_encode_groups<1><<<group_blocks, kGroupWarps * 32, 0, st>>>(scenes[0].haystack, H, N, out,
                                                                  nullptr, wlist, wcount, nullptr,
                                                                  nullptr, narrow);
    count_launches(1);
  };
  if (tensor) {
    const SearchScene &s0 = scenes[0];
    if (mid) {
      // CUDA-core encode of every needle (the fp16-class ones are int8-class too)
      k_encode_needles<<<blocks_for(Q), 32 * wpb, 0, st>>>(s0.needles, Q, N, nd, nm, mid_nflag,
                                                           mid_list, counts + 2, nrs);
      count_launches(1);
    }
    if (autom) {
      // the haystack of the sparse-needle form; its list of the images outside int8 also serves the
      // int64 pass below, so the tensor-core class encode has nothing to do when no needle is left
      // for it
      encode_words(hword, auto_narrow, auto_list, counts + 4);
      // each needle's form, decided before the tensor-core kernel runs
      k_sparse_needles<<<blocks_for(Q), 32 * wpb, 0, st>>>(nd, nm, Q, N, sent, scount);
      k_auto_assign<<<blocks_for(Q / 32 + 1), 256, 0, st>>>(scount, mid_nflag, Q, (int)(K / 4),
                                                            sparse_of, excl_dense, excl_sparse);
      k_auto_tiles<<<blocks_for(Q / 128 + 1), 256, 0, st>>>(excl_dense, Q, (Q + 127) / 128,
                                                            skip_tile, counts + 5);
      count_launches(3);
    }
    if ((e = launch_tc_encode_and_rank(tab, b.num_scenes, qscene, hscene, Q, H, b.tiles_total, N,
                                       tc_ws, nwide, hwide, wn_list, wh_list, counts, nflags, dt,
                                       rank, best, b.status, withhold, st, sparse_of,
                                       autom ? skip_tile : nullptr, counts + 5,
                                       mid ? s0.haystack : nullptr, split, left_list, left_count,
                                       hd)) != cudaSuccess)
      return e;
    if (mid) {
      // the haystack images of neither tensor-core class, compacted in list order (list and
      // count from the tensor-core encodes); narrow needles x those images on CUDA cores, and the
      // int64 kernel only for the compacted images outside the int8 class
      encode_rows(hd, mid_hflag, mid_list + Q, counts + 3, left_list, left_count);
      // (AUTO: counts[5] = 0 when no needle is left for the tensor-core side)
      if ((e = run_dense(autom ? excl_dense : nwide, mid_hflag, left_count, left_list,
                         autom ? counts + 5 : nullptr)) != cudaSuccess)
        return e;
      // needles outside the class, and images outside the int8 class: AUTO's word encode has listed
      // these, the compacted encode (as compact indices) those of its images
      if (autom) wide(0, nullptr, nullptr, auto_list, counts + 4);
      else wide(0, mid_list + Q, counts + 3, left_list);
    } else {
      wide(0);
    }
    if (autom) {
      // the sparse-needle form for its needles against every int8-class image
      if ((e = launch_sparse(sent, scount, excl_sparse, Q, hword, auto_narrow, H, N, dt, nflags,
                             rank, best, cnt, st)) != cudaSuccess)
        return e;
    }
  } else if (i8) {
    if ((e = launch_i8_encode_and_rank(tab, b.num_scenes, qscene, hscene, Q, H, b.tiles_total, N,
                                       i8_ws, nwide, hwide, wn_list, wh_list, counts, nflags, dt,
                                       rank, best, st)) != cudaSuccess)
      return e;
    wide(0);
  } else if (dense) {
    // single scene: launch-wide indices are the scene's own
    const SearchScene &s0 = scenes[0];
    k_encode_needles<<<blocks_for(Q), 32 * wpb, 0, st>>>(s0.needles, Q, N, nd, nm, nwide, wn_list,
                                                         counts + 0, nrs);
    count_launches(1);
    encode_rows(hd, hwide, wh_list, counts + 1, nullptr, nullptr);
    if ((e = run_dense(nwide, hwide, nullptr, nullptr)) != cudaSuccess) return e;
    wide(0);
  } else if (sparse) {
    const SearchScene &s0 = scenes[0];
    k_encode_needles<<<blocks_for(Q), 32 * wpb, 0, st>>>(s0.needles, Q, N, nd, nm, nwide, wn_list,
                                                         counts + 0, nullptr);
    uint32_t *const narrow = reinterpret_cast<uint32_t *>(hwide);
    encode_words(hd, narrow, wh_list, counts + 1);
    k_sparse_needles<<<blocks_for(Q), 32 * wpb, 0, st>>>(nd, nm, Q, N, sent, scount);
    count_launches(2);
    if ((e = launch_sparse(sent, scount, nwide, Q, hd, narrow, H, N, dt, nflags, rank, best, cnt,
                           st)) != cudaSuccess)
      return e;
    wide(0);
  } else {
    if ((e = cudaMemsetAsync(nwide, 0, sizeof(int) * Q, st)) != cudaSuccess) return e;
    wide(2);
  }
  const auto finalize_kernel = pairs ? k_finalize<true> : k_finalize<false>;
  finalize_kernel<<<(unsigned)(Q < kFinalizeBlocks ? Q : kFinalizeBlocks), kFinalizeWarps * 32, 0,
                    st>>>(tab, qscene, Q, N, rank, dt, best, nflags, t1flag);
  count_launches(1);
  if (out_distances && b.num_scenes == 1) {
    const auto distances_kernel = pairs ? k_distances<true> : k_distances<false>;
    distances_kernel<<<blocks_for(Q * H), 32 * wpb, 0, st>>>(scenes[0].needles, Q,
                                                             scenes[0].haystack, H, N,
                                                             out_distances);
    count_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_search(const SearchArgs &a, void *ws, cudaStream_t st) {
  SearchScene sc = {};
  sc.needles = a.needles;
  sc.haystack = a.haystack;
  sc.match = a.true_match;
  sc.rank = a.out_rank;
  sc.dtrue = a.out_true_distance;
  sc.top1 = a.out_top1;
  sc.Q = a.num_needles;
  sc.H = a.num_haystack;
  search_tiles(sc.Q, sc.H, &sc.tiles_m, &sc.tiles_n);
  SearchBatch b;
  b.num_scenes = 1;
  b.Qtot = sc.Q;
  b.Htot = sc.H;
  b.Hmax = sc.H;
  b.tiles_total = (int64_t)sc.tiles_m * sc.tiles_n;
  b.N = a.resolution;
  b.mode = a.mode;
  b.counters = a.counters;
  b.status = a.status;
  return launch_search_batch(&sc, b, ws, st, a.out_distances);
}

}  // namespace rici
