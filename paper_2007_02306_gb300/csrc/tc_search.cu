// Exact clutter-resistant search on the tcgen05 tensor cores (sm_103a).
//
// Listing 1's distance splits into a needle constant and two cross terms:
//   d(i,j) = sum_k m_ik (a_ik - b_jk)^2 = A_i + S_ij,
//   A_i = sum_k a_ik^2,   S_ij = sum_k m_ik b_jk^2 - 2 a_ik b_jk,
// with a, b the column deltas (delta of column 0 := 0) and m_ik = [a_ik != 0] (m a = a).
// S is one GEMM with K = 2 N^2:  needle row [m_i | a_i]  x  haystack row [b_j^2 | -2 b_j].
//
// Exactness (the fp16 class): a needle is in the class when every |a| <= 127, a haystack image
// when every |b| <= 45 and S2_j + 254 S1_j < 2^24, with S2_j = sum_k b_jk^2 and
// S1_j = sum_k |b_jk|.  Every operand is then an integer exactly representable in fp16 (m, a;
// b^2 <= 2025 < 2^11, |2b| <= 90), every product is an exact integer, and every partial sum of
// any subset of the products m_ik b_jk^2 - 2 a_ik b_jk is an integer of magnitude at most
// S2_j + 2 * 127 * S1_j < 2^24, so the FP32 accumulation in TMEM is exact in any order.  Pairs
// with a side outside the class go to the CUDA-core kernels (dense int8 or exact int64).  The rank
// test S_ij < d(i,match_i) - A_i, and the top-1 key (A_i + S_ij, j), are evaluated in the GEMM
// epilogue; S is never written to memory.
//
// Split-square class (single-scene calls): haystack images with some 45 < |b| <= 127 and the same
// bound S2_j + 254 S1_j < 2^24.  b^2 = 128 q + r with r < 128, q <= 126, and 128 q is exact in fp16
// (7 significant bits), so S = [m | a | m] x [r | -2b | 128 q]^T with K = 3 N^2 has the same exact
// partial sums; the third block of the needle row is its first one again, so only the haystack rows
// are new.  On the 5M-triangle scene 7 % of the images are in this class: 1.5 times a fp16-class
// pair's work on the tensor cores, against CUDA cores at a ninth of that rate (8,192 needles x
// 262,144 of its images: 35.7 ms with those pairs on k_dense, 24.5 ms here).
//
// Kernel structure of k_tc_rank (one CTA per SM, persistent over 128 x 256 output tiles):
//   warp 0: TMA producer (128B-swizzled K-major tiles, 4-stage mbarrier pipeline)
//   warp 1: TMEM allocator and single-thread tcgen05.mma issuer (M=128, N=256, K=16)
//   warps 2-5: epilogue; tcgen05.ld of the accumulator (double-buffered: 2 x 256 columns)
// Every wait on an mbarrier gives up after 2 s of %globaltimer, sets RICI_ERR_TIMEOUT and lets
// the CTA reach its teardown (TMEM is always freed).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace rici {
namespace {

constexpr int kBM = 128;          // needles per tile (TMEM lanes)
constexpr int kBN = 256;          // haystack images per tile (TMEM columns per buffer)
constexpr int kBK = 64;           // fp16 elements per k-block (one 128-byte swizzle row)
constexpr int kStages = 4;
constexpr int kTcThreads = 192;   // 6 warps
constexpr uint32_t kStageA = kBM * kBK * 2;  // 16 KB
constexpr uint32_t kStageB = kBN * kBK * 2;  // 32 KB
constexpr int kNarrowA = 127;     // |delta| limit of fp16-class needles (int8)
constexpr int kNarrowB = 45;      // |delta| limit of fp16-class haystack images (b^2 < 2^11)
constexpr int64_t kExactSum = 1ll << 24;  // bound on every partial sum (exact FP32 integers)
constexpr unsigned long long kWaitBudgetNs = 2000000000ull;
constexpr unsigned long long kDrainBudgetNs = 200000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase with the given parity; false (and RICI_ERR_TIMEOUT) on timeout.  The
// waits between loads and MMAs poll without a pause: a stage is due every 300 ns, and waking up late
// idles the tensor cores (8,192 x 262,144 images of 64 x 64: 22.9 -> 22.0 ms;
// 100 x 90,001 in k_tc_query 321.8 -> 318.9 us).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *status,
                                          int *abort_flag, unsigned pause_ns = 32) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*(volatile int *)abort_flag) return false;
    if (globaltimer() - t0 > kWaitBudgetNs) {
      set_status(status, RICI_ERR_TIMEOUT);
      *(volatile int *)abort_flag = 1;
      return false;
    }
    if (pause_ns) __nanosleep(pause_ns);
  }
}

// Bounded wait used while tearing down: no abort flag, a short budget (copies and MMAs that are
// still in flight after an abort finish within microseconds unless the GPU itself is stuck).
__device__ __forceinline__ void mbar_drain(uint64_t *bar, uint32_t parity, int *status) {
  const unsigned long long t0 = globaltimer();
  while (!mbar_try_wait(bar, parity)) {
    if (globaltimer() - t0 > kDrainBudgetNs) {
      set_status(status, RICI_ERR_TIMEOUT);
      return;
    }
    __nanosleep(32);
  }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                     // leading byte offset (unused with 128B swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                     // descriptor version
  d |= (uint64_t)2 << 61;                     // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16: D = F32, A = B = F16, both K-major, M = 128, N = 256.
constexpr uint32_t kIdesc = (1u << 4)                      // D format F32
                            | (0u << 7) | (0u << 10)       // A, B format F16
                            | ((uint32_t)(kBN >> 3) << 17) // N / 8
                            | ((uint32_t)(kBM >> 4) << 24);// M / 16

template <uint32_t kDesc = kIdesc>
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(kDesc), "r"(accumulate));
}

__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
      "%30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- epilogue

// One needle's row of an accumulator tile: S values are integers with |S| < 2^24 for images of the
// class.  Counts S < thr, and keeps the smallest S up to lim with its smallest image index.
//
// lim starts from the best distance any tile has reported so far (or thr), so that after the first
// tiles hardly a column passes it: 32 columns cost a minimum, a comparison and an addition each, and
// are only looked at one by one when their minimum reaches lim in some lane.  With a 64-bit key per
// column up to thr, some lane passed in nearly every column, and the four epilogue warps took 16,000
// cycles per tile of 128 x 256 and bound the kernel below 32 x 32 pixels: 8,000 x 200,000 images of
// 8 x 8 2.63 -> 0.68 ms, of 16 x 16 2.60 -> 0.66 ms (start of the best distance at thr: 1.25, 1.16).
struct RowRank {
  float thr, lim;
  uint32_t j;  // image of the smallest S so far, ~0 if none
  int count;
};

__device__ __forceinline__ float clamp_s(int64_t s) {  // exact below 2^24, beyond every S above
  return (float)(s > (1ll << 25) ? (1ll << 25) : (s < -(1ll << 25) ? -(1ll << 25) : s));
}

// Rows that are not ranked get thr = lim = -infinity.
__device__ __forceinline__ RowRank row_rank(bool row_ok, int64_t asum, const int64_t *dtrue,
                                            const unsigned long long *best) {
  RowRank r;
  r.thr = r.lim = -__int_as_float(0x7f800000);
  r.j = ~0u;
  r.count = 0;
  if (row_ok) {
    r.thr = clamp_s(*dtrue - asum);
    // (other blocks lower it meanwhile; any earlier value will do)
    r.lim = fminf(r.thr, clamp_s((int64_t)(__ldcg(best) >> 32) - asum));
  }
  return r;
}

// Columns 0..31 of v, bit e of valid: column e is an image of the class; index(e) is its number.
template <typename F>
__device__ __forceinline__ void rank_columns(RowRank &r, uint32_t (&v)[32], uint32_t valid,
                                             F index) {
  if (valid != 0xffffffffu) {  // uniform over the warp
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (!((valid >> e) & 1u)) v[e] = 0x7f800000u;  // +infinity
  }
  float m = __uint_as_float(v[0]);
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    m = fminf(m, __uint_as_float(v[e]));
    r.count += __uint_as_float(v[e]) < r.thr;
  }
  if (m <= r.lim) {
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (__uint_as_float(v[e]) == m) {
        const uint32_t j = index(e);
        if (m < r.lim || j < r.j) r.j = j;
        r.lim = m;
      }
    }
  }
}

// The row's results: count of smaller distances, smallest (distance, image).
__device__ __forceinline__ void row_report(const RowRank &r, int64_t asum, int *rank,
                                           unsigned long long *best) {
  if (r.count) atomicAdd(rank, r.count);
  if (r.j != ~0u)
    atomicMin(best, ((unsigned long long)(asum + (int64_t)r.lim) << 32) | (unsigned long long)r.j);
}

// ---------------------------------------------------------------- operand encoding (S2)

// The 8 pixels of an image at k0 (zeros past its K0): one 16-byte load where it is aligned.
__device__ __forceinline__ uint4 pixels8(const uint16_t *img, int k0, int K0, bool vec) {
  if (k0 >= K0) return make_uint4(0, 0, 0, 0);
  if (vec) return *reinterpret_cast<const uint4 *>(img + k0);
  const uint16_t *q = img + k0;
  return make_uint4(q[0] | (uint32_t)q[1] << 16, q[2] | (uint32_t)q[3] << 16,
                    q[4] | (uint32_t)q[5] << 16, q[6] | (uint32_t)q[7] << 16);
}

// One warp per image (launch-wide index).  Needle rows: [m | a]; haystack rows: [b^2 | -2b]
// (fp16, K = 2 N^2).  Also: the class flag (wide = outside the fp16 class, see the exactness
// note above), the list of wide images, and for needles A_i.  With row_map (the haystack of a single
// scene) the rows of the class are written without gaps, *row_count of them, row_map[r] the image of
// row r: the image is read a second time (from the caches) once its class is known, and the GEMM
// has no columns for the images that others rank (7 % on the 5M-triangle scene: 8,192 needles x
// 262,144 of its images 24.6 -> 22.9 ms).
__global__ void k_tc_encode(const SearchScene *__restrict__ tab, const int *__restrict__ scene_of,
                            int64_t n, int N, int needle_side, __half *__restrict__ op,
                            int *__restrict__ wide_flag, int *__restrict__ wide_list,
                            int *__restrict__ wide_count, int *__restrict__ asum,
                            uint32_t *__restrict__ valid_mask, const int *__restrict__ skip_tile,
                            const int *__restrict__ any_tile, int *__restrict__ row_map,
                            int *__restrict__ row_count) {
  const int lane = threadIdx.x & 31;
  // operand rows no tile will load are not written: needle rows of skipped needle tiles (their
  // classes are still computed), and the haystack's when no needle tile is left
  const bool hay_written = needle_side || !any_tile || *any_tile != 0;
  if (!hay_written) return;  // nor does anything read the haystack's classes then
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int K0 = N * N;
  for (int64_t i = w; i < n; i += nw) {
    const SearchScene &sc = tab[scene_at(scene_of, i)];
    const uint16_t *img = needle_side ? sc.needles + (i - sc.qoff) * K0
                                      : sc.haystack + (i - sc.hoff) * K0;
    const int lim = needle_side ? kNarrowA : kNarrowB;
    const bool vec = aligned16(img);
    // needles: a2 = sum a^2; haystack: a2 = S2_j, s1 = S1_j (wrapped, and not used, for an image
    // with a wide delta; its operand row, if it has one, is garbage that no result reads)
    unsigned a2 = 0, s1 = 0;
    int wide = 0;
    auto classify = [&](const int (&d)[8]) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        wide |= d[e] < -lim || d[e] > lim;
        a2 += (unsigned)d[e] * (unsigned)d[e];
        if (!needle_side) s1 += (unsigned)abs(d[e]);
      }
    };
    auto write_row = [&](__half *row, int k0, const int (&d)[8]) {
      __align__(16) __half2 lo[4], hi[4];
      // |d| <= 127 as halves without conversions: 0x6600 + d are the bits of 1536 + d (0x6400 is
      // 1024, steps of 1); differences, products and doubles of such integers are exact
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t bits = __byte_perm((uint32_t)(0x6600 + d[2 * e]),
                                          (uint32_t)(0x6600 + d[2 * e + 1]), 0x5410);
        const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&bits),
                                  __floats2half2_rn(1536.0f, 1536.0f));
        if (needle_side) {
          lo[e] = __hne2(h, __floats2half2_rn(0.0f, 0.0f));
          hi[e] = h;
        } else {
          lo[e] = __hmul2(h, h);
          hi[e] = __hmul2(h, __floats2half2_rn(-2.0f, -2.0f));
        }
      }
      if (k0 < K0) {
        *reinterpret_cast<int4 *>(row + k0) = *reinterpret_cast<int4 *>(lo);
        *reinterpret_cast<int4 *>(row + K0 + k0) = *reinterpret_cast<int4 *>(hi);
      }
    };
    const bool write = !(needle_side && skip_tile && skip_tile[i / kBM]);
#pragma unroll 4
    for (int base = 0; base < K0; base += 256) {
      const int k0 = base + lane * 8;
      int d[8];
      deltas8(pixels8(img, k0, K0, vec), lane, N, d);
      classify(d);
      if (write && !row_map) write_row(op + i * (int64_t)(2 * K0), k0, d);
    }
    wide = __any_sync(0xffffffffu, wide);
    a2 = __reduce_add_sync(0xffffffffu, a2);
    s1 = __reduce_add_sync(0xffffffffu, s1);
    if (!needle_side && (int64_t)a2 + 2ll * kNarrowA * s1 >= kExactSum) wide = 1;
    int r = 0;
    if (lane == 0) {
      wide_flag[i] = wide;
      if (wide) wide_list[atomicAdd(wide_count, 1)] = (int)i;
      if (asum) asum[i] = (int)a2;
      if (valid_mask && !wide) atomicOr(&valid_mask[i >> 5], 1u << (i & 31));
      if (row_map && !wide) {
        r = atomicAdd(row_count, 1);
        row_map[r] = (int)i;
      }
    }
    if (!row_map || wide) continue;
    r = __shfl_sync(0xffffffffu, r, 0);
#pragma unroll 4
    for (int base = 0; base < K0; base += 256) {
      const int k0 = base + lane * 8;
      int d[8];
      deltas8(pixels8(img, k0, K0, vec), lane, N, d);
      write_row(op + r * (int64_t)(2 * K0), k0, d);
    }
  }
}

// The haystack images outside the fp16 class (list[0 .. *count)), one warp each: those of the
// split-square class get a row [r | -2b | 128 q] of op (at most cap rows) and an entry of map, the
// others an entry of left.
__global__ void k_tc_encode_split(const uint16_t *__restrict__ imgs, int N,
                                  const int *__restrict__ list, const int *__restrict__ count,
                                  int cap, __half *__restrict__ op, int *__restrict__ map,
                                  int *__restrict__ map_count, int *__restrict__ left,
                                  int *__restrict__ left_count, const int *__restrict__ any_tile) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t n = *count;
  const int K0 = N * N;
  const bool wanted = !any_tile || *any_tile != 0;
  for (int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; p < n; p += nw) {
    const int j = list[p];
    const uint16_t *img = imgs + (int64_t)j * K0;
    const bool vec = aligned16(img);
    unsigned s2 = 0, s1 = 0;
    int wide = !wanted;
    for (int base = 0; base < K0; base += 256) {
      int d[8];
      deltas8(pixels8(img, base + lane * 8, K0, vec), lane, N, d);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        wide |= d[e] < -kNarrowA || d[e] > kNarrowA;
        s2 += (unsigned)d[e] * (unsigned)d[e];
        s1 += (unsigned)abs(d[e]);
      }
    }
    wide = __any_sync(0xffffffffu, wide);
    s2 = __reduce_add_sync(0xffffffffu, s2);
    s1 = __reduce_add_sync(0xffffffffu, s1);
    if ((int64_t)s2 + 2ll * kNarrowA * s1 >= kExactSum) wide = 1;  // (s2, s1 exact when not wide)
    int at = cap;
    if (lane == 0) {
      if (!wide) at = atomicAdd(map_count, 1);
      if (at < cap) map[at] = j;
      else left[atomicAdd(left_count, 1)] = j;
    }
    at = __shfl_sync(0xffffffffu, at, 0);
    if (at >= cap) continue;
    __half *row = op + (int64_t)at * (3 * K0);
    for (int base = 0; base < K0; base += 256) {
      const int k0 = base + lane * 8;
      int d[8];
      deltas8(pixels8(img, k0, K0, vec), lane, N, d);
      __align__(16) __half r[8], b[8], q[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int sq = d[e] * d[e];
        r[e] = __int2half_rn(sq & 127);
        b[e] = __int2half_rn(-2 * d[e]);
        q[e] = __int2half_rn(sq & ~127);
      }
      if (k0 < K0) {
        *reinterpret_cast<int4 *>(row + k0) = *reinterpret_cast<int4 *>(r);
        *reinterpret_cast<int4 *>(row + K0 + k0) = *reinterpret_cast<int4 *>(b);
        *reinterpret_cast<int4 *>(row + 2 * K0 + k0) = *reinterpret_cast<int4 *>(q);
      }
    }
  }
}

// ---------------------------------------------------------------- GEMM + rank epilogue (S3, S5)

struct TcArgs {
  const SearchScene *tab;
  int num_scenes;
  int64_t tiles;                  // all scenes' tiles
  int KT;                         // 2 N^2
  const int *nwide;               // needle wide flags (TC class)
  const int *nflags;              // per-needle state (0 = searchable)
  const int *asum;                // A_i
  const int64_t *dtrue;           // d(i, match_i)
  const uint32_t *hvalid;         // bit j: haystack image j is narrow (null: every one is)
  int *rank;
  unsigned long long *best;
  int *status;
  int withhold_first_load;  // test hook: CTA 0 never issues its first stage (its waits time out)
  int group_m;              // needle tiles per group of the tile order
  const int *skip_needle;   // optional: 1 = this needle is ranked by another form
  const int *skip_tile;     // optional (single scene): 1 = needle tile m has no needle here
  const int *any_tile;      // with skip_tile: 0 = every tile is skipped (the grid returns at once)
  int ka_blocks;            // k-blocks of a needle row (block kb of K reads block kb % ka_blocks)
  const int *hcount;        // optional (single scene): the haystack is min(*hcount, hcap) rows
  int hcap;
  const int *hmap;          // optional: column j is haystack image hmap[j] of the caller
};

// Tiles and their order: search_tile_of (common.cuh).
__device__ __forceinline__ TcTile tile_of(const SearchScene *tab, int ns, int64_t t, int group_m) {
  return search_tile_of(tab, ns, t, group_m);
}

__global__ void __launch_bounds__(kTcThreads, 1)
    k_tc_rank(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
              TcArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled stages
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sA = smem;
  unsigned char *sB = smem + kStages * kStageA;
  uint64_t *full = reinterpret_cast<uint64_t *>(sB + kStages * kStageB);
  uint64_t *empty = full + kStages;
  uint64_t *tfull = empty + kStages;
  uint64_t *tempty = tfull + 2;
  uint64_t *drain = tempty + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
  int *abort_flag = reinterpret_cast<int *>(tmem_slot + 1);

  __shared__ SearchScene counted;  // hcount: the table entry with that many haystack rows
  // nothing to rank: return before any barrier, TMEM or TMA work (uniform over the grid)
  if (a.any_tile && *a.any_tile == 0) return;
  int64_t tiles = a.tiles;
  const SearchScene *tab = a.tab;
  if (a.hcount) {
    SearchScene sc = a.tab[0];
    sc.H = *a.hcount < a.hcap ? *a.hcount : a.hcap;
    sc.tiles_n = (int)((sc.H + kBN - 1) / kBN);
    tiles = (int64_t)sc.tiles_m * sc.tiles_n;
    if (threadIdx.x == 0) counted = sc;
    tab = &counted;
  }
  if (blockIdx.x >= tiles) return;  // (uniform over the block)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = a.KT / kBK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const TcTile tt = tile_of(tab, a.num_scenes, t, a.group_m);
        if (a.skip_tile && a.skip_tile[tt.m]) continue;  // every role skips the same tiles
        const int ya = (int)(tt.qbeg + tt.m * kBM), yb = (int)(tt.hbeg + tt.n * kBN);
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const uint32_t s = it % kStages, round = it / kStages;
          if (!mbar_wait(&empty[s], (round & 1) ^ 1, a.status, abort_flag, 0)) {
            ok = false;
            break;
          }
          if (a.withhold_first_load && blockIdx.x == 0 && it == 0) continue;
          mbar_arrive_expect_tx(&full[s], kStageA + kStageB);
          tma_load_2d(sA + s * kStageA, &map_a, &full[s],
                      (kb < a.ka_blocks ? kb : kb - a.ka_blocks) * kBK, ya);
          tma_load_2d(sB + s * kStageB, &map_b, &full[s], kb * kBK, yb);
        }
      }
      // Loads issued in the last kStages iterations may be unconsumed after an abort: wait for
      // them before the CTA exits (already-complete phases return at once).
      for (uint32_t j = 1; j <= (uint32_t)kStages && j <= it; ++j) {
        const uint32_t i = it - j;
        if (a.withhold_first_load && blockIdx.x == 0 && i == 0) continue;
        mbar_drain(&full[i % kStages], (i / kStages) & 1, a.status);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (one thread)
    if (lane == 0) {
      uint32_t it = 0, lt = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        if (a.skip_tile && a.skip_tile[tile_of(tab, a.num_scenes, t, a.group_m).m]) continue;
        const uint32_t buf = lt & 1, use = lt >> 1;
        ++lt;  // local count of processed tiles (selects the accumulator buffer)
        if (!mbar_wait(&tempty[buf], (use & 1) ^ 1, a.status, abort_flag, 0)) break;
        tc_fence_after();
        const uint32_t tacc = tmem + buf * kBN;
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const uint32_t s = it % kStages, round = it / kStages;
          if (!mbar_wait(&full[s], round & 1, a.status, abort_flag, 0)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(sA + s * kStageA), b0 = smem_u32(sB + s * kStageB);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            tc_mma(tacc, smem_desc(a0 + kk * 32), smem_desc(b0 + kk * 32),
                   (kb > 0 || kk > 0) ? 1u : 0u);
          }
          tc_commit(&empty[s]);  // frees the stage once these MMAs have read it
        }
        if (!ok) break;
        tc_commit(&tfull[buf]);  // accumulator ready for the epilogue
      }
      // every MMA this thread issued has finished before TMEM is released
      tc_commit(drain);
      mbar_drain(drain, 0, a.status);
    }
  } else {
    // ---------------- epilogue: warps 2..5, TMEM lane quarter = warp % 4
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    uint32_t lt = 0;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
      const TcTile tt = tile_of(tab, a.num_scenes, t, a.group_m);
      if (a.skip_tile && a.skip_tile[tt.m]) continue;
      const uint32_t buf = lt & 1, use = lt >> 1;
      ++lt;
      // warp-uniform outcome before the .sync.aligned TMEM loads
      const bool ready =
          __all_sync(0xffffffffu, mbar_wait(&tfull[buf], use & 1, a.status, abort_flag));
      if (!ready) break;
      tc_fence_after();
      const int64_t il = tt.m * kBM + row;  // scene-local needle
      const int64_t i = tt.qbeg + il;         // launch-wide needle
      const bool row_ok = il < tt.Q && a.nflags[i] == 0 && !a.nwide[i] &&
                          !(a.skip_needle && a.skip_needle[i]);
      const int64_t asum = row_ok ? a.asum[i] : 0;
      RowRank r = row_rank(row_ok, asum, a.dtrue + i, a.best + i);
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + buf * kBN;
#pragma unroll 1
      for (int c0 = 0; c0 < kBN; c0 += 32) {
        const int64_t j0 = tt.n * kBN + c0;  // scene-local haystack column
        if (j0 >= tt.H) break;               // (uniform over the block)
        uint32_t v[32];
        tmem_ld32(taddr + c0, v);
        uint32_t vm = 0xffffffffu;  // bit e: column j0 + e is a narrow haystack image of this scene
        if (a.hvalid) {
          const int64_t g0 = tt.hbeg + j0;   // launch-wide index (any alignment)
          const uint32_t lo = a.hvalid[g0 >> 5], hi = a.hvalid[(g0 >> 5) + 1];
          const int sh = (int)(g0 & 31);
          vm = sh ? (lo >> sh) | (hi << (32 - sh)) : lo;
        }
        const int64_t rem = tt.H - j0;
        if (rem < 32) vm &= (1u << rem) - 1u;
        rank_columns(r, v, vm, [&](int e) {
          return a.hmap ? (uint32_t)a.hmap[j0 + e] : (uint32_t)(j0 + e);
        });
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[buf]);
      if (row_ok) row_report(r, asum, a.rank + i, a.best + i);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// ---------------------------------------------------------------- few needles: encode and GEMM in one
//
// With few needles the GEMM is short and the haystack's operand rows (16 KB per image at N = 64, from
// 8 KB of pixels) cost the time: written by one kernel, read by the next.  Here the pixels go from
// global to shared memory once and become operand tiles there; nothing of the haystack is written
// back but the list of the images outside the fp16 class.
//
// Persistent over items of (needle tile of 128, haystack tile of 128 images), needle tiles of one
// haystack tile next to each other (its pixels come from L2 then).  K runs in chunks of 64 pixels:
//   warp 0      TMA of the pixels: 128 images x 64 pixels, 128-byte swizzle, 3 stages
//   warp 1      TMEM allocator and MMA issuer: m x b^2 and a x (-2 b), M = N = 128, K = 64 each
//   warps 2-5   epilogue, as in k_tc_rank (double-buffered: 2 x 128 TMEM columns)
//   warps 6-21  converters: four threads per image, 16 pixels each, from the pixel stage to the two
//               operand tiles (K-major, same swizzle), and the image's class
//   warp 22     TMA of the needles' operand blocks [m | a] of the chunk, 2 stages
// Shared-memory bandwidth bounds it: per chunk 48 KB arrive, 48 KB pass through the converters and the
// MMAs read 64 KB, 1,280 cycles at 128 bytes each against 1,376 measured (0.2 ms for 90,001 images of
// 64 x 64 and a needle tile; their pixels alone take 0.11 ms of HBM).  Whole calls, operand rows
// written by an encode and read by k_tc_rank against this kernel: 100 needles 715 -> 355 us, 256
// 754 -> 554 us, 512 959 -> 916 us, 1,024 1,357 -> 1,712 us; 90,001 images of 32 x 32: 128 needles
// 262 -> 147 us, 512 352 -> 305 us; so up to 512 needles take it.  (100 needles since then: 319 us.)  Over
// N = 8 to 128, 1 to 512 needles and 300 to 100,000 images no call is slower than with the rows in memory
// (512 needles of 8 x 8: 48 against 51 us with 300 images, 87 against 150 us with 100,000).
constexpr int kQN = 128;          // haystack images per tile
constexpr int kQRaw = 3;          // pixel stages (16 KB)
constexpr int kQOps = 2;          // operand stages (needles 32 KB, haystack 32 KB)
constexpr int kQConvWarps = 16;
constexpr int kQThreads = (7 + kQConvWarps) * 32;
constexpr uint32_t kQTile = 128 * 128;  // one operand or pixel block: 128 rows of 128 bytes
constexpr uint32_t kIdescQ = (1u << 4) | ((uint32_t)(kQN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);

struct QueryArgs {
  int64_t Q, H;
  int N, tiles_m;
  int64_t items;
  const int *nwide, *nflags, *asum;
  const int64_t *dtrue;
  int *rank;
  unsigned long long *best;
  int *hwide, *wh_list, *wh_count;
  int *status;
  int withhold_first_load;  // test hook: block 0 skips the load of its first pixels
};

__global__ void __launch_bounds__(kQThreads, 1)
    k_tc_query(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_px,
               QueryArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *s_px = smem;                          // kQRaw tiles
  unsigned char *s_a = s_px + kQRaw * kQTile;          // kQOps x (m, a)
  unsigned char *s_b = s_a + kQOps * 2 * kQTile;       // kQOps x (b^2, -2b)
  uint64_t *px_full = reinterpret_cast<uint64_t *>(s_b + kQOps * 2 * kQTile);
  uint64_t *px_empty = px_full + kQRaw;
  uint64_t *a_full = px_empty + kQRaw;
  uint64_t *b_full = a_full + kQOps;
  uint64_t *op_empty = b_full + kQOps;
  uint64_t *tfull = op_empty + kQOps;
  uint64_t *tempty = tfull + 2;
  uint64_t *cls_full = tempty + 2;
  uint64_t *drain = cls_full + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
  int *abort_flag = reinterpret_cast<int *>(tmem_slot + 1);
  unsigned char *cls = reinterpret_cast<unsigned char *>(abort_flag + 1);  // [2][kQN]: fp16 class

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int K0 = a.N * a.N, chunks = K0 / 64;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kQRaw; ++s) {
      mbar_init(&px_full[s], 1);
      mbar_init(&px_empty[s], kQConvWarps);
    }
    for (int s = 0; s < kQOps; ++s) {
      mbar_init(&a_full[s], 1);
      mbar_init(&b_full[s], kQConvWarps);
      mbar_init(&op_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
      mbar_init(&cls_full[b], kQConvWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------- pixels
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.items && ok; t += gridDim.x) {
        const int y = (int)(t / a.tiles_m * kQN);
        for (int c = 0; c < chunks; ++c, ++it) {
          const uint32_t s = it % kQRaw, round = it / kQRaw;
          if (!mbar_wait(&px_empty[s], (round & 1) ^ 1, a.status, abort_flag, 0)) {
            ok = false;
            break;
          }
          if (a.withhold_first_load && blockIdx.x == 0 && it == 0) continue;
          mbar_arrive_expect_tx(&px_full[s], kQTile);
          tma_load_2d(s_px + s * kQTile, &map_px, &px_full[s], c * 64, y);
        }
      }
      for (uint32_t j = 1; j <= (uint32_t)kQRaw && j <= it; ++j) {
        if (a.withhold_first_load && blockIdx.x == 0 && it == j) continue;
        mbar_drain(&px_full[(it - j) % kQRaw], ((it - j) / kQRaw) & 1, a.status);
      }
    }
  } else if (warp == 6 + kQConvWarps) {
    // ---------------- needle operands
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.items && ok; t += gridDim.x) {
        const int y = (int)(t % a.tiles_m * kBM);
        for (int c = 0; c < chunks; ++c, ++it) {
          const uint32_t s = it % kQOps, round = it / kQOps;
          if (!mbar_wait(&op_empty[s], (round & 1) ^ 1, a.status, abort_flag, 0)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&a_full[s], 2 * kQTile);
          tma_load_2d(s_a + s * 2 * kQTile, &map_a, &a_full[s], c * 64, y);
          tma_load_2d(s_a + s * 2 * kQTile + kQTile, &map_a, &a_full[s], K0 + c * 64, y);
        }
      }
      for (uint32_t j = 1; j <= (uint32_t)kQOps && j <= it; ++j)
        mbar_drain(&a_full[(it - j) % kQOps], ((it - j) / kQOps) & 1, a.status);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (one thread)
    if (lane == 0) {
      uint32_t it = 0, lt = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.items && ok; t += gridDim.x) {
        const uint32_t buf = lt & 1, use = lt >> 1;
        ++lt;
        if (!mbar_wait(&tempty[buf], (use & 1) ^ 1, a.status, abort_flag, 0)) break;
        tc_fence_after();
        const uint32_t tacc = tmem + buf * kQN;
        for (int c = 0; c < chunks; ++c, ++it) {
          const uint32_t s = it % kQOps, round = it / kQOps;
          if (!mbar_wait(&a_full[s], round & 1, a.status, abort_flag, 0) ||
              !mbar_wait(&b_full[s], round & 1, a.status, abort_flag, 0)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = smem_u32(s_a + s * 2 * kQTile), b0 = smem_u32(s_b + s * 2 * kQTile);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {  // 4 steps of K = 16 in either block
            const uint32_t off = (kk >> 2) * kQTile + (kk & 3) * 32;
            tc_mma<kIdescQ>(tacc, smem_desc(a0 + off), smem_desc(b0 + off),
                            (c > 0 || kk > 0) ? 1u : 0u);
          }
          tc_commit(&op_empty[s]);
        }
        if (!ok) break;
        tc_commit(&tfull[buf]);
      }
      tc_commit(drain);
      mbar_drain(drain, 0, a.status);
    }
  } else if (warp >= 6) {
    // ---------------- converters: image `row` of the tile, 16 pixels from 16 `quad` of a chunk.  Two
    // pixels at a time: with w = (p0, p1) and v = (p before, p0), w - v + 0x66006600 are the bits of
    // the halves 1536 + d0, 1536 + d1 (as in k_tc_encode; the low half lends nothing to the high one
    // as long as |d0| < 0x6600), so a pair costs nine instructions in all.  Deltas past the halves'
    // range give halves past the class limit, infinities or NaN; pixels of 32,768 and more, whose
    // differences could wrap around, put the image outside the class too (the split-square encode
    // looks at those again).
    const int ct = threadIdx.x - 6 * 32, row = ct >> 2, quad = ct & 3;
    const __half2 k1536 = __floats2half2_rn(1536.0f, 1536.0f), km2 = __floats2half2_rn(-2.0f, -2.0f);
    uint32_t it = 0, lt = 0;
    bool ok = true;
    for (int64_t t = blockIdx.x; t < a.items && ok; t += gridDim.x) {
      const uint32_t buf = lt & 1, use = lt >> 1;
      ++lt;
      unsigned any = 0, last = 0;
      int s2 = 0, s1 = 0;
      __half2 top = __floats2half2_rn(0.0f, 0.0f);
      for (int c = 0; c < chunks; ++c, ++it) {
        const uint32_t s = it % kQRaw, o = it % kQOps;
        ok = __all_sync(0xffffffffu,
                        mbar_wait(&px_full[s], (it / kQRaw) & 1, a.status, abort_flag) &&
                            mbar_wait(&op_empty[o], ((it / kQOps) & 1) ^ 1, a.status, abort_flag));
        if (!ok) break;
        const unsigned char *src = s_px + s * kQTile + row * 128;
        unsigned char *dst = s_b + o * 2 * kQTile + row * 128;
        uint32_t w[8];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const uint4 x = *reinterpret_cast<const uint4 *>(src + (((quad * 2 + v) ^ (row & 7)) << 4));
          w[4 * v] = x.x;
          w[4 * v + 1] = x.y;
          w[4 * v + 2] = x.z;
          w[4 * v + 3] = x.w;
        }
        // the word before the first: the previous thread's last one, of this chunk, or (first thread;
        // only rows of 128 pixels continue there) of the chunk before
        const unsigned left = __shfl_up_sync(0xffffffffu, w[7], 1);
        const unsigned carry = __shfl_down_sync(0xffffffffu, last, 3);
        last = w[7];
        uint32_t prev = quad ? left : carry;
        __half2 sum = __floats2half2_rn(0.0f, 0.0f);  // sum |b| of the chunk's pairs: at most 8 x 45
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          // rows start at multiples of N pixels, so only at the first pixel of 8: delta 0 there
          if (((c * 64 + quad * 16 + v * 8) & (a.N - 1)) == 0) prev = w[4 * v] << 16;
          uint32_t sq[4], dbl[4], bits[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t x = w[4 * v + e];
            bits[e] = x - __funnelshift_l(prev, x, 16) + 0x66006600u;
            prev = x;
            any |= x;
            const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&bits[e]), k1536);
            const __half2 ha = __habs2(h);
            top = __hmax2_nan(top, ha);
            sum = __hadd2(sum, ha);
            const __half2 hs = __hmul2(h, h), hd = __hmul2(h, km2);
            sq[e] = *reinterpret_cast<const uint32_t *>(&hs);
            dbl[e] = *reinterpret_cast<const uint32_t *>(&hd);
          }
#pragma unroll
          for (int e = 0; e < 4; e += 2) {  // the low bytes of the halves' bits are the deltas'
            const int d4 = (int)__byte_perm(bits[e], bits[e + 1], 0x6420);
            s2 = __dp4a(d4, d4, s2);
          }
          const int at = ((quad * 2 + v) ^ (row & 7)) << 4;
          *reinterpret_cast<uint4 *>(dst + at) = make_uint4(sq[0], sq[1], sq[2], sq[3]);
          *reinterpret_cast<uint4 *>(dst + kQTile + at) = make_uint4(dbl[0], dbl[1], dbl[2], dbl[3]);
        }
        const float2 sf = __half22float2(sum);
        s1 += (int)fminf(sf.x + sf.y, 65536.0f);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&px_empty[s]);
          mbar_arrive(&b_full[o]);
        }
      }
      if (!ok) break;
      // the image's class, once the epilogue has read the buffer's previous one
      ok = __all_sync(0xffffffffu, mbar_wait(&tempty[buf], (use & 1) ^ 1, a.status, abort_flag));
      if (!ok) break;
      const float2 tf = __half22float2(top);
      int wide = !(tf.x <= (float)kNarrowB && tf.y <= (float)kNarrowB) || (any & 0x80008000u) != 0;
#pragma unroll
      for (int k = 1; k < 4; k <<= 1) {
        wide |= __shfl_xor_sync(0xffffffffu, wide, k);
        s2 += __shfl_xor_sync(0xffffffffu, s2, k);
        s1 += __shfl_xor_sync(0xffffffffu, s1, k);
      }
      // (s2, s1 exact when every |b| <= 45)
      if ((int64_t)s2 + 2ll * kNarrowA * s1 >= kExactSum) wide = 1;
      const int64_t j = t / a.tiles_m * kQN + row;
      if (quad == 0) {
        cls[buf * kQN + row] = j < a.H && !wide;
        if (j < a.H && t % a.tiles_m == 0) {
          a.hwide[j] = wide;
          if (wide) a.wh_list[atomicAdd(a.wh_count, 1)] = (int)j;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&cls_full[buf]);
    }
  } else {
    // ---------------- epilogue: warps 2..5, TMEM lane quarter = warp % 4
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    uint32_t lt = 0;
    for (int64_t t = blockIdx.x; t < a.items; t += gridDim.x) {
      const uint32_t buf = lt & 1, use = lt >> 1;
      ++lt;
      const bool ready = __all_sync(
          0xffffffffu, mbar_wait(&tfull[buf], use & 1, a.status, abort_flag) &&
                           mbar_wait(&cls_full[buf], use & 1, a.status, abort_flag));
      if (!ready) break;
      tc_fence_after();
      const int64_t i = t % a.tiles_m * kBM + row;
      const bool row_ok = i < a.Q && a.nflags[i] == 0 && !a.nwide[i];
      const int64_t asum = row_ok ? a.asum[i] : 0;
      RowRank r = row_rank(row_ok, asum, a.dtrue + i, a.best + i);
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + buf * kQN;
#pragma unroll 1
      for (int c0 = 0; c0 < kQN; c0 += 32) {
        uint32_t v[32];
        tmem_ld32(taddr + c0, v);
        const uint32_t in = __ballot_sync(0xffffffffu, cls[buf * kQN + c0 + lane] != 0);
        const uint32_t j0 = (uint32_t)(t / a.tiles_m * kQN + c0);
        rank_columns(r, v, in, [&](int e) { return j0 + e; });
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[buf]);
      if (row_ok) row_report(r, asum, a.rank + i, a.best + i);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Row-major 16-bit matrix [rows][KT] in boxes of 64 x box_rows, 128-byte swizzle.
cudaError_t encode_map(CUtensorMap *map, const void *base, int64_t rows, int KT, int box_rows,
                       bool half = true) {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void *p = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !p) return cudaErrorNotSupported;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  cuuint64_t dims[2] = {(cuuint64_t)KT, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)KT * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, half ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2,
                  const_cast<void *>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

// Rows kept for split-square images: an eighth of the haystack, in whole tiles (images beyond that go to
// the CUDA cores).
static int split_capacity(int64_t H) {
  const int64_t want = (H / 8 + kBN) / kBN * kBN;
  return (int)(want < H ? want : H);
}

int64_t tc_split_bytes(int64_t H, int N) {
  return split_capacity(H) * (3ll * N * N) * (int64_t)sizeof(__half);
}

// Most needles of a call that k_tc_query takes (measured above).
constexpr int64_t kQueryNeedles = 512;

bool tc_supported(int N) { return N == 8 || N == 16 || N == 32 || N == 64 || N == 128; }

int64_t tc_workspace_bytes(int64_t Q, int64_t H, int N, bool single_scene) {
  const int64_t KT = 2ll * N * N;
  const int cap = single_scene ? split_capacity(H) : 0;
  Carver c(nullptr);
  c.take<__half>(Q * KT);
  c.take<__half>(H * KT);
  c.take<int>(Q);                 // A_i
  c.take<uint32_t>(single_scene ? H : (H + 31) / 32 + 2);  // image of each row, or class bits
  c.take<int>(cap);               // images of the split-square rows
  return c.off + 256;
}

cudaError_t launch_tc_encode_and_rank(const SearchScene *tab, int num_scenes, const int *qscene,
                                      const int *hscene, int64_t Q, int64_t H,
                                      int64_t tiles_total, int N, void *ws, int *nwide, int *hwide,
                                      int *wn_list, int *wh_list, int *counts,
                                      const int *nflags, const int64_t *dtrue, int *rank,
                                      unsigned long long *best, int *status, int test_withhold,
                                      cudaStream_t st, const int *skip_needle,
                                      const int *skip_tile, const int *any_tile,
                                      const uint16_t *haystack, bool split, int *left_list,
                                      int *left_count, void *split_rows) {
  const int64_t KT = 2ll * N * N;
  const int cap = num_scenes == 1 ? split_capacity(H) : 0;
  Carver c(ws);
  __half *opa = c.take<__half>(Q * KT);
  __half *opb = c.take<__half>(H * KT);
  int *asum = c.take<int>(Q);
  const bool single = num_scenes == 1;
  uint32_t *hvalid = c.take<uint32_t>(single ? H : (H + 31) / 32 + 2);
  int *const row_map = single ? reinterpret_cast<int *>(hvalid) : nullptr;
  __half *const ops = static_cast<__half *>(split_rows);
  int *smap = c.take<int>(cap);
  int *const scount = counts + 7;  // their number (zeroed by the caller with the other counts)
  int *const rcount = counts + 8;  // rows of the fp16 class (zeroed likewise)
  cudaError_t e;
  if (!single &&
      (e = cudaMemsetAsync(hvalid, 0, sizeof(uint32_t) * ((H + 31) / 32 + 2), st)) != cudaSuccess)
    return e;
  auto blocks_for = [](int64_t warps) {
    int64_t b = (warps + 7) / 8;
    return (int)(b < 152 * 64 ? (b > 0 ? b : 1) : 152 * 64);
  };
  const int *any = skip_tile ? any_tile : nullptr;
  k_tc_encode<<<blocks_for(Q), 256, 0, st>>>(tab, qscene, Q, N, 1, opa, nwide, wn_list, counts + 0,
                                             asum, nullptr, skip_tile, nullptr, nullptr, nullptr);
  // few needles of one scene: the haystack's operands are built inside the GEMM kernel
  const bool query = haystack && !skip_tile && Q <= kQueryNeedles &&
                     (reinterpret_cast<uintptr_t>(haystack) & 15) == 0;  // (TMA)
  if (query) {
    CUtensorMap mq, mp;
    if ((e = encode_map(&mq, opa, Q, (int)KT, kBM)) != cudaSuccess) return e;
    if ((e = encode_map(&mp, haystack, H, (int)(KT / 2), kQN, false)) != cudaSuccess) return e;
    QueryArgs q;
    q.Q = Q;
    q.H = H;
    q.N = N;
    q.tiles_m = (int)((Q + kBM - 1) / kBM);
    q.items = q.tiles_m * ((H + kQN - 1) / kQN);
    q.nwide = nwide;
    q.nflags = nflags;
    q.asum = asum;
    q.dtrue = dtrue;
    q.rank = rank;
    q.best = best;
    q.hwide = hwide;
    q.wh_list = wh_list;
    q.wh_count = counts + 1;
    q.status = status;
    q.withhold_first_load = test_withhold;
    const size_t smem_q = 1024 + (kQRaw + 4 * kQOps) * kQTile + 512;
    if ((e = cudaFuncSetAttribute(k_tc_query, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem_q)) != cudaSuccess)
      return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_tc_query<<<(unsigned)(q.items < sms ? q.items : sms), kQThreads, smem_q, st>>>(mq, mp, q);
  } else {
    k_tc_encode<<<blocks_for(H), 256, 0, st>>>(tab, hscene, H, N, 0, opb, hwide, wh_list,
                                               counts + 1, nullptr, single ? nullptr : hvalid,
                                               nullptr, any, row_map, rcount);
  }
  count_launches(2);
  if (split) {
    k_tc_encode_split<<<blocks_for(cap), 256, 0, st>>>(haystack, N, wh_list, counts + 1, cap,
                                                       ops, smap, scount, left_list, left_count,
                                                       any);
    count_launches(1);
  }
  if (tiles_total == 0) return cudaGetLastError();
  CUtensorMap ma, mb;
  if ((e = encode_map(&ma, opa, Q, (int)KT, kBM)) != cudaSuccess) return e;
  if ((e = encode_map(&mb, opb, H, (int)KT, kBN)) != cudaSuccess) return e;
  TcArgs a;
  a.tab = tab;
  a.num_scenes = num_scenes;
  a.tiles = tiles_total;
  a.KT = (int)KT;
  a.nwide = nwide;
  a.nflags = nflags;
  a.asum = asum;
  a.dtrue = dtrue;
  a.hvalid = single ? nullptr : hvalid;
  a.rank = rank;
  a.best = best;
  a.status = status;
  a.withhold_first_load = test_withhold;
  a.group_m = current_tuning().tc_group_m;
  a.skip_needle = skip_needle;
  a.skip_tile = skip_tile;
  a.any_tile = any;
  a.ka_blocks = (int)(KT / kBK);
  a.hcount = single ? rcount : nullptr;
  a.hcap = (int)H;
  a.hmap = row_map;
  const size_t smem = 1024 + kStages * (kStageA + kStageB) + 256;
  if ((e = cudaFuncSetAttribute(k_tc_rank, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)) != cudaSuccess)
    return e;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = (int)(tiles_total < sms ? tiles_total : sms);
  if (!query) {
    k_tc_rank<<<grid, kTcThreads, smem, st>>>(ma, mb, a);
    count_launches(1);
  }
  if (split) {
    // the needles' tiles against the compacted split-square images (count on the device)
    if ((e = encode_map(&mb, ops, cap, (int)(KT / 2 * 3), kBN)) != cudaSuccess) return e;
    a.KT = (int)(KT / 2 * 3);
    a.hcount = scount;
    a.hcap = cap;
    a.hvalid = nullptr;
    a.hmap = smap;
    a.withhold_first_load = 0;
    k_tc_rank<<<grid, kTcThreads, smem, st>>>(ma, mb, a);
    count_launches(1);
  }
  return cudaGetLastError();
}

}  // namespace rici
