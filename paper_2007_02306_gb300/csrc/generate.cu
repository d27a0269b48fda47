// RICI generation on sm_103a (Section 3.1 of the paper).
//
// Pipeline per rici_generate call (all on the caller's stream, no host synchronisation):
//   1. k_tri_bbox     box of the triangles' bounding-sphere centres, per scene.
//   2. k_tri_bin      bounding sphere of every triangle; bin it by the Morton code of its centre
//                     on a 2^L grid over that box (8^L bins, L <= 7).
//   3. scan           bin counts -> bin starts.
//   4. k_tri_scatter  64-byte triangle records (sphere, FP32 vertices, global indices) in bin
//                     order: the records follow a space-filling curve, so runs of consecutive
//                     records are compact in space.
//   5. k_chunk_spheres  a bounding sphere of every run of 32 records (chunk) and of 1024
//                     records (group).
//   6. k_generate     one CTA per oriented point.  Its warps test the groups of the point's
//                     scene against the support cylinder, then the chunks of passing groups,
//                     then the records of passing chunks (a sphere fails only if every record
//                     in it fails), project the surviving triangles (Eqs.
//                     relativeLocation..secondRotation) and split the (triangle, layer) work
//                     evenly over the 32 lanes.  Each layer's single/double crossing radii
//                     (Section 3.1.2) become column intervals added to a shared-memory
//                     difference image, which is prefix summed, saturated and stored as packed
//                     uint16 (32- or 64-bit stores).
// The clutter measure (bottom of this file) walks the same sorted records; spin images bin
// triangles into a hashed uniform grid instead and scan the grid cells around each oriented point.
//
// Exactness: the FP32 path carries a forward error bound for every predicate (vertex side of a
// layer, |E| against alpha, the signs of E0.D and E1.D, the distance of the chord's closest point).
// A (triangle, layer) whose predicate lies inside its bound is evaluated again with pairs of floats
// (48 bits, their own bounds), and where those do not decide either in FP64 with the definition's
// operation order (explicit _rn intrinsics, no contraction), so every count equals the FP64
// definition bit for bit.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"

namespace rici {
namespace {

constexpr float kU = 5.9604644775390625e-08f;  // 2^-24: unit roundoff of FP32
constexpr float kSafety = 2.0f;                // multiplies every derived error bound
constexpr uint32_t kSkip = 0xFFFFFFFEu;
constexpr float kCellClamp = 1048576.0f;  // |cell coordinate| limit (2^20)
constexpr int kSlot = 20;  // words per staged triangle (a multiple of 4 whose first 8 multiples
                           // lie in 8 different groups of 4 banks: conflict-free 16-byte loads)
constexpr int kScanItems = kGenScanItems;
constexpr int kSpinMaxCellsPerReach = 3;  // spin images: up to (2 x 3 + 1)^3 cells per point
constexpr int kBandQ = 128;  // band queue of a warp: 31 left over + 3 layers of each of 32 triangles
// shared words per warp: candidate queue, band queue (triangle records, then their layers as
// bytes), place in the walk over groups, staged triangles; a multiple of 4
constexpr int kPerWarp = 64 + kBandQ + kBandQ / 4 + 4 + 32 * kSlot;

__host__ __device__ constexpr uint32_t bucket_count(int64_t nt) { return generate_bucket_count(nt); }

__device__ __forceinline__ int cell_coord(float x, float inv_cell) {
  float f = floorf(x * inv_cell);
  f = fminf(fmaxf(f, -kCellClamp), kCellClamp);
  return (int)f;
}

__device__ __forceinline__ uint32_t cell_hash(int ix, int iy, int iz, uint32_t mask) {
  return (((uint32_t)ix * 73856093u) ^ ((uint32_t)iy * 19349663u) ^ ((uint32_t)iz * 83492791u)) &
         mask;
}

// Order-preserving map of finite floats to int32 (a min / max of the ints is a min / max of the
// floats); the map is its own inverse.
__device__ __forceinline__ int float_order(float f) {
  const int i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float order_float(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// Bits of x (< 2^10) spread to every third position.
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
  x &= 0x3ffu;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

struct TriSphere {
  float cx, cy, cz, r;
};

// Bounding sphere of the triangle's AABB, inflated to cover rounding of centre and radius.
__device__ __forceinline__ TriSphere tri_sphere(const float v[9]) {
  float lx = fminf(fminf(v[0], v[3]), v[6]), hx = fmaxf(fmaxf(v[0], v[3]), v[6]);
  float ly = fminf(fminf(v[1], v[4]), v[7]), hy = fmaxf(fmaxf(v[1], v[4]), v[7]);
  float lz = fminf(fminf(v[2], v[5]), v[8]), hz = fmaxf(fmaxf(v[2], v[5]), v[8]);
  TriSphere s;
  s.cx = 0.5f * (lx + hx);
  s.cy = 0.5f * (ly + hy);
  s.cz = 0.5f * (lz + hz);
  float ex = 0.5f * (hx - lx), ey = 0.5f * (hy - ly), ez = 0.5f * (hz - lz);
  float cm = fmaxf(fabsf(s.cx), fmaxf(fabsf(s.cy), fabsf(s.cz)));
  s.r = sqrtf(ex * ex + ey * ey + ez * ez) * (1.0f + 1e-5f) + 1e-6f * cm + 1e-30f;
  return s;
}

struct GridParams {
  float inv_cell;
  float r_big;
  uint32_t mask;
};

// Scene of a launch-wide index: the last table entry whose offset is <= idx (entries with no
// items share their offset with the next one, so the match always owns idx).
__device__ __forceinline__ int scene_of_tri(const GenScene *tab, int ns, int64_t idx) {
  int lo = 0, hi = ns - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].tri_off <= idx) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ int scene_of_origin(const GenScene *tab, int ns, int64_t idx) {
  int lo = 0, hi = ns - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].origin_off <= idx) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Box of the bounding-sphere centres of each scene's valid triangles (ints of float_order; the
// table fill sets every box empty).  Triangles with a bad index or a non-finite vertex are left
// to k_tri_bin, which reports them.  Warps whose triangles all belong to one scene reduce first.
__global__ void k_tri_bbox(const GenScene *__restrict__ tab, int ns, int64_t nt_total,
                           int *__restrict__ bbox) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;  // a multiple of 32
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); t0 < nt_total;
       t0 += stride) {
    const int64_t t = t0 + lane < nt_total ? t0 + lane : nt_total - 1;
    const int sidx = scene_of_tri(tab, ns, t);
    const GenScene &sc = tab[sidx];
    const int64_t tl = t - sc.tri_off;
    const int64_t nv = sc.nv;
    bool ok = t0 + lane < nt_total;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (ok) {
      int id[3] = {sc.tris[3 * tl], sc.tris[3 * tl + 1], sc.tris[3 * tl + 2]};
      ok = id[0] >= 0 && id[0] < nv && id[1] >= 0 && id[1] < nv && id[2] >= 0 && id[2] < nv;
      if (ok) {
        float v[9];
        for (int k = 0; k < 3; ++k)
          for (int d = 0; d < 3; ++d) {
            v[3 * k + d] = sc.V[3 * (int64_t)id[k] + d];
            ok = ok && isfinite(v[3 * k + d]);
          }
        if (ok) {
          const TriSphere ts_ = tri_sphere(v);
          lo[0] = hi[0] = ts_.cx;
          lo[1] = hi[1] = ts_.cy;
          lo[2] = hi[2] = ts_.cz;
        }
      }
    }
    const int s0 = __shfl_sync(0xffffffffu, sidx, 0);
    if (__all_sync(0xffffffffu, sidx == s0)) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], d));
          hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], d));
        }
      // lanes 0-5 hold one side of the box each.  The box only grows, so a warp inside what it reads of
      // it has nothing to add: without that look its six atomics meet those of all others (the kernel
      // took 125 us for 1M triangles; 100 images of them 306 -> 198 us in all)
      if (lane < 6 && lo[0] <= hi[0]) {
        const float x = lane == 0   ? lo[0]
                        : lane == 1 ? lo[1]
                        : lane == 2 ? lo[2]
                        : lane == 3 ? hi[0]
                        : lane == 4 ? hi[1]
                                    : hi[2];
        int *const b = bbox + 8 * (int64_t)sidx + lane;
        const int v = float_order(x), now = __ldcg(b);
        if (lane < 3 && v < now) atomicMin(b, v);
        if (lane >= 3 && v > now) atomicMax(b, v);
      }
    } else if (ok) {
      int *bb = bbox + 8 * (int64_t)sidx;
      for (int k = 0; k < 3; ++k) {
        atomicMin(bb + k, float_order(lo[k]));
        atomicMax(bb + 3 + k, float_order(hi[k]));
      }
    }
  }
}

// Morton bin of a bounding-sphere centre on a 2^L grid over the box bb (ints of float_order) of its
// scene's centres, 8^L <= nbuckets.
__device__ __forceinline__ uint32_t morton_bin(const TriSphere &s, const int *bb, uint32_t nbuckets) {
  const float lo[3] = {order_float(bb[0]), order_float(bb[1]), order_float(bb[2])};
  const float ext = fmaxf(fmaxf(order_float(bb[3]) - lo[0], order_float(bb[4]) - lo[1]),
                          order_float(bb[5]) - lo[2]);
  const int L = (31 - __clz(nbuckets)) / 3;
  const float top = (float)((1 << L) - 1);
  const float scale = (ext > 0.0f && ext < 1e30f) ? (float)(1 << L) / ext : 0.0f;
  const float c[3] = {s.cx, s.cy, s.cz};
  uint32_t q[3];
  for (int k = 0; k < 3; ++k) {
    const float f = scale > 0.0f ? floorf((c[k] - lo[k]) * scale) : 0.0f;
    q[k] = (uint32_t)fminf(fmaxf(f, 0.0f), top);
  }
  return spread3(q[0]) | (spread3(q[1]) << 1) | (spread3(q[2]) << 2);
}

// Bins every triangle by its bounding sphere.  With bbox == nullptr (spin images): a hashed uniform
// grid of cell edge 1 / inv_cell, wide triangles in the scene's big list.  Otherwise (generation,
// clutter measure): every triangle by the Morton code of its centre on a 2^L grid
// over its scene's box of centres (8^L <= the scene's bucket count), so that records sorted by
// bucket follow a space-filling curve and runs of consecutive records are compact.
__global__ void k_tri_bin(const GenScene *__restrict__ tab, int ns, int64_t nt_total, GridParams g,
                          const int *__restrict__ bbox, int *__restrict__ counts,
                          uint32_t *__restrict__ tb, int *__restrict__ ts, int *status) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt_total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const GenScene &sc = tab[scene_of_tri(tab, ns, t)];
    const int64_t tl = t - sc.tri_off;
    const int64_t nv = sc.nv;
    int id[3] = {sc.tris[3 * tl], sc.tris[3 * tl + 1], sc.tris[3 * tl + 2]};
    if (id[0] < 0 || id[0] >= nv || id[1] < 0 || id[1] >= nv || id[2] < 0 || id[2] >= nv) {
      set_status(status, RICI_ERR_INDEX_OUT_OF_RANGE);
      tb[t] = kSkip;
      continue;
    }
    float v[9];
    bool fin = true;
    for (int k = 0; k < 3; ++k)
      for (int d = 0; d < 3; ++d) {
        v[3 * k + d] = sc.V[3 * (int64_t)id[k] + d];
        fin = fin && isfinite(v[3 * k + d]);
      }
    if (!fin) {
      set_status(status, RICI_ERR_NONFINITE_INPUT);
      tb[t] = kSkip;
      continue;
    }
    TriSphere s = tri_sphere(v);
    uint32_t b = sc.nbuckets;  // the scene's big list
    if (bbox) {
      b = morton_bin(s, bbox + 8 * (int64_t)scene_of_tri(tab, ns, t), sc.nbuckets);
    } else {
      const float lim = kCellClamp - 4.0f;
      bool big = s.r > g.r_big || !(fabsf(s.cx * g.inv_cell) < lim) ||
                 !(fabsf(s.cy * g.inv_cell) < lim) || !(fabsf(s.cz * g.inv_cell) < lim);
      if (!big)
        b = cell_hash(cell_coord(s.cx, g.inv_cell), cell_coord(s.cy, g.inv_cell),
                      cell_coord(s.cz, g.inv_cell), sc.nbuckets - 1);
    }
    const uint32_t gb = (uint32_t)(sc.bucket_off + b);
    tb[t] = gb;
    ts[t] = atomicAdd(&counts[gb], 1);
  }
}

__global__ void k_tri_scatter(const GenScene *__restrict__ tab, int ns, int64_t nt_total,
                              const uint32_t *__restrict__ tb, const int *__restrict__ ts,
                              const int *__restrict__ starts, float4 *__restrict__ rec) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt_total;
       t += (int64_t)gridDim.x * blockDim.x) {
    uint32_t b = tb[t];
    if (b == kSkip) continue;
    const GenScene &sc = tab[scene_of_tri(tab, ns, t)];
    const int64_t tl = t - sc.tri_off;
    const int64_t pos = (int64_t)starts[b] + ts[t];
    int id[3] = {sc.tris[3 * tl], sc.tris[3 * tl + 1], sc.tris[3 * tl + 2]};
    float v[9];
    for (int k = 0; k < 3; ++k)
      for (int d = 0; d < 3; ++d) v[3 * k + d] = sc.V[3 * (int64_t)id[k] + d];
    TriSphere s = tri_sphere(v);
    // four columns of nt_total records: the culling pass streams only the first (16 bytes per
    // triangle), the set-up of survivors reads the other three
    rec[pos] = make_float4(s.cx, s.cy, s.cz, s.r);
    rec[nt_total + pos] = make_float4(v[0], v[1], v[2], v[3]);
    rec[2 * nt_total + pos] = make_float4(v[4], v[5], v[6], v[7]);
    rec[3 * nt_total + pos] = make_float4(v[8], __int_as_float(id[0]), __int_as_float(id[1]),
                                          __int_as_float(id[2]));
  }
}

// Warp collective: a sphere containing every lane's sphere c (c.w < 0: none).  Returns w < 0 when
// no lane has one and an infinite radius when the result is not finite.  The centre is that of
// the box of the spheres; the radius is the largest |c - C| + c.w, raised to cover its rounding.
__device__ __forceinline__ float4 sphere_of_spheres(float4 c) {
  const bool v = c.w >= 0.0f;
  float lo[3] = {v ? c.x - c.w : INFINITY, v ? c.y - c.w : INFINITY, v ? c.z - c.w : INFINITY};
  float hi[3] = {v ? c.x + c.w : -INFINITY, v ? c.y + c.w : -INFINITY, v ? c.z + c.w : -INFINITY};
#pragma unroll
  for (int d = 16; d > 0; d >>= 1)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], d));
      hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], d));
    }
  if (!__any_sync(0xffffffffu, v)) return make_float4(0.0f, 0.0f, 0.0f, -1.0f);
  const float Cx = 0.5f * (lo[0] + hi[0]), Cy = 0.5f * (lo[1] + hi[1]), Cz = 0.5f * (lo[2] + hi[2]);
  float e = 0.0f;
  if (v) {
    const float dx = c.x - Cx, dy = c.y - Cy, dz = c.z - Cz;
    e = sqrtf(dx * dx + dy * dy + dz * dz) + c.w;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, d));
  const float rho = e * (1.0f + 1e-5f) + 1e-6f * (fabsf(Cx) + fabsf(Cy) + fabsf(Cz)) + 1e-30f;
  if (!(isfinite(Cx) && isfinite(Cy) && isfinite(Cz) && rho < 1e30f))
    return make_float4(0.0f, 0.0f, 0.0f, INFINITY);
  return make_float4(Cx, Cy, Cz, rho);
}

constexpr int kChunkShift = 5;   // 32 records per chunk
constexpr int kGroupShift = 10;  // 32 chunks (1024 records) per group

// Bounding spheres of every 32-record chunk and every 1024-record group of the sorted records
// (*nrec of them), each containing the bounding spheres of its records; a chunk or group at a
// scene boundary covers the records of both scenes.  One block of 32 warps per group.
__global__ void __launch_bounds__(1024) k_chunk_spheres(const float4 *__restrict__ rec,
                                                        const int *__restrict__ nrec,
                                                        float4 *__restrict__ chk,
                                                        float4 *__restrict__ grp) {
  __shared__ float4 cs[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t n = *nrec;
  const int64_t g = blockIdx.x;
  const int64_t ci = (g << (kGroupShift - kChunkShift)) + w;
  const int64_t t = (ci << kChunkShift) + lane;
  float4 c = make_float4(0.0f, 0.0f, 0.0f, -1.0f);
  if (t < n) c = rec[t];
  const float4 sc = sphere_of_spheres(c);
  if (lane == 0) {
    cs[w] = sc;
    if (sc.w >= 0.0f) chk[ci] = sc;
  }
  __syncthreads();
  if (w == 0) {
    const float4 gs = sphere_of_spheres(cs[lane]);
    if (lane == 0 && gs.w >= 0.0f) grp[g] = gs;
  }
}

// Writes up to kFillChunk scene-table entries passed by value (no host memory is read later) and
// sets their boxes of triangle centres empty.
constexpr int kFillChunk = 200;
struct GenFill {
  GenScene e[kFillChunk];
  int n;
};
__global__ void k_fill_gen_table(GenScene *dst, GenFill f, int *bbox) {
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) {
    dst[i] = f.e[i];
    for (int k = 0; k < 3; ++k) {
      bbox[8 * i + k] = 0x7fffffff;
      bbox[8 * i + 3 + k] = (int)0x80000000;
    }
  }
}

// ------------------------------------------------------------------ exclusive scan (int32)

__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = lane < nw ? warp_sums[lane] : 0;
    int wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= d) wi += y;
    }
    if (lane < nw) warp_sums[lane] = wi - w;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  int r = warp_sums[warp] + x - v;
  __syncthreads();
  return r;
}

__global__ void k_scan_partials(const int *__restrict__ in, int64_t n, int *__restrict__ partials) {
  __shared__ int ws[32];
  __shared__ int tot;
  int64_t base = (int64_t)blockIdx.x * kScanItems;
  int s = 0;
  for (int i = threadIdx.x; i < kScanItems; i += blockDim.x)
    if (base + i < n) s += in[base + i];
  block_exclusive_scan(s, ws, &tot);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

__global__ void k_scan_top(int *partials, int nb) {
  __shared__ int ws[32];
  __shared__ int tot;
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nb; base += blockDim.x) {
    int i = base + threadIdx.x;
    int v = i < nb ? partials[i] : 0;
    int ex = block_exclusive_scan(v, ws, &tot);
    if (i < nb) partials[i] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[nb] = carry;
}

__global__ void k_scan_final(const int *__restrict__ in, int64_t n, const int *__restrict__ partials,
                             int *__restrict__ out) {
  __shared__ int ws[32];
  __shared__ int tot;
  const int per = kScanItems / 256;  // blockDim.x == 256
  int64_t base = (int64_t)blockIdx.x * kScanItems + threadIdx.x * per;
  int v[per];
  int s = 0;
#pragma unroll
  for (int k = 0; k < per; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0;
    s += v[k];
  }
  int run = partials[blockIdx.x] + block_exclusive_scan(s, ws, &tot);
#pragma unroll
  for (int k = 0; k < per; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = partials[gridDim.x];
}

// ------------------------------------------------------------------ small meshes

// The whole preparation of one small scene in one block: table entry, box of centres, Morton bins,
// scan, sorted records, bounding spheres (the steps of k_tri_bbox .. k_chunk_spheres, with the
// bins in shared memory).  Nine dependent launches of a few microseconds each cost more than the
// work of up to kSmallTris triangles: 162 images of a 320-triangle mesh 62 us with them, 37 us
// with this launch and the generation's (most of it the call's host side).  One block takes 5 us per
// 1,000 triangles, so the sides meet between 5,000 (one image 60 us here, 63 us in nine launches) and
// 6,000 (66 and 63 us; 8,192: 83 and 67 us).
constexpr int kSmallTris = 5120;
constexpr int kSmallBins = 4096;  // 8^L bins in use: L <= 4 for up to 2^14 buckets
__global__ void __launch_bounds__(1024) k_sort_small(GenScene sc, GenScene *__restrict__ tab,
                                                     uint32_t *__restrict__ tb,
                                                     int *__restrict__ ts,
                                                     int *__restrict__ starts,
                                                     float4 *rec, float4 *__restrict__ chk,
                                                     float4 *__restrict__ grp, int *status) {
  __shared__ int bins[kSmallBins];
  __shared__ int bb[6];
  __shared__ int ws[32];
  __shared__ int tot;
  __shared__ float4 cs[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = (int)sc.nt;
  for (int b = tid; b < kSmallBins; b += 1024) bins[b] = 0;
  if (tid < 6) bb[tid] = tid < 3 ? 0x7fffffff : (int)0x80000000;
  if (tid == 0) *tab = sc;
  __syncthreads();
  // reads a triangle; false when it is skipped (`report`: its status bits are raised)
  auto read = [&](int t, int (&id)[3], float (&v)[9], bool report) -> bool {
    for (int k = 0; k < 3; ++k) id[k] = sc.tris[3 * (int64_t)t + k];
    if (id[0] < 0 || id[0] >= sc.nv || id[1] < 0 || id[1] >= sc.nv || id[2] < 0 || id[2] >= sc.nv) {
      if (report) set_status(status, RICI_ERR_INDEX_OUT_OF_RANGE);
      return false;
    }
    bool fin = true;
    for (int k = 0; k < 3; ++k)
      for (int d = 0; d < 3; ++d) {
        v[3 * k + d] = sc.V[3 * (int64_t)id[k] + d];
        fin = fin && isfinite(v[3 * k + d]);
      }
    if (!fin && report) set_status(status, RICI_ERR_NONFINITE_INPUT);
    return fin;
  };
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int t = tid; t < nt; t += 1024) {
    int id[3];
    float v[9];
    if (!read(t, id, v, true)) continue;
    const TriSphere s = tri_sphere(v);
    const float c[3] = {s.cx, s.cy, s.cz};
    for (int k = 0; k < 3; ++k) {
      lo[k] = fminf(lo[k], c[k]);
      hi[k] = fmaxf(hi[k], c[k]);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], d));
      hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], d));
    }
  if (lane == 0 && lo[0] <= hi[0])
    for (int k = 0; k < 3; ++k) {
      atomicMin(&bb[k], float_order(lo[k]));
      atomicMax(&bb[3 + k], float_order(hi[k]));
    }
  __syncthreads();
  for (int t = tid; t < nt; t += 1024) {
    int id[3];
    float v[9];
    uint32_t b = kSkip;
    if (read(t, id, v, false)) {
      b = morton_bin(tri_sphere(v), bb, sc.nbuckets);
      ts[t] = atomicAdd(&bins[b], 1);
    }
    tb[t] = b;
  }
  __syncthreads();
  {  // exclusive scan of the bins, 4 per thread
    int c[4], s = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c[k] = bins[4 * tid + k];
      s += c[k];
    }
    int run = block_exclusive_scan(s, ws, &tot);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      bins[4 * tid + k] = run;
      run += c[k];
    }
  }
  __syncthreads();
  const int n = tot;
  // the scene's record range: all that k_generate reads of the bin starts
  if (tid == 0) {
    starts[0] = 0;
    starts[sc.nbuckets + 1] = n;
  }
  for (int t = tid; t < nt; t += 1024) {
    const uint32_t b = tb[t];
    if (b == kSkip) continue;
    int id[3];
    float v[9];
    read(t, id, v, false);
    const TriSphere s = tri_sphere(v);
    const int64_t pos = bins[b] + ts[t];
    rec[pos] = make_float4(s.cx, s.cy, s.cz, s.r);
    rec[nt + pos] = make_float4(v[0], v[1], v[2], v[3]);
    rec[2 * (int64_t)nt + pos] = make_float4(v[4], v[5], v[6], v[7]);
    rec[3 * (int64_t)nt + pos] = make_float4(v[8], __int_as_float(id[0]), __int_as_float(id[1]),
                                             __int_as_float(id[2]));
  }
  __syncthreads();
  for (int g = 0; g * 1024 < n; ++g) {
    const int ci = g * 32 + warp, t = ci * 32 + lane;
    // written by this block before the barrier: read past the first-level cache
    const float4 c = t < n ? __ldcg(rec + t) : make_float4(0.0f, 0.0f, 0.0f, -1.0f);
    const float4 sp = sphere_of_spheres(c);
    if (lane == 0) {
      cs[warp] = sp;
      if (sp.w >= 0.0f) chk[ci] = sp;
    }
    __syncthreads();
    if (warp == 0) {
      const float4 gs = sphere_of_spheres(cs[lane]);
      if (lane == 0 && gs.w >= 0.0f) grp[g] = gs;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ generation kernel

struct KArgs {
  const GenScene *tab;
  int num_scenes;
  int64_t origin_base;  // first launch-wide origin index of this grid
  const float4 *rec;    // triangle records, 4 columns: rec[k * rs + t]
  int64_t rs;           // column stride of rec (the launch's triangle count)
  const int *starts;
  float inv_cell;
  float cell;       // grid cell edge (1 / inv_cell)
  float reach;      // support-sphere radius + largest small-triangle radius (+ margin)
  float R;
  int N;
  float alpha_cull;  // pretest radius limit (alpha_{N-1} plus margin)
  float beta_cull;   // pretest height limit (beta_{N-1} plus margin)
  int mode;
  int nhalf;        // neighbourhood half-width in cells (cell edge > reach / nhalf)
  float r_big;      // largest bounding radius of a binned triangle
  double per;       // generation: N / R, columns and layers per unit of length
  const float4 *chk;  // generation: bounding spheres of 32-record chunks of rec
  const float4 *grp;  // generation: bounding spheres of 1024-record groups of rec
  uint32_t *sort_bin;  // scratch of the sort, free afterwards: one word per triangle
  int *sort_slot;      // the same
  unsigned long long *counters;
  int *status;
};

struct Pair;
struct Shared {
  int *diff;     // [N][N + 1] difference image (the last column takes interval ends at N; the odd
                 // stride spreads equal columns of consecutive layers over the banks)
  double *a2d;   // alpha_c^2 (FP64 definition)
  double *bd;    // beta_r (FP64 definition)
  double *fr;    // S (3 doubles), Nax, Nay, Nbx, Nbz
  Pair *fp;      // the frame for layer_pairs (6 pairs)
  float4 *ff;    // gax, gay, gbx, gbz; fax, fay, N / R; S and the sphere test's margin; the axis: read
                 // where they are used, so that they hold no registers in between
  int *wq;       // this warp's candidate queue [64]
  int *bq_rec;   // this warp's band queue: triangle record [kBandQ]
  unsigned char *bq_r;  // this warp's band queue: layer [kBandQ]
  int *walk;     // this warp's place in the walk over groups: next window, window and mask left in it
  float *slots;  // this warp's staged triangles [32][kSlot]
};

// A staged triangle, in units of R / N (one column, one layer), heights Z counted in layers (layer
// r at Z = r), vertices sorted by height: 0 lowest, 1 middle, 2 highest.  Layers between 0 and 1
// cross the edges 0-2 and 0-1, layers between 1 and 2 cross 0-2 and 1-2, so both crossed edges
// start at vertex 0 for the former and at vertex 2 for the latter, and the crossing points are
// E = (x, y) + (r - Z) (slope) with the slopes dx/dZ, dy/dZ of the two edges.
enum {
  S_V0 = 0,     // x0, y0, Z0, column margin of the lower segment (see item margins below)
  S_V2 = 4,     // x2, y2, Z2, column margin of the upper segment
  S_LONG = 8,   // slope of edge 0-2, slope of edge 0-1
  S_UP = 12,    // slope of edge 1-2, first item (int), layers (int: first layer of the lower
                // segment, its layer count << 8, (first upper layer - that count) << 16)
  S_REC = 16    // triangle record (int)
};

// Adding kRound to a float of magnitude below 2^22 rounds it to an integer, held in the low bits.
constexpr float kRound = 12582912.0f;  // 1.5 * 2^23

__device__ __forceinline__ float rsqrt_fast(float x) {  // relative error below 2^-22.9
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_fast(float x) {  // at most 1 ulp off
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ int lower_count_d(double x, const double *a2d, int N) {
  // number of columns c with a2d[c] <= x (a2d strictly increasing)
  int lo = 0, hi = N;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a2d[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Eq. rotationCoefficients (second pair on the rotated x component) with the identity rule,
// in FP64 with the definition's operation order: fr = (Nax, Nay, Nbx, Nbz).
__device__ __forceinline__ void frame_fp64(float nxf, float nyf, float nzf, double *fr) {
  const double nx = nxf, ny = nyf, nz = nzf;
  const double h = __dsqrt_rn(__dadd_rn(__dmul_rn(nx, nx), __dmul_rn(ny, ny)));
  double Nax = 1.0, Nay = 0.0;
  if (h != 0.0) {
    Nax = __ddiv_rn(nx, h);
    Nay = __ddiv_rn(ny, h);
  }
  const double n2x = __dadd_rn(__dmul_rn(Nax, nx), __dmul_rn(Nay, ny));
  const double g = __dsqrt_rn(__dadd_rn(__dmul_rn(n2x, n2x), __dmul_rn(nz, nz)));
  double Nbx = 0.0, Nbz = 1.0;
  if (g != 0.0) {
    Nbx = __ddiv_rn(n2x, g);
    Nbz = __ddiv_rn(nz, g);
  }
  fr[0] = Nax;
  fr[1] = Nay;
  fr[2] = Nbx;
  fr[3] = Nbz;
}

// Eqs. relativeLocation, firstRotation, secondRotation in FP32 with explicit roundings (the
// frame coefficients rounded to FP32).  Returns |dx| + |dy| + |dz|, the scale of the error bound
// |T32 - T64| <= 10 u (|dx| + |dy| + |dz|) used by the generation kernel.
__device__ __forceinline__ float project_fp32(float px, float py, float pz, float Sx, float Sy,
                                              float Sz, float fax, float fay, float fbx,
                                              float fbz, float &tx, float &ty, float &tz) {
  const float dx = __fsub_rn(px, Sx), dy = __fsub_rn(py, Sy), dz = __fsub_rn(pz, Sz);
  const float qx = __fmaf_rn(fay, dy, __fmul_rn(fax, dx));
  const float qy = __fmaf_rn(fax, dy, -__fmul_rn(fay, dx));
  tx = __fmaf_rn(fbz, qx, -__fmul_rn(fbx, dz));
  ty = qy;
  tz = __fmaf_rn(fbx, qx, __fmul_rn(fbz, dz));
  return fabsf(dx) + fabsf(dy) + fabsf(dz);
}

// Projection of n points into one oriented point's frame with the generation kernel's FP32
// stage (one thread per point; each computes the frame).
__global__ void k_project_fp32(const float *__restrict__ pts, int64_t n, const float *__restrict__ sv,
                               const float *__restrict__ sn, float *__restrict__ out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    double fr[4];
    frame_fp64(sn[0], sn[1], sn[2], fr);
    float tx, ty, tz;
    project_fp32(pts[3 * k], pts[3 * k + 1], pts[3 * k + 2], sv[0], sv[1], sv[2],
                 __double2float_rn(fr[0]), __double2float_rn(fr[1]), __double2float_rn(fr[2]),
                 __double2float_rn(fr[3]), tx, ty, tz);
    out[3 * k] = tx;
    out[3 * k + 1] = ty;
    out[3 * k + 2] = tz;
  }
}

__device__ __forceinline__ void project64(float px, float py, float pz, const double *fr,
                                          double T[3]) {
  double dx = __dsub_rn((double)px, fr[0]);
  double dy = __dsub_rn((double)py, fr[1]);
  double dz = __dsub_rn((double)pz, fr[2]);
  const double Nax = fr[3], Nay = fr[4], Nbx = fr[5], Nbz = fr[6];
  double qx = __dadd_rn(__dmul_rn(Nax, dx), __dmul_rn(Nay, dy));
  double qy = __dadd_rn(__dmul_rn(-Nay, dx), __dmul_rn(Nax, dy));
  T[0] = __dsub_rn(__dmul_rn(Nbz, qx), __dmul_rn(Nbx, dz));
  T[1] = qy;
  T[2] = __dadd_rn(__dmul_rn(Nbx, qx), __dmul_rn(Nbz, dz));
}

// FP64 evaluation of one (triangle, layer) with the definition's operation order.
// Returns false when the triangle does not cross the layer; otherwise the single-crossing
// columns are [lo, hi) and the double-crossing columns [dlo, lo).
// (Plain pointer arguments: no structure has to live in local memory.)
__device__ __noinline__ bool layer_fp64(const float4 *__restrict__ recs, int64_t rs,
                                        const double *fr, const double *bd, const double *a2d,
                                        int N, int rec, int r, int &lo, int &hi, int &dlo) {
  float4 r1 = recs[rs + rec], r2 = recs[2 * rs + rec], r3 = recs[3 * rs + rec];
  double T[3][3];
  project64(r1.x, r1.y, r1.z, fr, T[0]);
  project64(r1.w, r2.x, r2.y, fr, T[1]);
  project64(r2.z, r2.w, r3.x, fr, T[2]);
  const int gid[3] = {__float_as_int(r3.y), __float_as_int(r3.z), __float_as_int(r3.w)};
  const double beta = bd[r];
  int s0 = T[0][2] >= beta, s1 = T[1][2] >= beta, s2 = T[2][2] >= beta;
  if (s0 == s1 && s1 == s2) return false;
  int lone = (s0 != s1 && s0 != s2) ? 0 : ((s1 != s0 && s1 != s2) ? 1 : 2);
  int oa = lone == 0 ? 1 : 0;
  int ob = lone == 2 ? 1 : 2;
  // crossed edges evaluated from the lower to the higher global vertex index
  int ua = gid[lone] < gid[oa] ? lone : oa, va = gid[lone] < gid[oa] ? oa : lone;
  int ub = gid[lone] < gid[ob] ? lone : ob, vb = gid[lone] < gid[ob] ? ob : lone;
  double la = __ddiv_rn(__dsub_rn(beta, T[ua][2]), __dsub_rn(T[va][2], T[ua][2]));
  double lb = __ddiv_rn(__dsub_rn(beta, T[ub][2]), __dsub_rn(T[vb][2], T[ub][2]));
  double Eax = __dadd_rn(T[ua][0], __dmul_rn(la, __dsub_rn(T[va][0], T[ua][0])));
  double Eay = __dadd_rn(T[ua][1], __dmul_rn(la, __dsub_rn(T[va][1], T[ua][1])));
  double Ebx = __dadd_rn(T[ub][0], __dmul_rn(lb, __dsub_rn(T[vb][0], T[ub][0])));
  double Eby = __dadd_rn(T[ub][1], __dmul_rn(lb, __dsub_rn(T[vb][1], T[ub][1])));
  bool swap = gid[ub] < gid[ua] || (gid[ub] == gid[ua] && gid[vb] < gid[va]);
  double E0x = swap ? Ebx : Eax, E0y = swap ? Eby : Eay;
  double E1x = swap ? Eax : Ebx, E1y = swap ? Eay : Eby;
  double e0 = __dadd_rn(__dmul_rn(E0x, E0x), __dmul_rn(E0y, E0y));
  double e1 = __dadd_rn(__dmul_rn(E1x, E1x), __dmul_rn(E1y, E1y));
  int c0 = lower_count_d(e0, a2d, N), c1 = lower_count_d(e1, a2d, N);
  lo = min(c0, c1);
  hi = max(c0, c1);
  dlo = lo;
  if (lo > 0) {
    double Dx = __dsub_rn(E1x, E0x), Dy = __dsub_rn(E1y, E0y);
    double d0 = __dadd_rn(__dmul_rn(E0x, Dx), __dmul_rn(E0y, Dy));
    double d1 = __dadd_rn(__dmul_rn(E1x, Dx), __dmul_rn(E1y, Dy));
    if (d0 < 0.0 && d1 > 0.0) {
      double cr = __dsub_rn(__dmul_rn(E0x, Dy), __dmul_rn(E0y, Dx));
      double dd = __dadd_rn(__dmul_rn(Dx, Dx), __dmul_rn(Dy, Dy));
      double cr2 = __dmul_rn(cr, cr);
      // first column with alpha^2 * dd > cr^2 (monotone in the column)
      int l = 0, h = lo;
      while (l < h) {
        int mid = (l + h) >> 1;
        if (__dmul_rn(a2d[mid], dd) > cr2) h = mid; else l = mid + 1;
      }
      dlo = l;
    }
  }
  return true;
}

// Column count of a distance w from the axis (in columns, at most N + 1/4): alpha_c = c + 1/2, so
// the columns with alpha_c <= w are [0, round(w)).  f is the distance to that integer: the count
// is certain for an error of w below 1/2 - |f|.
__device__ __forceinline__ int column_count(float w, float &f) {
  const float m = __fadd_rn(w, kRound);
  f = __fsub_rn(w, __fsub_rn(m, kRound));
  return __float_as_int(m) - __float_as_int(kRound);
}

// Double crossings of one segment E0, E1 (in columns): the columns [dlo, lo) below lo, the count of
// the nearer end, whose circles cross the segment twice because its closest point C to the axis
// is strictly inside it (E0.D < 0 < E1.D) and nearer than they are.  v0, v1: |E0| and |E1|, w the
// smaller, cut off at wmax = N + 1/4.  hd = 1/2 - delta with delta >= 2 x sqrt(2) dE (dE the error
// of a point's component) + the rounding of a distance.  Returns false when the test lies inside
// its error bound.
__device__ __forceinline__ bool double_columns(float E0x, float E0y, float E1x, float E1y, float v0,
                                               float v1, float w, float hd, float wmax, int lo,
                                               int &dlo) {
  dlo = lo;
  // the products E.D are known to vm 2 sqrt(2) dE + L sqrt(2) dE + 4 dE^2 + 3 u vm L, vm the larger
  // distance, L = |Dx| + |Dy|; tau is over twice that
  const float Dx = __fsub_rn(E1x, E0x), Dy = __fsub_rn(E1y, E0y);
  const float d0 = __fmaf_rn(E0x, Dx, __fmul_rn(E0y, Dy));
  const float d1 = __fmaf_rn(E1x, Dx, __fmul_rn(E1y, Dy));
  const float delta = 0.5f - hd;
  const float vm = fmaxf(v0, v1), L = fabsf(Dx) + fabsf(Dy);
  const float tau = __fmaf_rn(2.0f * delta, vm + L + 1.0f, 8.0f * kU * vm * L);
  if (lo == 0 || d0 > tau || d1 < -tau) return true;
  // C is inside, or may be.  Nothing happens if no column lies between the nearer end and C: C is at
  // least sqrt(w^2 - (l/2)^2) away, l the segment's length, so the column boundary lo - 1/2 below
  // w is out of reach when (w - delta)^2 - (lo - 1/2)^2 >= (l/2 + delta)^2, for which the test
  // below is sufficient.
  const float l2 = __fmaf_rn(Dx, Dx, __fmul_rn(Dy, Dy));
  const float fd = w - ((float)lo - 0.5f);
  if ((fd - delta) * w * 0.999f > 0.27f * l2 + 20.0f * delta * delta) return true;
  // distance of C: both ends moved by at most sqrt(2) dE, plus the rounding of the cross product,
  // the length and the root (l2 > 1e-30: the product is then no NaN that the minimum would hide)
  const float cr = __fmaf_rn(E0x, Dy, -__fmul_rn(E0y, Dx));
  float f;
  const int ch = column_count(fminf(fabsf(cr) * rsqrt_fast(l2), wmax), f);
  dlo = min(ch, lo);
  return d0 < -tau && d1 > tau && l2 > 1e-30f && l2 < 1e30f && fabsf(f) < hd - 16.0f * kU * vm;
}

// FP32 evaluation of one (triangle, layer) from its two crossing points (in columns, frame origin on
// the axis) with forward error bounds against the FP64 definition; hd as above.  Returns false when
// a predicate lies inside its bound (or hd is not a positive number); otherwise the
// single-crossing columns are [lo, hi) and the double-crossing columns [dlo, lo), each plus
// kRoundBits.  E0 and E1 may be exchanged.
constexpr int kRoundBits = 0x4B400000;  // the bits of kRound
__device__ __forceinline__ bool layer_fp32(float E0x, float E0y, float E1x, float E1y, float hd,
                                           float wmax, int &lo, int &hi, int &dlo) {
  // e is kept off zero for the reciprocal root (columns start at 1/2)
  const float e0 = __fmaf_rn(E0x, E0x, __fmaf_rn(E0y, E0y, 1e-30f));
  const float e1 = __fmaf_rn(E1x, E1x, __fmaf_rn(E1y, E1y, 1e-30f));
  const float v0 = __fmul_rn(e0, rsqrt_fast(e0)), v1 = __fmul_rn(e1, rsqrt_fast(e1));
  const float w0 = fminf(v0, wmax), w1 = fminf(v1, wmax);
  float f0, f1;
  const int c0 = column_count(w0, f0) + kRoundBits, c1 = column_count(w1, f1) + kRoundBits;
  lo = min(c0, c1);
  hi = max(c0, c1);
  dlo = lo;
  bool ok = fmaxf(fabsf(f0), fabsf(f1)) < hd;
  // Most segments have their closest point to the axis at an end, which E0.D > 0 or E1.D < 0 tells:
  // E0.E1 - |E0|^2 > 0 or E0.E1 - |E1|^2 > 0.  With both ends within vm < 4 N, |D| <= 2 vm and dE as
  // above these are known to vm 2 sqrt(2) dE + 2 vm sqrt(2) dE + 4 dE^2 + 5 u vm^2 <= 2 delta vm +
  // delta^2 + 20 u N vm; delta >= 12 u N and vm >= 1/2 (where lo > 0) make that below 5 delta vm.
  const float vm = fmaxf(v0, v1);
  const float out = __fmaf_rn(E0x, E1x, __fmul_rn(E0y, E1y)) - fminf(e0, e1);
  const bool ends = out > vm * __fmaf_rn(-10.0f, hd, 5.0f) && vm < 4.0f * wmax - 1.0f;
  if (!ends && lo > kRoundBits) {
    ok = double_columns(E0x, E0y, E1x, E1y, v0, v1, fminf(w0, w1), hd, wmax, lo - kRoundBits, dlo) &&
         ok;
    dlo += kRoundBits;
  }
  return ok;
}

// ---- pairs of floats: h + l with |l| <= u |h|.  Each operation's error is below kUU times the sum
// of its operands' (a product's: its own) magnitudes.
struct Pair {
  float h, l;
};
constexpr float kUU = 5.6843418860808015e-14f;  // 2^-44 = 16 u^2

__device__ __forceinline__ Pair pair_norm(float s, float e) {  // |s| >= |e|
  const float h = __fadd_rn(s, e);
  return Pair{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ Pair two_sum(float a, float b) {  // exact (Knuth)
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair operator-(Pair a) { return Pair{-a.h, -a.l}; }
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
  const Pair s = two_sum(a.h, b.h);
  return pair_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Pair operator-(Pair a, Pair b) { return a + (-b); }
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.h, b.h, -p);  // exact
  return pair_norm(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, e)));
}
__device__ __forceinline__ Pair operator/(Pair n, Pair d) {
  const float rc = rcp_fast(d.h), q = __fmul_rn(n.h, rc);
  const float r = __fadd_rn(__fmaf_rn(-q, d.h, n.h), __fmaf_rn(-q, d.l, n.l));
  return pair_norm(q, __fmul_rn(r, rc));
}
__device__ __forceinline__ Pair to_pair(double x) {
  const float h = __double2float_rn(x);
  return Pair{h, __double2float_rn(x - (double)h)};
}

// Evaluation of one (triangle, layer) with pairs of floats, by the steps of the FP32 path with kUU
// in the place of u.  fp: Nax, Nay, then Nax, Nay, Nbx, Nbz scaled by perd = N / R, as pairs.
// Returns 0: no crossing, 1: intervals valid, 2: a predicate lies inside its error bound.
// Band items that would take about 110 FP64 operations at 1/64 of the FP32 rate take about 600 FP32
// operations here, and about one in 10^4 of them is left to FP64.
__device__ __forceinline__ int layer_pairs(const float4 *__restrict__ recs, int64_t rs,
                                           const float *S, const Pair *fp, float perd, int N,
                                           int rec, int r, int &lo, int &hi, int &dlo) {
  const float4 r1 = recs[rs + rec], r2 = recs[2 * rs + rec], r3 = recs[3 * rs + rec];
  const float P[9] = {r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w, r3.x};
  Pair X[3], Y[3], H[3];  // H: height above the layer
  float M = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Pair dx = two_sum(P[3 * k], -S[0]), dy = two_sum(P[3 * k + 1], -S[1]),
               dz = two_sum(P[3 * k + 2], -S[2]);
    const Pair qx = fp[0] * dx + fp[1] * dy;
    X[k] = fp[5] * qx - fp[4] * dz;
    Y[k] = fp[2] * dy - fp[3] * dx;
    H[k] = (fp[4] * qx + fp[5] * dz) + Pair{0.5f * (float)(N - 1) - (float)r, 0.0f};
    M = fmaxf(M, fabsf(dx.h) + fabsf(dy.h) + fabsf(dz.h));
  }
  const float dT = 10.1f * kUU * M * perd + 2.0f * kUU * (float)N + 1e-37f;
  const float dside = kSafety * (dT + kUU * (float)N);
  if (!(fminf(fminf(fabsf(H[0].h), fabsf(H[1].h)), fabsf(H[2].h)) > dside)) return 2;
  const bool s0 = H[0].h > 0.0f, s1 = H[1].h > 0.0f, s2 = H[2].h > 0.0f;
  if (s0 == s1 && s1 == s2) return 0;
  // the vertex alone on its side to place 0
  const bool m1 = s1 != s0 && s1 != s2, m2 = s2 != s0 && s2 != s1;
  auto to_front = [](bool b, Pair &p, Pair &q) {
    const Pair t = p;
    p.h = b ? q.h : p.h;
    p.l = b ? q.l : p.l;
    q.h = b ? t.h : q.h;
    q.l = b ? t.l : q.l;
  };
  to_front(m1, X[0], X[1]);
  to_front(m1, Y[0], Y[1]);
  to_front(m1, H[0], H[1]);
  to_front(m2, X[0], X[2]);
  to_front(m2, Y[0], Y[2]);
  to_front(m2, H[0], H[2]);
  float mag = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) mag = fmaxf(mag, fmaxf(fabsf(X[k].h), fabsf(Y[k].h)));
  Pair Ex[2], Ey[2];
  float v[2], w[2], dE = 0.0f, magE = 0.0f;
  int c[2];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const Pair den = H[k + 1] - H[0], dx = X[k + 1] - X[0], dy = Y[k + 1] - Y[0];
    const float ad = fabsf(den.h), ext = fmaxf(fabsf(dx.h), fabsf(dy.h));
    ok = ok && ad > 40.0f * dT;
    const Pair lam = -H[0] / den;
    Ex[k] = X[0] + lam * dx;
    Ey[k] = Y[0] + lam * dy;
    const float el = 3.3f * dT * rcp_fast(ad) + 7.0f * kUU;
    const float de = 1.1f * (3.0f * dT + 4.0f * kUU * (ext + mag) + (ext + 2.0f * dT) * el);
    dE = fmaxf(dE, de);
    const Pair e = Ex[k] * Ex[k] + Ey[k] * Ey[k];
    const float A = fabsf(Ex[k].h) + fabsf(Ey[k].h) + 2.0f * de;
    const float dd = kSafety * (2.0f * A * de + 8.0f * kUU * e.h) + 1e-37f;
    const float eh = fmaxf(e.h, 1e-30f);
    v[k] = __fmul_rn(eh, rsqrt_fast(eh));
    w[k] = fminf(v[k], (float)N + 0.25f);
    float f;
    c[k] = column_count(w[k], f);
    // alpha^2 of the columns on either side of the count (exact): a wrong count fails one of the two
    const float b0 = (float)c[k] - 0.5f, b1 = (float)c[k] + 0.5f;
    ok = ok && (c[k] == 0 || __fadd_rn(__fsub_rn(e.h, __fmul_rn(b0, b0)), e.l) > dd) &&
         (c[k] >= N || __fsub_rn(__fsub_rn(__fmul_rn(b1, b1), e.h), e.l) > dd);
    magE = fmaxf(magE, fmaxf(fabsf(Ex[k].h), fabsf(Ey[k].h)));
  }
  if (!ok) return 2;
  lo = min(c[0], c[1]);
  hi = max(c[0], c[1]);
  // the double crossings decide on coarser predicates, for which the points' leading parts do
  const float hd = 0.5f - (kSafety * 1.4143f * (dE + kU * magE) + 12.0f * kU * (float)(N + 1));
  return double_columns(Ex[0].h, Ey[0].h, Ex[1].h, Ey[1].h, v[0], v[1], fminf(w[0], w[1]), hd,
                        (float)N + 0.25f, lo, dlo)
             ? 1
             : 2;
}

// One (triangle, layer) that FP32 could not decide, or every one of the reference mode: pairs of
// floats, then the FP64 definition.  Bits 0-7: 1 when the triangle crosses the layer; then lo, hi,
// dlo (at most 128).  Called, not inlined: few warps are in here at a time, and the batch code
// stays small.
__device__ __noinline__ unsigned band_item(const float4 *__restrict__ recs, int64_t rs,
                                           const double *fr, const Pair *fp, const double *bd,
                                           const double *a2d, float perd, int N, bool fp64_only,
                                           int rec, int r) {
  int lo = 0, hi = 0, dlo = 0, res = 2;
  if (!fp64_only) {
    const float S[3] = {(float)fr[0], (float)fr[1], (float)fr[2]};
    res = layer_pairs(recs, rs, S, fp, perd, N, rec, r, lo, hi, dlo);
  }
  if (res == 2) res = layer_fp64(recs, rs, fr, bd, a2d, N, rec, r, lo, hi, dlo);
  return (unsigned)res | ((unsigned)lo << 8) | ((unsigned)hi << 16) | ((unsigned)dlo << 24);
}

__device__ __forceinline__ void red_shared(uint32_t addr, int v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Adds the intervals to a row of the difference image at shared address `row`.
__device__ __forceinline__ void add_intervals(uint32_t row, int lo, int hi, int dlo) {
  if (lo < hi) {
    red_shared(row + 4u * (unsigned)lo, 1);
    red_shared(row + 4u * (unsigned)hi, -1);
  }
  if (dlo < lo) {
    red_shared(row + 4u * (unsigned)dlo, 2);
    red_shared(row + 4u * (unsigned)lo, -2);
  }
}

// Candidate ranges of the grid cells around an oriented point, for every thread of the block:
// the (2 nhalf + 1)^3 cells around the spin vertex's cell (cell edge > reach / nhalf).  A
// triangle binned in a cell (by its bounding-sphere centre, radius <= r_big) can reach the
// support volume only if the cell's box lies within `reach` of the spin vertex and the box's
// bounding sphere lies within r_big of the support cylinder (axis along the normal); other
// cells are skipped, and cells that hash to an already listed bucket are listed once.  On
// return entry i <= nneigh (the last one is the scene's big list) holds the candidate range
// [buckets[i], bdup[i]) (empty for skipped entries).  Ends with a block barrier.
__device__ __forceinline__ void neighbour_ranges(const KArgs &a, int64_t bucket_off,
                                                 uint32_t nbuckets, float Sx, float Sy, float Sz,
                                                 float nxf, float nyf, float nzf, int *buckets,
                                                 int *bdup, int tid, int nthreads) {
  const int nw_ = 2 * a.nhalf + 1, nneigh = nw_ * nw_ * nw_;
  float ux = 0.0f, uy = 0.0f, uz = 1.0f;  // axis direction (identity rule for a zero normal)
  {
    const float n2 = nxf * nxf + nyf * nyf + nzf * nzf;
    if (n2 > 1e-30f) {
      const float inv = rsqrtf(n2);
      ux = nxf * inv;
      uy = nyf * inv;
      uz = nzf * inv;
    }
  }
  for (int cidx = tid; cidx < nneigh; cidx += nthreads) {
    const int ix = cell_coord(Sx, a.inv_cell) + cidx % nw_ - a.nhalf;
    const int iy = cell_coord(Sy, a.inv_cell) + (cidx / nw_) % nw_ - a.nhalf;
    const int iz = cell_coord(Sz, a.inv_cell) + cidx / (nw_ * nw_) - a.nhalf;
    const float c = a.cell;
    const float gx = fmaxf(fmaxf((float)ix * c - Sx, Sx - (float)(ix + 1) * c), 0.0f);
    const float gy = fmaxf(fmaxf((float)iy * c - Sy, Sy - (float)(iy + 1) * c), 0.0f);
    const float gz = fmaxf(fmaxf((float)iz * c - Sz, Sz - (float)(iz + 1) * c), 0.0f);
    // box centre relative to the spin vertex, its axial and radial distances to the axis
    const float hb = 0.8660254f * c * 1.001f + 1e-3f * c;  // half diagonal (+ cell rounding)
    const float cx = ((float)ix + 0.5f) * c - Sx, cy = ((float)iy + 0.5f) * c - Sy,
                cz = ((float)iz + 0.5f) * c - Sz;
    const float ax = fabsf(cx * ux + cy * uy + cz * uz);
    const float rad2 = cx * cx + cy * cy + cz * cz - ax * ax;
    const float marg = hb + a.r_big + 1e-3f * a.reach + 1e-5f * (fabsf(cx) + fabsf(cy) + fabsf(cz));
    const float rl = a.alpha_cull + marg;
    const bool near = gx * gx + gy * gy + gz * gz <= a.reach * a.reach &&
                      ax <= a.beta_cull + marg && rad2 <= rl * rl;
    buckets[cidx] = near ? (int)(bucket_off + cell_hash(ix, iy, iz, nbuckets - 1)) : -1;
  }
  if (tid == 0) buckets[nneigh] = (int)(bucket_off + nbuckets);  // the scene's big list
  __syncthreads();
  for (int cidx = tid; cidx < nneigh; cidx += nthreads) {
    const int b = buckets[cidx];
    bool dup = b < 0;
    for (int k = 0; k < cidx && !dup; ++k) dup = buckets[k] == b;
    bdup[cidx] = dup ? 1 : 0;
  }
  if (tid == 0) bdup[nneigh] = 0;
  __syncthreads();
  // candidate range of every listed bucket, fetched once per block
  for (int cidx = tid; cidx <= nneigh; cidx += nthreads) {
    int beg = 0, end = 0;
    if (!bdup[cidx]) {
      const int b = buckets[cidx];
      beg = a.starts[b];
      end = a.starts[b + 1];
    }
    buckets[cidx] = beg;
    bdup[cidx] = end;
  }
  __syncthreads();
}

// One oriented point.  Bound by instruction issue and, behind it, by the latency of each warp's
// chain from records to items (75 % issue-active at R = 0.6 on the 5M-triangle scene, 28 warps per
// SM), so the layout buys few instructions per (triangle, layer) item and many resident warps:
//  - the set-up sorts a triangle's vertices by height and works in columns and layers (R / N), so an
//    item is one base vertex, two slopes and one margin (three 16-byte loads, 4 fused
//    multiply-adds), a column count is one rounding, and its margin test one comparison;
//  - what is read once per batch or chunk (frame, spin vertex, walk over the groups) stays in shared
//    memory: 72 registers, 7 blocks of 4 warps per SM at N = 64 (5, 6, 7 blocks 306, 281, 265 ms for
//    one set of 32,768 points at R = 0.6; 64 registers for 8 blocks spill: 284 ms);
//  - undecided items go to pairs of floats, not to FP64: 0.6 % of the items, at FP64's 1/64 rate
//    1/6 of the time before.
// One set of inputs (another differs by a quarter), against edge selection, table lookups and a dozen
// margin tests per item and band items in FP64: 32,768 points of a 5M-triangle scene at R = 0.6 553 ->
// 256 ms; 131,072 at R = 0.15 170 -> 73.8 ms; every point of a 189k-triangle scene at R = 0.3 33.5 ->
// 15.0 ms.
template <int NW, bool kCount>
__global__ void __launch_bounds__(NW * 32, NW == 4 ? 7 : 3) k_generate(KArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = a.N, NS = N + 1;  // NS: row stride of the difference image
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t o = blockIdx.x;
  Shared s;
  {
    unsigned char *p = smem;
    s.diff = reinterpret_cast<int *>(p);
    p += ((size_t)N * NS * 4 + 15) & ~(size_t)15;
    s.a2d = reinterpret_cast<double *>(p);
    s.bd = s.a2d + N;
    s.fr = s.bd + N;
    s.fp = reinterpret_cast<Pair *>(s.fr + 8);
    s.ff = reinterpret_cast<float4 *>(s.fp + 6);
    int *wbase = reinterpret_cast<int *>(s.ff + 4);
    s.wq = wbase + warp * kPerWarp;
    s.bq_rec = s.wq + 64;
    s.bq_r = reinterpret_cast<unsigned char *>(s.bq_rec + kBandQ);
    s.walk = s.bq_rec + kBandQ + kBandQ / 4;
    s.slots = reinterpret_cast<float *>(s.walk + 4);
  }

  const int64_t og = a.origin_base + o;  // launch-wide origin index
  const GenScene &sc = a.tab[scene_of_origin(a.tab, a.num_scenes, og)];
  const int64_t ol = og - sc.origin_off;  // origin index within its scene
  const int vid = sc.origins[ol];
  if (vid < 0 || vid >= sc.nv) {
    if (tid == 0) set_status(a.status, RICI_ERR_INDEX_OUT_OF_RANGE);
    return;
  }
  const float Sx = sc.V[3 * (int64_t)vid], Sy = sc.V[3 * (int64_t)vid + 1],
              Sz = sc.V[3 * (int64_t)vid + 2];
  const float nxf = sc.Nrm[3 * (int64_t)vid], nyf = sc.Nrm[3 * (int64_t)vid + 1],
              nzf = sc.Nrm[3 * (int64_t)vid + 2];
  const int64_t bucket_off = sc.bucket_off;
  const uint32_t nbuckets = sc.nbuckets;
  if (!(isfinite(Sx) && isfinite(Sy) && isfinite(Sz) && isfinite(nxf) && isfinite(nyf) &&
        isfinite(nzf))) {
    if (tid == 0) set_status(a.status, RICI_ERR_NONFINITE_INPUT);
    return;
  }

  for (int i = tid; i < N * NS; i += NW * 32) s.diff[i] = 0;
  const double Rd = (double)a.R;
  for (int i = tid; i < N; i += NW * 32) {
    const double al = __ddiv_rn(__dmul_rn(Rd, (double)(2 * i + 1)), (double)(2 * N));
    s.a2d[i] = __dmul_rn(al, al);
    s.bd[i] = __ddiv_rn(__dmul_rn(Rd, (double)(2 * i + 1 - N)), (double)(2 * N));
  }
  // The frame is one thread's chain in FP64 while the block waits, so its steps that do not depend on
  // each other go to lanes, and N / R comes from the host: 200,000 points of a mesh of 50 triangles
  // 3.38 -> 3.05 ms at N = 1, 2.89 -> 2.61 ms at N = 64.
  if (warp == 0) {
    if (lane == 0) {
      s.fr[0] = Sx;
      s.fr[1] = Sy;
      s.fr[2] = Sz;
      frame_fp64(nxf, nyf, nzf, s.fr + 3);
    }
    __syncwarp();
    // lanes 0-5: Nax, Nay, then Nax, Nay, Nbx, Nbz scaled to columns and layers
    if (lane < 6) s.fp[lane] = to_pair(s.fr[lane < 2 ? 3 + lane : 1 + lane] * (lane < 2 ? 1.0 : a.per));
    __syncwarp();
    if (lane == 0) {
      // frame coefficients of the FP32 path, and those scaled to columns and layers
      s.ff[0] = make_float4(s.fp[2].h, s.fp[3].h, s.fp[4].h, s.fp[5].h);
      s.ff[1] = make_float4(s.fp[0].h, s.fp[1].h, __double2float_rn(a.per), 0.0f);
      s.ff[2] = make_float4(Sx, Sy, Sz, 4e-7f * (fabsf(Sx) + fabsf(Sy) + fabsf(Sz)));
      // central axis in world coordinates
      const float fbx = __double2float_rn(s.fr[5]), fbz = __double2float_rn(s.fr[6]);
      s.ff[3] = make_float4(fbx * s.fp[0].h, fbx * s.fp[1].h, fbz, 0.0f);
    }
  }
  __syncthreads();

  const float R = a.R;
  const float zmid = 0.5f * (float)(N - 1);  // height of the spin vertex in layers
  const float wmax = (float)N + 0.25f;       // distances beyond the last column
  const uint32_t diff_at = static_cast<uint32_t>(__cvta_generic_to_shared(s.diff));
  const bool fp64_only = a.mode == RICI_GEN_FP64;

  // (per lane and block; a lane sees each of its block's items once, fewer than 2^32)
  unsigned n_tri = 0, n_items = 0, n_band = 0, n_cand = 0;
  int qn = 0;  // warp-uniform candidate queue length
  int bn = 0;  // warp-uniform band queue length

  // warp collective: queue an item for re-evaluation where `add`
  auto push_band = [&](bool add, int rec, int r) {
    const unsigned bal = __ballot_sync(0xffffffffu, add);
    if (add) {
      const int pos = bn + __popc(bal & ((1u << lane) - 1u));
      s.bq_rec[pos] = rec;
      s.bq_r[pos] = (unsigned char)r;
      if (kCount) ++n_band;
    }
    bn += __popc(bal);
  };

  auto evaluate_band = [&](int rec, int r) {
    const unsigned v =
        band_item(a.rec, a.rs, s.fr, s.fp, s.bd, s.a2d, s.ff[1].z, N, fp64_only, rec, r);
    if (v & 0xffu)
      add_intervals(diff_at + 4u * (unsigned)(r * NS), (v >> 8) & 0xff, (v >> 16) & 0xff, v >> 24);
  };
  // Processes the first cnt queued candidates; up to 31 items may be left in the band queue.
  auto process_batch = [&](int cnt) {
    // ---- per-triangle setup: one survivor per lane
    int nlow = 0, nup = 0;            // layers certainly inside the lower and the upper segment
    int rlow = 0, rup = 0;            // the first of each
    int rec = 0;
    int a0 = 0, a1 = 0, a2 = 0;       // first layer not certainly below vertex 0, 1, 2
    int b0 = -1, b1 = -1, b2 = -1;    // last layer not certainly above it
    float4 v0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), v2 = v0, sl = v0;
    float2 su = make_float2(0.0f, 0.0f);
    if (lane < cnt) {
      rec = s.wq[lane];
      const float4 r1 = a.rec[a.rs + rec], r2 = a.rec[2 * a.rs + rec], r3 = a.rec[3 * a.rs + rec];
      const float P[9] = {r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w, r3.x};
      const float4 fg = s.ff[0], fa = s.ff[1], S = s.ff[2];
      const float gax = fg.x, gay = fg.y, gbx = fg.z, gbz = fg.w, fax = fa.x, fay = fa.y;
      float x[3], y[3], z[3], M = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float dx = __fsub_rn(P[3 * k], S.x), dy = __fsub_rn(P[3 * k + 1], S.y),
                    dz = __fsub_rn(P[3 * k + 2], S.z);
        const float qx = __fmaf_rn(fay, dy, __fmul_rn(fax, dx));
        x[k] = __fmaf_rn(gbz, qx, -__fmul_rn(gbx, dz));
        y[k] = __fmaf_rn(gax, dy, -__fmul_rn(gay, dx));
        z[k] = __fmaf_rn(gbx, qx, __fmaf_rn(gbz, dz, zmid));
        M = fmaxf(M, fabsf(dx) + fabsf(dy) + fabsf(dz));
      }
      // |T32 - T64| <= dT for every coordinate, in columns (first-order bound 7 u M per unit, 10 u M
      // with slack; the height's offset adds u N)
      const float dT = 10.01f * kU * M * fa.z + kU * (float)N + 1e-37f;
      const float xl = fminf(fminf(x[0], x[1]), x[2]), xh = fmaxf(fmaxf(x[0], x[1]), x[2]);
      const float yl = fminf(fminf(y[0], y[1]), y[2]), yh = fmaxf(fmaxf(y[0], y[1]), y[2]);
      const float gx = fmaxf(0.0f, fmaxf(xl, -xh)), gy = fmaxf(0.0f, fmaxf(yl, -yh));
      const float lim = ((float)N - 0.5f) * (1.0f + 1.0f / 4096.0f) + 2.0f * dT;
      if (!(gx * gx + gy * gy > lim * lim)) {
        auto order = [&](int i, int j) {  // the lower of vertices i, j to place i
          const bool sw = z[j] < z[i];
          const float tx = x[i], ty = y[i], tz = z[i];
          x[i] = sw ? x[j] : tx;
          y[i] = sw ? y[j] : ty;
          z[i] = sw ? z[j] : tz;
          x[j] = sw ? tx : x[j];
          y[j] = sw ? ty : y[j];
          z[j] = sw ? tz : z[j];
        };
        order(0, 1);
        order(1, 2);
        order(0, 1);
        // a layer within dside of a vertex has an uncertain side (conversions saturate)
        const float dside = kSafety * (dT + 4.0f * kU * (float)N);
        a0 = __float2int_ru(z[0] - dside);
        b0 = min(__float2int_rd(z[0] + dside), N);
        a1 = __float2int_ru(z[1] - dside);
        b1 = min(__float2int_rd(z[1] + dside), N);
        a2 = __float2int_ru(z[2] - dside);
        b2 = min(__float2int_rd(z[2] + dside), N);
        if (fp64_only || !(dside < 0.25f)) {
          // every layer it may cross goes to the band queue, through items without a margin
          const bool known = dside < 1e30f;
          rlow = known ? max(a0, 0) : 0;
          nlow = max(min(known ? b2 : N - 1, N - 1) - rlow + 1, 0);
          rup = nlow;
          v0.w = -1.0f;
          a0 = a1 = a2 = 0;
          b0 = b1 = b2 = -1;
        } else {
          rlow = max(b0, -1) + 1;
          nlow = max(min(a1, N) - rlow, 0);
          rup = max(b1, -1) + 1;
          nup = max(min(a2, N) - rup, 0);
          // Per-edge bound on |E32 - E64| per component.  E = T_u + (r - Z_u) slope; the slope's
          // relative error is that of 1 / (Z_v - Z_u) (heights off by dT each, at most 1/20 of the
          // difference, else the edge's items go to FP64), of the difference x_v - x_u and three
          // roundings; with lambda = (r - Z_u) / (Z_v - Z_u) in [0, 1]:
          //   dE <= 1.1 (3 dT + u (ext + mag) + (ext + 2 dT) el),  el <= 3.3 dT / |Z_v - Z_u| + 7 u,
          // ext = max(|x_v - x_u|, |y_v - y_u|), mag the largest coordinate (u mag <= dT / 10).
          const float d01x = x[1] - x[0], d01y = y[1] - y[0], h01 = z[1] - z[0];
          const float d02x = x[2] - x[0], d02y = y[2] - y[0], h02 = z[2] - z[0];
          const float d12x = x[2] - x[1], d12y = y[2] - y[1], h12 = z[2] - z[1];
          auto slope = [&](float dx, float dy, float h, float &sx, float &sy) -> float {
            const float inv = rcp_fast(h);
            sx = __fmul_rn(dx, inv);
            sy = __fmul_rn(dy, inv);
            const float steep = fmaxf(fabsf(sx), fabsf(sy)), ext = fmaxf(fabsf(dx), fabsf(dy));
            return h > 40.0f * dT ? dT * (3.9f + 3.7f * steep) + 9.0f * kU * ext
                                  : __int_as_float(0x7f800000);
          };
          const float de02 = slope(d02x, d02y, h02, sl.x, sl.y);
          const float de01 = slope(d01x, d01y, h01, sl.z, sl.w);
          const float de12 = slope(d12x, d12y, h12, su.x, su.y);
          // margin of an item's distances |E| <= N + 1/4: sqrt(2) dE with the safety factor, and
          // the rounding of |E| (below 5 u N) with slack; hd = 1/2 - delta
          const float round_n = 12.0f * kU * (float)(N + 1);
          v0 = make_float4(x[0], y[0], z[0],
                           0.5f - (kSafety * 1.4143f * fmaxf(de02, de01) + round_n));
          v2 = make_float4(x[2], y[2], z[2],
                           0.5f - (kSafety * 1.4143f * fmaxf(de02, de12) + round_n));
        }
      }
    }
    // ---- stage the triangles that have items, without gaps, and lay out their items in a row
    const int nlay = nlow + nup;
    const unsigned has = __ballot_sync(0xffffffffu, nlay > 0);
    int incl = nlay;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const int first = nlay > 0 ? incl - nlay : 0x7fffffff;
    if (nlay > 0) {
      if (kCount) ++n_tri;
      float4 *t4 = reinterpret_cast<float4 *>(s.slots + __popc(has & ((1u << lane) - 1u)) * kSlot);
      t4[S_V0 / 4] = v0;
      t4[S_V2 / 4] = v2;
      t4[S_LONG / 4] = sl;
      t4[S_UP / 4] = make_float4(su.x, su.y, __int_as_float(first),
                                 __int_as_float(rlow | (nlow << 8) | ((rup - nlow) << 16)));
      reinterpret_cast<int *>(t4)[S_REC] = rec;
    }
    // ---- layers whose side is uncertain for a vertex, each once
    if (__any_sync(0xffffffffu, a0 <= b0 || a1 <= b1 || a2 <= b2)) {
      const bool e0 = a0 <= b0 && a0 >= 0 && a0 < N;
      const bool e1 = a1 <= b1 && a1 >= 0 && a1 < N && !(a0 <= b0 && a1 == a0);
      const bool e2 = a2 <= b2 && a2 >= 0 && a2 < N && !(a1 <= b1 && a2 == a1);
      push_band(e0, rec, a0);
      push_band(e1, rec, a1);
      push_band(e2, rec, a2);
      if (kCount) n_items += (int)e0 + (int)e1 + (int)e2;
    }
    __syncwarp();
    // ---- the items, 32 at a time: an item's triangle is the last one that starts at or before it
    int started = 0;  // triangles that started in earlier windows
    for (int base = 0;;) {
      if (bn >= 32) {
        // re-evaluate queued band items, one per lane
        evaluate_band(s.bq_rec[lane], s.bq_r[lane]);
        __syncwarp();
        bn -= 32;
        for (int q = 0; q < bn; q += 32) {  // the rest moves down (to entries already read)
          const int mr = q + lane < bn ? s.bq_rec[32 + q + lane] : 0;
          const int ml = q + lane < bn ? s.bq_r[32 + q + lane] : 0;
          __syncwarp();
          if (q + lane < bn) {
            s.bq_rec[q + lane] = mr;
            s.bq_r[q + lane] = (unsigned char)ml;
          }
          __syncwarp();
        }
        continue;
      }
      if (base >= total) break;
      const int d = first - base;
      const unsigned starts = __reduce_or_sync(0xffffffffu, (unsigned)d < 32u ? 1u << d : 0u);
      const int owner = started + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
      started += __popc(starts);
      const int it = base + lane;
      bool band = false;
      int r = 0;
      const float *ts = s.slots + owner * kSlot;
      if (it < total) {
        const float4 up4 = *reinterpret_cast<const float4 *>(ts + S_UP);
        const float4 lg4 = *reinterpret_cast<const float4 *>(ts + S_LONG);
        const int k = it - __float_as_int(up4.z);
        const unsigned meta = __float_as_uint(up4.w);
        const bool up = k >= (int)((meta >> 8) & 0xffu);
        r = k + (int)(up ? meta >> 16 : meta & 0xffu);
        const float4 v = *reinterpret_cast<const float4 *>(ts + (up ? S_V2 : S_V0));
        const float h = __fsub_rn((float)r, v.z);
        const float E0x = __fmaf_rn(h, lg4.x, v.x), E0y = __fmaf_rn(h, lg4.y, v.y);
        const float E1x = __fmaf_rn(h, up ? up4.x : lg4.z, v.x);
        const float E1y = __fmaf_rn(h, up ? up4.y : lg4.w, v.y);
        int lo, hi, dlo;
        band = !layer_fp32(E0x, E0y, E1x, E1y, v.w, wmax, lo, hi, dlo);
        if (!band)
          add_intervals(diff_at - 4u * (unsigned)kRoundBits + 4u * (unsigned)(r * NS), lo, hi, dlo);
        if (kCount) ++n_items;
      }
      // items inside the error band wait in the queue (evaluated 32 at a time)
      if (__any_sync(0xffffffffu, band)) {
        push_band(band, band ? __float_as_int(ts[S_REC]) : 0, r);
        __syncwarp();
      }
      base += 32;
    }
    __syncwarp();
  };

  // ---- candidate triangles: the records of this point's scene, culled by the bounding spheres of
  // their 1024-record groups, then of the 32-record chunks of passing groups, then one by one.  A
  // sphere containing the bounding spheres of its records fails its test only if every record
  // fails the record test: the record test widened by the sphere's radius, with a margin that
  // covers the record test's own and both tests' rounding.
  auto sphere_pass = [&](const float4 c) -> bool {
    if (!(c.w < 1e30f)) return true;
    const float4 S = s.ff[2], w = s.ff[3];
    const float dx = c.x - S.x, dy = c.y - S.y, dz = c.z - S.z;
    const float z = fmaf(w.x, dx, fmaf(w.y, dy, w.z * dz));
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float m = 2e-3f * R + 2e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz) + 2.0f * c.w) + S.w;
    const float al = a.alpha_cull + c.w + m;
    return fabsf(z) <= a.beta_cull + c.w + m && d2 - z * z <= al * al;
  };
  const int rb = a.starts[bucket_off], re = a.starts[bucket_off + nbuckets + 1];
  {
    // group base + lane * NW + warp: consecutive groups (neighbours in space) go to different warps.
    // The walk below keeps its place (k0, the masks of passing groups and chunks) and hands over
    // 32 passing records at a time, so the batch code exists once.
    const int gend = re > rb ? ((re - 1) >> kGroupShift) + 1 : 0;
    if (lane == 0) {
      s.walk[0] = rb >> kGroupShift;
      s.walk[2] = 0;
    }
    __syncwarp();
    int chunk0 = 0, t = 0;  // first chunk of the current group; this lane's record of a passing chunk
    unsigned cm = 0;        // passing chunks left in the group
    bool more = false;      // t is in a chunk that passed and has not been tested
    // moves to the next passing chunk
    auto advance = [&]() {
      if (cm == 0) {
        int k0 = s.walk[0], gk = s.walk[1];
        unsigned gm = (unsigned)s.walk[2];
        do {
          while (gm == 0) {
            if (k0 >= gend) {
              more = false;
              return;
            }
            const int gi = k0 + lane * NW + warp;
            const bool gp = gi < gend && sphere_pass(a.grp[gi]);
            gm = __ballot_sync(0xffffffffu, gp);
            gk = k0;
            k0 += 32 * NW;
          }
          chunk0 = (gk + (__ffs(gm) - 1) * NW + warp) << (kGroupShift - kChunkShift);
          gm &= gm - 1;
          const int ci = chunk0 + lane;
          const bool cp = ci >= (rb >> kChunkShift) && ci <= ((re - 1) >> kChunkShift) &&
                          sphere_pass(a.chk[ci]);
          cm = __ballot_sync(0xffffffffu, cp);
        } while (cm == 0);
        __syncwarp();
        if (lane == 0) {
          s.walk[0] = k0;
          s.walk[1] = gk;
          s.walk[2] = (int)gm;
        }
        __syncwarp();
      }
      t = ((chunk0 + __ffs(cm) - 1) << kChunkShift) + lane;
      cm &= cm - 1;
      more = true;
    };
    advance();
    while (true) {
      float4 cn = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (more && t >= rb && t < re) cn = a.rec[t];
      while (more && qn < 32) {
        // the next chunk's spheres are loaded before the current ones are tested and queued, so the
        // load's latency overlaps that work
        const int tc = t;
        const float4 c = cn;
        advance();
        if (more && t >= rb && t < re) cn = a.rec[t];
        bool pass = false;
        if (tc >= rb && tc < re) {
          const float4 S = s.ff[2], w = s.ff[3];
          float dx = c.x - S.x, dy = c.y - S.y, dz = c.z - S.z;
          float z = fmaf(w.x, dx, fmaf(w.y, dy, w.z * dz));
          float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          float m = 1e-3f * R + 1e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz));
          float al = a.alpha_cull + c.w + m;
          pass = fabsf(z) <= a.beta_cull + c.w + m && d2 - z * z <= al * al;
          if (kCount) ++n_cand;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, pass);
        if (pass) s.wq[qn + __popc(bal & ((1u << lane) - 1u))] = tc;
        qn += __popc(bal);
      }
      if (qn == 0) break;
      __syncwarp();
      const int cnt = min(qn, 32);
      process_batch(cnt);
      qn -= cnt;
      const int moved = lane < qn ? s.wq[32 + lane] : 0;
      __syncwarp();
      if (lane < qn) s.wq[lane] = moved;
      __syncwarp();
    }
  }
  // what is left of the warps' band queues, shared out over the warps 32 at a time: an evaluation costs
  // a warp the same for one item as for 32 (every point of a 189k-triangle scene, 103 undecided items
  // each: 15.9 -> 15.1 ms; 131,072 points with 485: 78.2 -> 74.5 ms)
  if (lane == 0) s.walk[3] = bn;
  __syncthreads();
  {
    const int *const queue0 = s.wq - warp * kPerWarp;  // warp 0's queues
    constexpr int kQueue = 64, kLeft = 64 + kBandQ + kBandQ / 4 + 3;  // words: band queue, its length
    int total = 0;
    for (int w = 0; w < NW; ++w) total += queue0[w * kPerWarp + kLeft];
    for (int k0 = warp * 32; k0 < total; k0 += NW * 32) {
      int k = k0 + lane, w = 0;
      if (k < total) {
        while (k >= queue0[w * kPerWarp + kLeft]) k -= queue0[w++ * kPerWarp + kLeft];
        const int *const q = queue0 + w * kPerWarp + kQueue;
        evaluate_band(q[k], reinterpret_cast<const unsigned char *>(q + kBandQ)[k]);
      }
    }
  }

  if (kCount) {
    const unsigned n[4] = {n_tri, n_items, n_band, n_cand};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      unsigned long long v = n[k];
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
      if (lane == 0) atomicAdd(a.counters + k, v);
    }
  }
  __syncthreads();

  // ---- prefix-sum each row of the difference image, saturate, store uint16
  uint16_t *out = sc.out + ol * (int64_t)N * N;
  const int cpl = (N + 31) / 32;
  if ((N == 64 || N == 128) && (reinterpret_cast<uintptr_t>(out) & 7) == 0) {
    // each lane owns 2 (N = 64) or 4 (N = 128) consecutive columns and makes one 32- or 64-bit
    // store of the packed counts
    for (int r = warp; r < N; r += NW) {
      const int *row = s.diff + r * NS + cpl * lane;
      const int v0 = row[0], v1 = row[1];
      const int v2 = cpl == 4 ? row[2] : 0, v3 = cpl == 4 ? row[3] : 0;
      const int sum = v0 + v1 + v2 + v3;
      int incl = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      const int p0 = incl - sum + v0, p1 = p0 + v1, p2 = p1 + v2, p3 = p2 + v3;
      const uint32_t w0 = (uint32_t)min(max(p0, 0), 65535) | ((uint32_t)min(max(p1, 0), 65535) << 16);
      if (cpl == 2) {
        *reinterpret_cast<uint32_t *>(out + r * N + 2 * lane) = w0;
      } else {
        const uint32_t w1 =
            (uint32_t)min(max(p2, 0), 65535) | ((uint32_t)min(max(p3, 0), 65535) << 16);
        *reinterpret_cast<uint2 *>(out + r * N + 4 * lane) = make_uint2(w0, w1);
      }
    }
    return;
  }
  for (int r = warp; r < N; r += NW) {
    const int *row = s.diff + r * NS;
    const int c0 = lane * cpl, c1 = min(N, c0 + cpl);
    int sum = 0;
    for (int c = c0; c < c1; ++c) sum += row[c];
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    int run = incl - sum;
    for (int c = c0; c < c1; ++c) {
      run += row[c];
      out[r * N + c] = (uint16_t)min(max(run, 0), 65535);
    }
  }
}

size_t generate_smem_bytes(int N, int warps) {
  size_t b = ((size_t)N * (N + 1) * 4 + 15) & ~(size_t)15;
  b += (size_t)(2 * N + 8) * sizeof(double) + 6 * sizeof(Pair) + 4 * sizeof(float4);
  b += (size_t)warps * kPerWarp * 4;
  return b;
}

template <int NW>
cudaError_t launch_k_generate(const KArgs &k, int64_t total_origins, cudaStream_t st) {
  const size_t smem = generate_smem_bytes(k.N, NW);
  auto kern = k.counters ? k_generate<NW, true> : k_generate<NW, false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  for (int64_t o0 = 0; o0 < total_origins; o0 += 0x7fffffff) {
    const int64_t cnt = total_origins - o0 < 0x7fffffff ? total_origins - o0 : 0x7fffffff;
    KArgs kk = k;
    kk.origin_base = o0;
    kern<<<(unsigned)cnt, NW * 32, smem, st>>>(kk);
    count_launches(1);
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------ clutter measure
// Eq. clutter (Section 4.1): clutter = (A_all - A_object) / A_all with A_all the surface area
// inside the support volume of an oriented point and A_object the part on the object of
// interest.  The support volume is the image's cylinder: Tx^2 + Ty^2 <= R^2, |Tz| <= R/2 in the
// frame of Eqs. relativeLocation..secondRotation (a rotation, so frame areas are scene areas).

// Signed area of the triangle (0, p, q) that lies inside the disk |x| <= R (R2 = R^2), in the
// (Tx, Ty) plane.  The segment p-q is inside the disk for t in [t1, t2] (roots of
// |p + t (q - p)|^2 = R^2) and outside elsewhere; clipped to [0, 1] this gives three pieces: an
// outer piece adds the circular sector it subtends, the inner one the triangle with the origin.
__device__ double disk_wedge(double px, double py, double qx, double qy, double R2) {
  const double dx = qx - px, dy = qy - py;
  const double A = dx * dx + dy * dy;
  double ta = 1.0, tb = 1.0;  // no crossing: the whole segment is outside
  if (A > 0.0) {
    const double B = px * dx + py * dy, C = px * px + py * py - R2;
    const double disc = B * B - A * C;
    if (disc > 0.0) {
      const double sq = sqrt(disc);
      ta = fmin(fmax((-B - sq) / A, 0.0), 1.0);
      tb = fmin(fmax((-B + sq) / A, 0.0), 1.0);
    }
  }
  const double ax = px + ta * dx, ay = py + ta * dy, bx = px + tb * dx, by = py + tb * dy;
  // an outer piece never spans opposite directions (the segment between them would cross the
  // disk), so a zero cross product means an empty sector; a piece that the clipping leaves empty has
  // none either: its ends differ by rounding alone, which near the axis is any angle
  const double c0 = px * ay - py * ax, c1 = bx * qy - by * qx;
  double sectors = 0.0;
#pragma unroll 1  // (one atan2 in the code: k_clutter does not spill then)
  for (int k = 0; k < 2; ++k) {  // p .. P(ta), P(tb) .. q
    const double c = k ? c1 : c0;
    if (c != 0.0 && (k ? tb < 1.0 : ta > 0.0))
      sectors += atan2(c, k ? bx * qx + by * qy : px * ax + py * ay);
  }
  return 0.5 * R2 * sectors + 0.5 * (ax * by - ay * bx);
}

// Area of the part of one projected triangle inside the support volume: clip it to the slab
// |Tz| <= R/2, then area(projection onto (Tx, Ty) within the disk) / |cos|, cos the z component
// of the unit normal.  Planes with |cos| < 1e-7 count as parallel to the axis: the polygon is cut
// by the two lines where the plane, at its mean distance p from the axis, meets the cylinder
// (|h| <= sqrt(R^2 - p^2), h the horizontal in-plane coordinate).
__device__ double support_area64(const double T[3][3], double R) {
  const double ux = T[1][0] - T[0][0], uy = T[1][1] - T[0][1], uz = T[1][2] - T[0][2];
  const double vx = T[2][0] - T[0][0], vy = T[2][1] - T[0][1], vz = T[2][2] - T[0][2];
  const double nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
  const double nn = sqrt(nx * nx + ny * ny + nz * nz);
  if (nn == 0.0) return 0.0;
  const double H = 0.5 * R;
  // the volume is convex: a triangle whose vertices all lie in it lies in it whole
  bool whole = true;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    whole = whole && T[i][0] * T[i][0] + T[i][1] * T[i][1] <= R * R && fabs(T[i][2]) <= H;
  if (whole) return 0.5 * nn;
  // slab clip (z <= H, then -z <= H), at most 5 vertices
  double P[5][3], Q[5][3];
  int m = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int j = i == 2 ? 0 : i + 1;
    const double di = H - T[i][2], dj = H - T[j][2];
    if (di >= 0.0) {
      P[m][0] = T[i][0]; P[m][1] = T[i][1]; P[m][2] = T[i][2];
      ++m;
    }
    if ((di >= 0.0) != (dj >= 0.0)) {
      const double f = di / (di - dj);
      P[m][0] = T[i][0] + f * (T[j][0] - T[i][0]);
      P[m][1] = T[i][1] + f * (T[j][1] - T[i][1]);
      P[m][2] = T[i][2] + f * (T[j][2] - T[i][2]);
      ++m;
    }
  }
  if (m < 3) return 0.0;
  int k = 0;
  for (int i = 0; i < m; ++i) {
    const int j = i + 1 == m ? 0 : i + 1;
    const double di = H + P[i][2], dj = H + P[j][2];
    if (di >= 0.0) {
      Q[k][0] = P[i][0]; Q[k][1] = P[i][1]; Q[k][2] = P[i][2];
      ++k;
    }
    if ((di >= 0.0) != (dj >= 0.0)) {
      const double f = di / (di - dj);
      Q[k][0] = P[i][0] + f * (P[j][0] - P[i][0]);
      Q[k][1] = P[i][1] + f * (P[j][1] - P[i][1]);
      Q[k][2] = P[i][2] + f * (P[j][2] - P[i][2]);
      ++k;
    }
  }
  if (k < 3) return 0.0;
  const double cz = fabs(nz) / nn;
  if (cz >= 1e-7) {
    double a = 0.0;
    for (int i = 0; i < k; ++i) {
      const int j = i + 1 == k ? 0 : i + 1;
      a += disk_wedge(Q[i][0], Q[i][1], Q[j][0], Q[j][1], R * R);
    }
    return fabs(a) / cz;
  }
  // plane parallel to the axis: in-plane coordinates (h, z), h along (-ny, nx) / |n_xy|
  const double hxy = sqrt(nx * nx + ny * ny);
  const double ex = -ny / hxy, ey = nx / hxy;
  double p = 0.0;
  for (int i = 0; i < k; ++i) p += (Q[i][0] * nx + Q[i][1] * ny) / hxy;
  p /= (double)k;
  if (fabs(p) >= R) return 0.0;
  const double c = sqrt(R * R - p * p);
  // area of the polygon's part with |h| <= c: shoelace over the polygon clipped to the band
  double G[7][2], E[7][2];
  for (int i = 0; i < k; ++i) {
    G[i][0] = Q[i][0] * ex + Q[i][1] * ey;
    G[i][1] = Q[i][2];
  }
  int g = k;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const double sg = side == 0 ? 1.0 : -1.0;
    int e = 0;
    for (int i = 0; i < g; ++i) {
      const int j = i + 1 == g ? 0 : i + 1;
      const double di = c - sg * G[i][0], dj = c - sg * G[j][0];
      if (di >= 0.0) {
        E[e][0] = G[i][0]; E[e][1] = G[i][1];
        ++e;
      }
      if ((di >= 0.0) != (dj >= 0.0)) {
        const double f = di / (di - dj);
        E[e][0] = G[i][0] + f * (G[j][0] - G[i][0]);
        E[e][1] = G[i][1] + f * (G[j][1] - G[i][1]);
        ++e;
      }
    }
    for (int i = 0; i < e; ++i) {
      G[i][0] = E[i][0];
      G[i][1] = E[i][1];
    }
    g = e;
  }
  if (g < 3) return 0.0;
  double a = 0.0;
  for (int i = 0; i < g; ++i) {
    const int j = i + 1 == g ? 0 : i + 1;
    a += G[i][0] * G[j][1] - G[j][0] * G[i][1];
  }
  return 0.5 * fabs(a);
}

// World-frame area of sorted record t (FP64; projections keep it), as two 32-bit halves.
__device__ __forceinline__ void store_area(const KArgs &a, int64_t t, uint32_t *area_hi,
                                           int *area_lo) {
  const float4 r1 = a.rec[a.rs + t], r2 = a.rec[2 * a.rs + t], r3 = a.rec[3 * a.rs + t];
  const double ux = (double)r1.w - r1.x, uy = (double)r2.x - r1.y, uz = (double)r2.y - r1.z;
  const double vx = (double)r2.z - r1.x, vy = (double)r2.w - r1.y, vz = (double)r3.x - r1.z;
  const double nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
  const double ar = 0.5 * sqrt(nx * nx + ny * ny + nz * nz);
  area_hi[t] = (uint32_t)__double2hiint(ar);
  area_lo[t] = __double2loint(ar);
}

// The area of every record (*nrec of them).  FP64 bounds it: 64 us for 1M triangles.
__global__ void k_tri_area(KArgs a, const int *__restrict__ nrec, uint32_t *__restrict__ area_hi,
                           int *__restrict__ area_lo) {
  const int64_t n = *nrec;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    store_area(a, t, area_hi, area_lo);
}

// The areas that few oriented points can ask for: none of a group of 1024 records, or of a chunk of 32
// of them, that the walk of no point in k_clutter reaches (its bounds, over all directions of the
// axis).  One block per group, the group's points to shared memory, one warp per chunk.
// Taken for at most kAreaPoints points (one pass of a block) in kAreaTris triangles or more, where the
// areas left out take longer than the tests.  One point in 1M triangles (a shell of radius 1) at R = 0.05:
// the call took 220 us on the hashed grid that came before this sort, 367 us with every area and the
// box's atomics of all warps, 206 us so; 1,000 points at R = 0.01 in 3M triangles 628, 1,080, 629 us.
constexpr int64_t kAreaPoints = 1024, kAreaTris = 1 << 17;
__global__ void __launch_bounds__(1024) k_tri_area_near(KArgs a, const int *__restrict__ nrec,
                                                        int num_origins,
                                                        uint32_t *__restrict__ area_hi,
                                                        int *__restrict__ area_lo) {
  __shared__ float near[kAreaPoints][3];
  __shared__ int count;
  const int64_t n = *nrec, t0 = blockIdx.x * (int64_t)1024;
  if (t0 >= n) return;  // (uniform over the block)
  const GenScene &sc = a.tab[0];
  auto reached = [&](const float4 c, float Sx, float Sy, float Sz) -> bool {  // (sphere_pass there)
    if (!(c.w < 1e30f)) return true;
    const float dx = c.x - Sx, dy = c.y - Sy, dz = c.z - Sz;
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float m = 2e-3f * a.R + 2e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz) + 2.0f * c.w) +
                    4e-7f * (fabsf(Sx) + fabsf(Sy) + fabsf(Sz));
    const float al = a.alpha_cull + c.w + m, be = a.beta_cull + c.w + m;
    return d2 <= 1.0001f * (al * al + be * be);
  };
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  if ((int)threadIdx.x < num_origins) {
    const int vid = sc.origins[threadIdx.x];
    if (vid >= 0 && vid < sc.nv) {
      const float *S = sc.V + 3 * (int64_t)vid;
      if (reached(a.grp[blockIdx.x], S[0], S[1], S[2])) {
        float *const p = near[atomicAdd(&count, 1)];
        p[0] = S[0];
        p[1] = S[1];
        p[2] = S[2];
      }
    }
  }
  __syncthreads();
  const int64_t t = t0 + threadIdx.x;
  if ((t & ~(int64_t)31) >= n) return;  // (uniform over the warp)
  const float4 c = a.chk[t >> kChunkShift];
  bool hit = false;
  for (int o = threadIdx.x & 31; o < count && !hit; o += 32)
    hit = reached(c, near[o][0], near[o][1], near[o][2]);
  if (__any_sync(0xffffffffu, hit) && t < n) store_area(a, t, area_hi, area_lo);
}

// Share of a triangle's area at heights in [-H, H], from its vertices' heights.  The slab is closed: a
// triangle that lies in an end plane is inside.
__device__ double slab_share(double z0, double z1, double z2, double H) {
  const double lo = fmin(z0, fmin(z1, z2)), hi = fmax(z0, fmax(z1, z2));
  const double mid = fmax(fmin(z0, z1), fmin(fmax(z0, z1), z2));
  // share below a height between lo and hi: quadratic on either side of the middle vertex
  auto below = [&](double h) -> double {
    const double d = h <= mid ? h - lo : hi - h;
    const double f = d * d / ((h <= mid ? mid - lo : hi - mid) * (hi - lo));
    return h <= mid ? f : 1.0 - f;
  };
  const double upper = H >= hi ? 1.0 : (H <= lo ? 0.0 : below(H));
  const double lower = -H <= lo ? 0.0 : (-H >= hi ? 1.0 : below(-H));
  return upper - lower;
}

// Area within the disk |x| <= R of the projection (onto (Tx, Ty)) of a triangle inside the slab,
// signed by its orientation: disk_wedge of its three edges, with one atan2.  An outer piece from p
// to q subtends the argument of (p.q, p x q); the pieces' arguments add up to the argument of the
// product, up to a multiple of 2 pi that their single-precision sum tells.  FP64 runs at 1/64 of
// the FP32 rate here and an atan2 is about 60 of its operations, so six of them cost more than all
// the rest.
__device__ double disk_area(const double T[3][3], double R2) {
  double sum = 0.0, zr = 1.0, zi = 0.0;
  float th = 0.0f;
  auto sector = [&](double px, double py, double qx, double qy) {
    const double c = px * qy - py * qx;
    if (c == 0.0) return;  // (as in disk_wedge: an empty sector)
    const double d = px * qx + py * qy;
    // by a power of two, so that the product stays near 1
    const int e = __double2hiint(fmax(fabs(c), fabs(d))) & 0x7ff00000;
    const double k = __hiloint2double(0x7fe00000 - max(e, 0x00100000), 0);
    const double cr = c * k, dr = d * k;
    th += atan2f((float)cr, (float)dr);
    const double t = zr * dr - zi * cr;
    zi = zr * cr + zi * dr;
    zr = t;
  };
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    const double px = i == 0 ? T[0][0] : (i == 1 ? T[1][0] : T[2][0]);
    const double py = i == 0 ? T[0][1] : (i == 1 ? T[1][1] : T[2][1]);
    const double qx = i == 0 ? T[1][0] : (i == 1 ? T[2][0] : T[0][0]);
    const double qy = i == 0 ? T[1][1] : (i == 1 ? T[2][1] : T[0][1]);
    const double dx = qx - px, dy = qy - py;
    const double A = dx * dx + dy * dy;
    double ta = 1.0, tb = 1.0;  // no crossing: the whole segment is outside
    if (A > 0.0) {
      const double B = px * dx + py * dy, C = px * px + py * py - R2;
      const double disc = B * B - A * C;
      if (disc > 0.0) {
        const double sq = sqrt(disc), inv = 1.0 / A;
        ta = fmin(fmax((-B - sq) * inv, 0.0), 1.0);
        tb = fmin(fmax((-B + sq) * inv, 0.0), 1.0);
      }
    }
    const double ax = px + ta * dx, ay = py + ta * dy, bx = px + tb * dx, by = py + tb * dy;
    if (ta > 0.0) sector(px, py, ax, ay);
    if (tb < 1.0) sector(bx, by, qx, qy);
    sum += ax * by - ay * bx;
  }
  double theta = 0.0;
  if (zi != 0.0 || zr < 0.0) theta = atan2(zi, zr);
  theta += 6.283185307179586476925 * (double)rintf((th - (float)theta) * 0.15915494f);
  return 0.5 * (R2 * theta + sum);
}

constexpr int kClutterWarps = 4;
constexpr int kSpinMaxCells = 7 * 7 * 7 + 1;  // spin images: neighbourhoods of nhalf <= 3, + the big list

// One block per oriented point: the records of its scene, culled by the sphere hierarchy with the
// limits of the full cylinder as in k_generate, queue per warp.  A projection in FP32 with its
// error bound then sorts them:
//   outside the volume (above, below or beside it): nothing;
//   inside: the triangle's area (k_tri_area), no FP64 beyond the sum;
//   certainly within the radius, not certainly between the planes: its area times the share of it
//     between them (slab_share);
//   certainly between the planes, not within the radius: disk_area over the plane's tilt;
//   neither: the general clipping (support_area64).
// The last three queue apart, so that a warp's lanes run one of the FP64 paths together; what is
// left at the end is shared out over the block's warps.  A triangle belongs to the object when
// its first vertex index is below object_vertices.
// FP64 (1/64 of the FP32 rate) bounds it, 64 % of the pipe's cycles, behind it the block's last barrier
// and instruction fetches: before, every candidate was projected in FP64 and every triangle not wholly
// inside was clipped with up to six atan2.  10,242 points, 189k triangles, R = 0.3: 18.3 -> 5.8 ms.
__global__ void __launch_bounds__(kClutterWarps * 32, 5)
    k_clutter(KArgs a, const uint32_t *__restrict__ area_hi, const int *__restrict__ area_lo,
              int64_t object_vertices, double *__restrict__ out_all, double *__restrict__ out_obj,
              double *__restrict__ out_clutter) {
  __shared__ double fr[7];
  __shared__ int wq[kClutterWarps][64];
  __shared__ int cq[3][kClutterWarps][64];  // records waiting for an FP64 path
  __shared__ int cq_n[3][kClutterWarps];
  __shared__ double part[kClutterWarps][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t og = a.origin_base + blockIdx.x;
  const GenScene &sc = a.tab[scene_of_origin(a.tab, a.num_scenes, og)];
  const int vid = sc.origins[og - sc.origin_off];
  if (vid < 0 || vid >= sc.nv) {
    if (tid == 0) {
      set_status(a.status, RICI_ERR_INDEX_OUT_OF_RANGE);
      out_all[og] = out_obj[og] = nan("");
      if (out_clutter) out_clutter[og] = nan("");
    }
    return;
  }
  const float Sx = sc.V[3 * (int64_t)vid], Sy = sc.V[3 * (int64_t)vid + 1],
              Sz = sc.V[3 * (int64_t)vid + 2];
  const float nxf = sc.Nrm[3 * (int64_t)vid], nyf = sc.Nrm[3 * (int64_t)vid + 1],
              nzf = sc.Nrm[3 * (int64_t)vid + 2];
  if (!(isfinite(Sx) && isfinite(Sy) && isfinite(Sz) && isfinite(nxf) && isfinite(nyf) &&
        isfinite(nzf))) {
    if (tid == 0) {
      set_status(a.status, RICI_ERR_NONFINITE_INPUT);
      out_all[og] = out_obj[og] = nan("");
      if (out_clutter) out_clutter[og] = nan("");
    }
    return;
  }
  if (tid == 0) {
    fr[0] = Sx;
    fr[1] = Sy;
    fr[2] = Sz;
    frame_fp64(nxf, nyf, nzf, fr + 3);
  }
  __syncthreads();
  const float fax = __double2float_rn(fr[3]), fay = __double2float_rn(fr[4]);
  const float fbx = __double2float_rn(fr[5]), fbz = __double2float_rn(fr[6]);
  const float wx = fbx * fax, wy = fbx * fay, wz = fbz;  // central axis in world coordinates
  const float R = a.R, H = 0.5f * R;
  double acc_all = 0.0, acc_obj = 0.0;
  int qn = 0;                 // warp-uniform candidate queue length
  int cn[3] = {0, 0, 0};      // warp-uniform lengths of the FP64 queues
  auto add = [&](double ar, bool obj) {
    acc_all += ar;
    if (obj) acc_obj += ar;
  };
  auto area_of = [&](int r) { return __hiloint2double((int)area_hi[r], area_lo[r]); };
  // one record through FP64 path c
  auto evaluate = [&](int c, int r) {
    const float4 r1 = a.rec[a.rs + r], r2 = a.rec[2 * a.rs + r], r3 = a.rec[3 * a.rs + r];
    double T[3][3];
    project64(r1.x, r1.y, r1.z, fr, T[0]);
    project64(r1.w, r2.x, r2.y, fr, T[1]);
    project64(r2.z, r2.w, r3.x, fr, T[2]);
    double ar;
    const double nz = (T[1][0] - T[0][0]) * (T[2][1] - T[0][1]) -
                      (T[1][1] - T[0][1]) * (T[2][0] - T[0][0]);
    const double whole2 = 2.0 * area_of(r);  // the normal's length
    if (c == 0) {
      ar = 0.5 * whole2 * slab_share(T[0][2], T[1][2], T[2][2], 0.5 * (double)R);
    } else if (c == 1 && fabs(nz) >= 1e-7 * whole2 && whole2 > 0.0) {
      ar = fabs(disk_area(T, (double)R * R)) * (whole2 / fabs(nz));
    } else {
      ar = support_area64(T, R);
    }
    add(ar, __float_as_int(r3.y) < object_vertices);
  };
  auto process = [&](int cnt) {
    int cls = -1, r = 0;  // FP64 path
    if (lane < cnt) {
      r = wq[warp][lane];
      const float4 r1 = a.rec[a.rs + r], r2 = a.rec[2 * a.rs + r], r3 = a.rec[3 * a.rs + r];
      float x[3], y[3], z[3], M = 0.0f;
      M = fmaxf(M, project_fp32(r1.x, r1.y, r1.z, Sx, Sy, Sz, fax, fay, fbx, fbz, x[0], y[0], z[0]));
      M = fmaxf(M, project_fp32(r1.w, r2.x, r2.y, Sx, Sy, Sz, fax, fay, fbx, fbz, x[1], y[1], z[1]));
      M = fmaxf(M, project_fp32(r2.z, r2.w, r3.x, Sx, Sy, Sz, fax, fay, fbx, fbz, x[2], y[2], z[2]));
      // |T32 - T64| <= 10 u M per coordinate; m covers it, and the rounding of the tests below at
      // distances near R (8 u R), with the safety factor
      const float dT = 10.0f * kU * M + 1e-37f;
      const float m = kSafety * (1.4143f * dT + 8.0f * kU * R);
      const float zl = fminf(fminf(z[0], z[1]), z[2]), zh = fmaxf(fmaxf(z[0], z[1]), z[2]);
      const float rin = R - m, rout = R + m;
      float d2 = 0.0f;
#pragma unroll
      for (int k = 0; k < 3; ++k) d2 = fmaxf(d2, fmaf(x[k], x[k], y[k] * y[k]));
      const bool in_slab = zl >= m - H && zh <= H - m;
      const bool in_disk = rin > 0.0f && d2 <= rin * rin;
      bool out = zl > H + m || zh < -H - m;
      const float gx = fmaxf(0.0f, fmaxf(fminf(fminf(x[0], x[1]), x[2]), -fmaxf(fmaxf(x[0], x[1]), x[2])));
      const float gy = fmaxf(0.0f, fmaxf(fminf(fminf(y[0], y[1]), y[2]), -fmaxf(fmaxf(y[0], y[1]), y[2])));
      out = out || gx * gx + gy * gy > rout * rout;
      // beside the volume: the axis lies more than R beyond an edge, seen from the triangle
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int j = k == 2 ? 0 : k + 1, i = 3 - k - j;  // i: the vertex opposite edge k-j
        const float dx = x[j] - x[k], dy = y[j] - y[k];
        const float c = x[k] * y[j] - y[k] * x[j];        // twice the area of (axis, k, j)
        const float len = sqrtf(dx * dx + dy * dy);
        const float err = 4.0f * dT * (fabsf(x[k]) + fabsf(y[k]) + fabsf(x[j]) + fabsf(y[j]) + 2.0f * dT) +
                          8.0f * kU * (fabsf(x[k] * y[j]) + fabsf(y[k] * x[j]));
        // vertex i certainly across the edge's line from the axis: all of the triangle is at least as
        // far from it as the line is
        const float ori = (x[i] - x[k]) * dy - (y[i] - y[k]) * dx;
        const float eori = 8.0f * dT * (fabsf(dx) + fabsf(dy) + fabsf(x[i] - x[k]) + fabsf(y[i] - y[k])) +
                           8.0f * kU * (fabsf((x[i] - x[k]) * dy) + fabsf((y[i] - y[k]) * dx));
        out = out || (fabsf(c) > rout * len * 1.0001f + err && fabsf(ori) > eori &&
                      (ori > 0.0f) == (c > 0.0f));
      }
      if (!out) {
        if (in_slab && in_disk) add(area_of(r), __float_as_int(r3.y) < object_vertices);
        else cls = in_disk ? 0 : (in_slab ? 1 : 2);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const unsigned bal = __ballot_sync(0xffffffffu, cls == c);
      if (cls == c) cq[c][warp][cn[c] + __popc(bal & ((1u << lane) - 1u))] = r;
      cn[c] += __popc(bal);
    }
    __syncwarp();
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
      const int have = c == 0 ? cn[0] : (c == 1 ? cn[1] : cn[2]);
      if (have < 32) continue;
      const int first = cq[c][warp][lane];
      const int moved = lane < have - 32 ? cq[c][warp][32 + lane] : 0;
      __syncwarp();
      if (lane < have - 32) cq[c][warp][lane] = moved;
      if (c == 0) cn[0] -= 32;
      if (c == 1) cn[1] -= 32;
      if (c == 2) cn[2] -= 32;
      __syncwarp();
      evaluate(c, first);
    }
  };
  const float mpos = 4e-7f * (fabsf(Sx) + fabsf(Sy) + fabsf(Sz));
  auto sphere_pass = [&](const float4 c) -> bool {  // as in k_generate
    if (!(c.w < 1e30f)) return true;
    const float dx = c.x - Sx, dy = c.y - Sy, dz = c.z - Sz;
    const float z = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float m = 2e-3f * R + 2e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz) + 2.0f * c.w) + mpos;
    const float al = a.alpha_cull + c.w + m;
    return fabsf(z) <= a.beta_cull + c.w + m && d2 - z * z <= al * al;
  };
  const int rb = a.starts[sc.bucket_off], re = a.starts[sc.bucket_off + sc.nbuckets + 1];
  const int gend = re > rb ? ((re - 1) >> kGroupShift) + 1 : 0;
  for (int k0 = rb >> kGroupShift; k0 < gend; k0 += 32 * kClutterWarps) {
    const int gi = k0 + lane * kClutterWarps + warp;
    const bool gp = gi < gend && sphere_pass(a.grp[gi]);
    unsigned gm = __ballot_sync(0xffffffffu, gp);
    while (gm) {
      const int chunk0 = (k0 + (__ffs(gm) - 1) * kClutterWarps + warp) << (kGroupShift - kChunkShift);
      gm &= gm - 1;
      const int ci = chunk0 + lane;
      const bool cp = ci >= (rb >> kChunkShift) && ci <= ((re - 1) >> kChunkShift) &&
                      sphere_pass(a.chk[ci]);
      unsigned cm = __ballot_sync(0xffffffffu, cp);
      while (cm) {
        const int t = ((chunk0 + __ffs(cm) - 1) << kChunkShift) + lane;
        cm &= cm - 1;
        bool pass = false;
        if (t >= rb && t < re) {
          const float4 c = a.rec[t];
          const float dx = c.x - Sx, dy = c.y - Sy, dz = c.z - Sz;
          const float z = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
          const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          const float mg = 1e-3f * R + 1e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz));
          const float al = a.alpha_cull + c.w + mg;
          pass = fabsf(z) <= a.beta_cull + c.w + mg && d2 - z * z <= al * al;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, pass);
        if (pass) wq[warp][qn + __popc(bal & ((1u << lane) - 1u))] = t;
        qn += __popc(bal);
        const bool end = !cm && !gm && k0 + 32 * kClutterWarps >= gend;
        __syncwarp();
        while (qn >= 32 || (end && qn > 0)) {
          const int n = min(qn, 32);
          process(n);
          qn -= n;
          const int moved = lane < qn ? wq[warp][32 + lane] : 0;
          __syncwarp();
          if (lane < qn) wq[warp][lane] = moved;
          __syncwarp();
        }
      }
    }
  }
  if (qn > 0) process(qn);  // (the last group or chunk did not pass)
  // what is left of the FP64 queues, over all warps
  if (lane < 3) cq_n[lane][warp] = lane == 0 ? cn[0] : (lane == 1 ? cn[1] : cn[2]);
  __syncthreads();
#pragma unroll 1
  for (int c = 0; c < 3; ++c) {
    int total = 0;
    for (int w = 0; w < kClutterWarps; ++w) total += cq_n[c][w];
    int k = ((warp + c) % kClutterWarps) * 32 + lane;  // at most 31 of each warp: one item per thread
    if (k < total) {
      int w = 0;
      while (k >= cq_n[c][w]) k -= cq_n[c][w++];
      evaluate(c, cq[c][w][k]);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    acc_all += __shfl_down_sync(0xffffffffu, acc_all, d);
    acc_obj += __shfl_down_sync(0xffffffffu, acc_obj, d);
  }
  if (lane == 0) {
    part[warp][0] = acc_all;
    part[warp][1] = acc_obj;
  }
  __syncthreads();
  if (tid == 0) {
    double sa = 0.0, so = 0.0;
    for (int w = 0; w < kClutterWarps; ++w) {
      sa += part[w][0];
      so += part[w][1];
    }
    out_all[og] = sa;
    out_obj[og] = so;
    // Eq. clutter: the share of the area inside the support volume not on the object
    if (out_clutter) out_clutter[og] = sa > 0.0 ? __ddiv_rn(__dsub_rn(sa, so), sa) : nan("");
  }
}

// ------------------------------------------------------------------ spin images
// Spin images (Section 2.1) from point samples of the mesh, with the FP32 projection stage of
// the generation kernel (Eqs. relativeLocation..secondRotation, frame rounded from FP64).
// Samples: m^2 per triangle at the centroids of the m^2 congruent sub-triangles of a division of
// every side into m parts, P = A + a (B - A) + b (C - A) with barycentric (a, b) = ((3i+1)/3m,
// (3j+1)/3m) for the upward sub-triangles (i + j <= m - 1) and ((3i+2)/3m, (3j+2)/3m) for the
// downward ones (i + j <= m - 2).  The plane is R wide and R high with the spin vertex at half
// height, N x N bins centred at alpha_c = (c + 1/2) R/N and beta_r = (r + 1/2 - N/2) R/N; a
// sample with alpha^2 < R^2 and -R/2 <= beta < R/2 adds bilinear weights to the four bins around
// it (weight on a bin outside the image is dropped).  Weights are formed in FP32 with explicit
// roundings and summed exactly as integers in units of 2^-24 (w * 2^24 rounded to the nearest
// integer) in shared memory, so the sums do not depend on the order of the samples; the image
// stores float32(sum * 2^-24).
constexpr int kSpinWarps = 4;
constexpr int kSpinMaxSide = 16;  // samples per triangle <= 256

__global__ void __launch_bounds__(kSpinWarps * 32) k_spin(KArgs a, int m, float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char spin_smem[];
  __shared__ int buckets[kSpinMaxCells], bdup[kSpinMaxCells];
  __shared__ double fr[7];
  __shared__ float smp_a[kSpinMaxSide * kSpinMaxSide], smp_b[kSpinMaxSide * kSpinMaxSide];
  __shared__ int wq[kSpinWarps][64];
  const int N = a.N;
  unsigned long long *img = reinterpret_cast<unsigned long long *>(spin_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t og = a.origin_base + blockIdx.x;
  const GenScene &sc = a.tab[scene_of_origin(a.tab, a.num_scenes, og)];
  float *dst = out + og * (int64_t)N * N;
  const int vid = sc.origins[og - sc.origin_off];
  bool bad = vid < 0 || vid >= sc.nv;
  float Sx = 0.0f, Sy = 0.0f, Sz = 0.0f, nxf = 0.0f, nyf = 0.0f, nzf = 1.0f;
  if (!bad) {
    Sx = sc.V[3 * (int64_t)vid];
    Sy = sc.V[3 * (int64_t)vid + 1];
    Sz = sc.V[3 * (int64_t)vid + 2];
    nxf = sc.Nrm[3 * (int64_t)vid];
    nyf = sc.Nrm[3 * (int64_t)vid + 1];
    nzf = sc.Nrm[3 * (int64_t)vid + 2];
  }
  const bool nonfinite = !bad && !(isfinite(Sx) && isfinite(Sy) && isfinite(Sz) &&
                                   isfinite(nxf) && isfinite(nyf) && isfinite(nzf));
  if (bad || nonfinite) {
    if (tid == 0)
      set_status(a.status, bad ? RICI_ERR_INDEX_OUT_OF_RANGE : RICI_ERR_NONFINITE_INPUT);
    for (int i = tid; i < N * N; i += kSpinWarps * 32) dst[i] = 0.0f;
    return;
  }
  for (int i = tid; i < N * N; i += kSpinWarps * 32) img[i] = 0ull;
  if (tid == 0) {
    fr[0] = Sx;
    fr[1] = Sy;
    fr[2] = Sz;
    frame_fp64(nxf, nyf, nzf, fr + 3);
    // sample table: upward sub-triangles row by row, then the downward ones
    const float den = (float)(3 * m);
    int k = 0;
    for (int i = 0; i < m; ++i)
      for (int j = 0; i + j <= m - 1; ++j, ++k) {
        smp_a[k] = __fdiv_rn((float)(3 * i + 1), den);
        smp_b[k] = __fdiv_rn((float)(3 * j + 1), den);
      }
    for (int i = 0; i + 1 < m; ++i)
      for (int j = 0; i + j <= m - 2; ++j, ++k) {
        smp_a[k] = __fdiv_rn((float)(3 * i + 2), den);
        smp_b[k] = __fdiv_rn((float)(3 * j + 2), den);
      }
  }
  neighbour_ranges(a, sc.bucket_off, sc.nbuckets, Sx, Sy, Sz, nxf, nyf, nzf, buckets, bdup, tid,
                   kSpinWarps * 32);
  const float fax = __double2float_rn(fr[3]), fay = __double2float_rn(fr[4]);
  const float fbx = __double2float_rn(fr[5]), fbz = __double2float_rn(fr[6]);
  const float wx = fbx * fax, wy = fbx * fay, wz = fbz;  // central axis in world coordinates
  const float R = a.R, R2 = __fmul_rn(R, R), H = __fmul_rn(0.5f, R);
  const float scale = __fdiv_rn((float)N, R);
  const int ns = m * m;
  int qn = 0;
  auto process = [&](int cnt) {
    if (lane < cnt) {
      const int64_t r = wq[warp][lane];
      const float4 r1 = a.rec[a.rs + r], r2 = a.rec[2 * a.rs + r], r3 = a.rec[3 * a.rs + r];
      const float A[3] = {r1.x, r1.y, r1.z}, B[3] = {r1.w, r2.x, r2.y}, C[3] = {r2.z, r2.w, r3.x};
      const float ba[3] = {__fsub_rn(B[0], A[0]), __fsub_rn(B[1], A[1]), __fsub_rn(B[2], A[2])};
      const float ca[3] = {__fsub_rn(C[0], A[0]), __fsub_rn(C[1], A[1]), __fsub_rn(C[2], A[2])};
      for (int k = 0; k < ns; ++k) {
        const float sa = smp_a[k], sb = smp_b[k];
        const float px = __fmaf_rn(sb, ca[0], __fmaf_rn(sa, ba[0], A[0]));
        const float py = __fmaf_rn(sb, ca[1], __fmaf_rn(sa, ba[1], A[1]));
        const float pz = __fmaf_rn(sb, ca[2], __fmaf_rn(sa, ba[2], A[2]));
        float tx, ty, tz;
        project_fp32(px, py, pz, Sx, Sy, Sz, fax, fay, fbx, fbz, tx, ty, tz);
        const float a2 = __fmaf_rn(tx, tx, __fmul_rn(ty, ty));
        if (!(a2 < R2) || !(tz >= -H) || !(tz < H)) continue;
        const float u = __fmaf_rn(__fsqrt_rn(a2), scale, -0.5f);
        const float v = __fmaf_rn(__fadd_rn(tz, H), scale, -0.5f);
        const float cu = floorf(u), rv = floorf(v);
        const float fu = __fsub_rn(u, cu), fv = __fsub_rn(v, rv);
        const float gu = __fsub_rn(1.0f, fu), gv = __fsub_rn(1.0f, fv);
        const int c = (int)cu, rr = (int)rv;
        const bool c0 = c >= 0, c1 = c + 1 < N, r0 = rr >= 0, r1_ = rr + 1 < N;
        constexpr float kUnit = 16777216.0f;  // 2^24 units per sample
        if (r0 && c0)
          atomicAdd(img + rr * N + c, __float2ull_rn(__fmul_rn(__fmul_rn(gu, gv), kUnit)));
        if (r0 && c1)
          atomicAdd(img + rr * N + c + 1, __float2ull_rn(__fmul_rn(__fmul_rn(fu, gv), kUnit)));
        if (r1_ && c0)
          atomicAdd(img + (rr + 1) * N + c, __float2ull_rn(__fmul_rn(__fmul_rn(gu, fv), kUnit)));
        if (r1_ && c1)
          atomicAdd(img + (rr + 1) * N + c + 1,
                    __float2ull_rn(__fmul_rn(__fmul_rn(fu, fv), kUnit)));
      }
    }
    __syncwarp();
  };
  const int nneigh = (2 * a.nhalf + 1) * (2 * a.nhalf + 1) * (2 * a.nhalf + 1);
  for (int nb = 0; nb <= nneigh; ++nb) {
    const int64_t beg = buckets[nb], end = bdup[nb];
    for (int64_t base = beg + warp * 32; base < end; base += kSpinWarps * 32) {
      const int64_t t = base + lane;
      bool pass = false;
      if (t < end) {
        const float4 c = a.rec[t];
        const float dx = c.x - Sx, dy = c.y - Sy, dz = c.z - Sz;
        const float z = fmaf(wx, dx, fmaf(wy, dy, wz * dz));
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float mg = 1e-3f * a.R + 1e-5f * (fabsf(dx) + fabsf(dy) + fabsf(dz));
        const float al = a.alpha_cull + c.w + mg;
        pass = fabsf(z) <= a.beta_cull + c.w + mg && d2 - z * z <= al * al;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, pass);
      if (pass) wq[warp][qn + __popc(bal & ((1u << lane) - 1u))] = (int)t;
      qn += __popc(bal);
      __syncwarp();
      if (qn >= 32) {
        process(32);
        const int rest = qn - 32;
        const int moved = lane < rest ? wq[warp][32 + lane] : 0;
        __syncwarp();
        if (lane < rest) wq[warp][lane] = moved;
        qn = rest;
        __syncwarp();
      }
    }
  }
  if (qn > 0) process(qn);
  __syncthreads();
  for (int i = tid; i < N * N; i += kSpinWarps * 32)
    dst[i] = __double2float_rn(__dmul_rn(__ull2double_rn(img[i]), 1.0 / 16777216.0));
}

}  // namespace

cudaError_t launch_project_fp32(const float *pts, int64_t n, const float *sv, const float *sn,
                                float *out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const int64_t want = (n + 255) / 256;
  k_project_fp32<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, st>>>(pts, n, sv, sn, out);
  count_launches(1);
  return cudaGetLastError();
}

// Sorts the triangles of the scenes into records: along a Morton curve with the bounding spheres of
// chunks and groups (morton: generation, clutter measure), or by the cells of a hashed grid (spin
// images), whose cells suit support volumes of radius amax and half-height bmax around each
// oriented point.  Fills the fields of k that the kernels read (table, records, starts, spheres, pretest
// limits, grid).
static cudaError_t bin_triangles(const GenScene *scenes, int num_scenes, int64_t nt, int64_t TB,
                                 double R, double amax, double bmax, void *ws, int *status,
                                 cudaStream_t st, KArgs &k, bool morton) {
  Carver c(ws);
  GenScene *tab = c.take<GenScene>(num_scenes);
  int *counts = c.take<int>(TB);
  int *starts = c.take<int>(TB + 1);
  int *partials = c.take<int>(TB / kScanItems + 2);
  uint32_t *tb = c.take<uint32_t>(nt);
  int *ts = c.take<int>(nt);
  float4 *rec = c.take<float4>(4 * nt);
  int *bbox = c.take<int>(8 * (int64_t)num_scenes);
  float4 *chk = c.take<float4>((nt + 31) / 32);
  float4 *grp = c.take<float4>((nt + 1023) / 1024);

  cudaError_t e;
  const bool small = morton && num_scenes == 1 && nt <= kSmallTris;
  for (int s0 = 0; s0 < num_scenes && !small; s0 += kFillChunk) {
    GenFill f;
    f.n = num_scenes - s0 < kFillChunk ? num_scenes - s0 : kFillChunk;
    for (int i = 0; i < f.n; ++i) f.e[i] = scenes[s0 + i];
    k_fill_gen_table<<<1, 256, 0, st>>>(tab + s0, f, bbox + 8 * (int64_t)s0);
    count_launches(1);
  }

  // enclosing sphere radius of the support cylinder
  const double rho = sqrt(amax * amax + bmax * bmax) * (1.0 + 1.0 / 1024.0) + 1e-3 * R;
  const Tuning tu = current_tuning();
  GridParams gp;
  gp.r_big = (float)(tu.gen_big_radius * rho);
  // a triangle (centre c, radius <= r_big) reaching the support volume has |c - S| <= reach;
  // with cell > reach / nhalf its cell lies within +-nhalf cells of the spin vertex's cell
  const double reach = (rho + gp.r_big) * 1.001;
  const int cpr = tu.gen_cells_per_reach < kSpinMaxCellsPerReach ? tu.gen_cells_per_reach
                                                                 : kSpinMaxCellsPerReach;
  const double cell = reach / cpr * 1.01;
  gp.inv_cell = (float)(1.0 / cell);
  gp.mask = 0;

  if (small) {
    k_sort_small<<<1, 1024, 0, st>>>(scenes[0], tab, tb, ts, starts, rec, chk, grp, status);
    count_launches(1);
  } else if ((e = cudaMemsetAsync(counts, 0, sizeof(int) * TB, st)) != cudaSuccess) {
    return e;
  }
  const int tpb = 256;
  const int64_t want = (nt + tpb - 1) / tpb;
  const int grid = (int)(want < 152 * 32 ? (want > 0 ? want : 1) : 152 * 32);
  if (nt > 0 && !small) {
    if (morton) {
      k_tri_bbox<<<grid, tpb, 0, st>>>(tab, num_scenes, nt, bbox);
      count_launches(1);
    }
    k_tri_bin<<<grid, tpb, 0, st>>>(tab, num_scenes, nt, gp, morton ? bbox : nullptr, counts, tb,
                                    ts, status);
    count_launches(1);
  }
  const int nb = (int)((TB + kScanItems - 1) / kScanItems);
  if (!small) {
    k_scan_partials<<<nb, 256, 0, st>>>(counts, TB, partials);
    k_scan_top<<<1, 1024, 0, st>>>(partials, nb);
    k_scan_final<<<nb, 256, 0, st>>>(counts, TB, partials, starts);
    count_launches(3);
  }
  if (nt > 0 && !small) {
    k_tri_scatter<<<grid, tpb, 0, st>>>(tab, num_scenes, nt, tb, ts, starts, rec);
    count_launches(1);
    if (morton) {
      k_chunk_spheres<<<(unsigned)((nt + 1023) / 1024), 1024, 0, st>>>(rec, starts + TB, chk, grp);
      count_launches(1);
    }
  }
  k.chk = chk;
  k.grp = grp;
  k.sort_bin = tb;
  k.sort_slot = ts;

  k.tab = tab;
  k.num_scenes = num_scenes;
  k.rec = rec;
  k.rs = nt;
  k.starts = starts;
  k.inv_cell = gp.inv_cell;
  k.cell = (float)cell;
  k.reach = (float)(reach + 1e-3 * cell);  // slack for the rounding of cell coordinates
  k.R = (float)R;
  k.alpha_cull = (float)(amax * (1.0 + 1.0 / 1024.0) + 1e-3 * R);
  k.beta_cull = (float)(bmax * (1.0 + 1.0 / 1024.0) + 1e-3 * R);
  k.nhalf = cpr;
  k.r_big = gp.r_big;
  k.status = status;
  return cudaSuccess;
}

cudaError_t launch_generate_batch(const GenScene *scenes, const GenerateBatch &g, void *ws,
                                  cudaStream_t st) {
  const int N = g.N;
  if (g.total_origins == 0) return cudaSuccess;
  // support cylinder: alpha <= alpha_{N-1}, |beta| <= beta_{N-1}
  const double R = g.R;
  const double amax = R * (2.0 * N - 1.0) / (2.0 * N);
  const double bmax = R * (N - 1.0) / (2.0 * N);
  KArgs k;
  cudaError_t e = bin_triangles(scenes, g.num_scenes, g.total_tris, g.total_buckets, R, amax,
                                bmax, ws, g.status, st, k, true);
  if (e != cudaSuccess) return e;
  k.nhalf = 0;  // no neighbour-cell list: candidates come from the sphere hierarchy
  k.R = g.R;
  k.N = N;
  k.per = (double)N / (double)k.R;
  k.mode = g.mode;
  k.counters = reinterpret_cast<unsigned long long *>(g.counters);
  const Tuning tu = current_tuning();
  return tu.gen_warps == 8 ? launch_k_generate<8>(k, g.total_origins, st)
                           : launch_k_generate<4>(k, g.total_origins, st);
}

cudaError_t launch_clutter(const ClutterArgs &a, void *ws, cudaStream_t st) {
  if (a.num_origins == 0) return cudaSuccess;
  GenScene sc = {};
  sc.V = a.vertices;
  sc.Nrm = a.normals;
  sc.tris = a.triangles;
  sc.origins = a.origins;
  sc.nv = a.num_vertices;
  sc.nt = a.num_triangles;
  sc.no = a.num_origins;
  sc.nbuckets = bucket_count(a.num_triangles);
  // the whole support cylinder: alpha <= R, |beta| <= R/2
  const double R = a.support_radius;
  KArgs k;
  cudaError_t e = bin_triangles(&sc, 1, a.num_triangles, (int64_t)sc.nbuckets + 1, R, R, 0.5 * R,
                                ws, a.status, st, k, true);
  if (e != cudaSuccess) return e;
  k.N = 0;
  k.mode = 0;
  k.counters = nullptr;
  // the bins and slots of the sort are free now: the records' areas take their place
  uint32_t *const area_hi = k.sort_bin;
  int *const area_lo = k.sort_slot;
  if (a.num_triangles > 0) {
    const int *const nrec = k.starts + sc.nbuckets + 1;
    if (a.num_origins <= kAreaPoints && a.num_triangles >= kAreaTris) {
      k_tri_area_near<<<(unsigned)((a.num_triangles + 1023) / 1024), 1024, 0, st>>>(
          k, nrec, (int)a.num_origins, area_hi, area_lo);
    } else {
      const int64_t want = (a.num_triangles + 255) / 256;
      k_tri_area<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), 256, 0, st>>>(k, nrec, area_hi,
                                                                               area_lo);
    }
    count_launches(1);
  }
  for (int64_t o0 = 0; o0 < a.num_origins; o0 += 0x7fffffff) {
    const int64_t cnt = a.num_origins - o0 < 0x7fffffff ? a.num_origins - o0 : 0x7fffffff;
    KArgs kk = k;
    kk.origin_base = o0;
    k_clutter<<<(unsigned)cnt, kClutterWarps * 32, 0, st>>>(kk, area_hi, area_lo,
                                                             a.object_vertices, a.out_area_all,
                                                             a.out_area_object, a.out_clutter);
    count_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_spin(const SpinArgs &a, void *ws, cudaStream_t st) {
  if (a.num_origins == 0) return cudaSuccess;
  GenScene sc = {};
  sc.V = a.vertices;
  sc.Nrm = a.normals;
  sc.tris = a.triangles;
  sc.origins = a.origins;
  sc.nv = a.num_vertices;
  sc.nt = a.num_triangles;
  sc.no = a.num_origins;
  sc.nbuckets = bucket_count(a.num_triangles);
  // the support cylinder of the plane: alpha <= R, |beta| <= R/2
  const double R = a.support_radius;
  KArgs k;
  cudaError_t e = bin_triangles(&sc, 1, a.num_triangles, (int64_t)sc.nbuckets + 1, R, R, 0.5 * R,
                                ws, a.status, st, k, false);
  if (e != cudaSuccess) return e;
  k.N = a.resolution;
  k.mode = 0;
  k.counters = nullptr;
  const size_t smem = sizeof(unsigned long long) * (size_t)a.resolution * a.resolution;
  if ((e = cudaFuncSetAttribute(k_spin, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)) != cudaSuccess)
    return e;
  for (int64_t o0 = 0; o0 < a.num_origins; o0 += 0x7fffffff) {
    const int64_t cnt = a.num_origins - o0 < 0x7fffffff ? a.num_origins - o0 : 0x7fffffff;
    KArgs kk = k;
    kk.origin_base = o0;
    k_spin<<<(unsigned)cnt, kSpinWarps * 32, smem, st>>>(kk, a.samples_side, a.out_images);
    count_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_generate(const GenerateArgs &a, void *ws, cudaStream_t st) {
  GenScene sc = {};
  sc.V = a.vertices;
  sc.Nrm = a.normals;
  sc.tris = a.triangles;
  sc.origins = a.origins;
  sc.out = a.out_images;
  sc.nv = a.num_vertices;
  sc.nt = a.num_triangles;
  sc.no = a.num_origins;
  sc.nbuckets = bucket_count(a.num_triangles);
  GenerateBatch b;
  b.num_scenes = 1;
  b.total_tris = a.num_triangles;
  b.total_origins = a.num_origins;
  b.total_buckets = (int64_t)sc.nbuckets + 1;
  b.R = a.support_radius;
  b.N = a.resolution;
  b.mode = a.mode;
  b.counters = a.counters;
  b.status = a.status;
  return launch_generate_batch(&sc, b, ws, st);
}

}  // namespace rici
