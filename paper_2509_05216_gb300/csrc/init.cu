// Point-cloud initialisation of the Gaussians on the GPU: isosurface edge
// crossings of a volume and k-nearest-neighbour scales.
//
// The paper starts 3D-GS from the isosurface of a scientific volume,
// extracted as a point cloud instead of SfM points (Method Overview).  The
// crossings are the contour filter's vertices: every grid edge whose end
// values lie on different sides of the level gives the linearly
// interpolated point, with the volume gradient (central differences,
// one-sided at the border) interpolated the same way as its normal, emitted
// in vertex order (x fastest, then y, then z; per vertex its +x, +y, +z
// edges).  One pass over the volume keeps a side bit per vertex; counting
// and placing the crossings works on those bits.  Each Gaussian's initial scale is log sqrt of the mean squared
// distance to its 3 nearest other points, found exactly with a grid: points
// are sorted by the Morton code of a fine cell (the onesweep radix sort), the
// level of the grid whose occupied cells hold a few points is picked on the
// device (points of a surface fill a small part of a volume's cells, so the
// cell size follows the occupied cells), its cells go into an open-addressing
// table, and each query examines growing cubes of cells until the third
// distance lies inside the examined radius.
#include <algorithm>
#include <cmath>

#include "gs_internal.cuh"
#include "launch.h"

namespace gs {

// ---------------------------------------------------------------- crossings

namespace {

__device__ __forceinline__ float vol_at(const IsoArgs& a, int x, int y, int z) {
  return __ldg(a.vol + ((int64_t)z * a.ny + y) * a.nx + x);
}

// Gradient of the volume at a vertex: central differences inside, one-sided
// at the border (0 along an axis of one sample).
__device__ __forceinline__ float3 vol_grad(const IsoArgs& a, int x, int y, int z) {
  float3 g;
  const int xm = max(x - 1, 0), xp = min(x + 1, a.nx - 1);
  const int ym = max(y - 1, 0), yp = min(y + 1, a.ny - 1);
  const int zm = max(z - 1, 0), zp = min(z + 1, a.nz - 1);
  g.x = xp > xm ? (vol_at(a, xp, y, z) - vol_at(a, xm, y, z)) / ((float)(xp - xm) * a.h[0]) : 0.f;
  g.y = yp > ym ? (vol_at(a, x, yp, z) - vol_at(a, x, ym, z)) / ((float)(yp - ym) * a.h[1]) : 0.f;
  g.z = zp > zm ? (vol_at(a, x, y, zp) - vol_at(a, x, y, zm)) / ((float)(zp - zm) * a.h[2]) : 0.f;
  return g;
}

constexpr int kIsoThreads = 256;
// Words per block of the counting and emitting passes: 1,024 (32,768 vertices), or
// 64 below 256 blocks of those, whose threads would take a block's crossings in a
// long chain of rounds.  Whole call with 64 / 1,024: 33^3 75 / 122 us, 33 x 512 x 40 74 / 121, 128^3
// 72 / 96, 200^3 90 / 92, 256^3 110 / 99, 512^3 491 / 245.
constexpr int kIsoMany = 1024, kIsoFew = 64;
constexpr int64_t kIsoFewBelow = 256 * kIsoMany;

// Exclusive prefix of `c` over the block (256 threads); *total = block sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t c, uint32_t* warp_tot, uint32_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t inc = c;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += y;
  }
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  uint32_t pre = 0, all = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
    pre += w < wid ? warp_tot[w] : 0u;
    all += warp_tot[w];
  }
  *total = all;
  return pre + inc - c;
}

// Remainder of a vertex index: 32-bit arithmetic where the volume allows it.
__device__ __forceinline__ int64_t vert_mod(const IsoArgs& a, int64_t v, int64_t m) {
  return a.nverts <= 0xffffffffll ? (int64_t)((uint32_t)v % (uint32_t)m) : v % m;
}

__device__ __forceinline__ uint32_t side_word(const IsoArgs& a, int64_t w) { return w < a.nwords ? a.sides[w] : 0u; }

// The 32 side bits of the vertices `off` after those of word w.
__device__ __forceinline__ uint32_t sides_at(const IsoArgs& a, int64_t w, int64_t off) {
  const int64_t q = w + (off >> 5);
  const int r = (int)(off & 31);
  const uint32_t lo = side_word(a, q);
  return r ? __funnelshift_r(lo, side_word(a, q + 1), r) : lo;
}

// Crossing +x, +y, +z edges of the 32 vertices of word w (bit b: vertex
// 32 w + b): the side bits that differ from those one vertex, row and plane
// on, where that neighbour exists.  A word may span rows and planes; bits at
// or past the last vertex are 0 on both sides.
__device__ __forceinline__ void crossing_masks(const IsoArgs& a, int64_t w, uint32_t& ex, uint32_t& ey, uint32_t& ez) {
  const uint32_t s = side_word(a, w);
  const int64_t v0 = 32 * w, plane = (int64_t)a.nx * a.ny;
  ex = s ^ __funnelshift_r(s, side_word(a, w + 1), 1);
  ey = s ^ sides_at(a, w, a.nx);
  ez = s ^ sides_at(a, w, plane);
  if (!(ex | ey | ez)) return;
  // the last vertex of a row has no +x edge
  uint32_t last = 0;
  for (int64_t p = a.nx - 1 - vert_mod(a, v0, a.nx); p < 32; p += a.nx) last |= 1u << p;
  ex &= ~last;
  // the last row of a plane has no +y edge
  uint32_t inner = 0;
  const int64_t seg = plane - a.nx;
  int64_t q = vert_mod(a, v0, plane);
  for (int64_t p = 0; p < 32;) {
    const int64_t run = min(32 - p, (q < seg ? seg : plane) - q);
    if (q < seg) inner |= (uint32_t)(((1ull << run) - 1ull) << p);
    p += run;
    q += run;
    if (q == plane) q = 0;
  }
  ey &= inner;
  // the last plane has no +z edge
  const int64_t zrem = plane * (a.nz - 1) - v0;
  ez &= zrem >= 32 ? 0xffffffffu : zrem <= 0 ? 0u : (1u << zrem) - 1u;
}

}  // namespace

// Side of the level of every vertex, one bit each: a warp reads 1,024
// consecutive samples (32 coalesced loads in flight per lane) and writes 32
// ballot words.  The only pass over the volume: bound by its 4 bytes per
// vertex; what follows reads 1/32 of that, and the volume again only at the
// crossings.  A 512^3 volume (2.5M crossings), whole call: 5.11 -> 0.24 ms
// against one thread per vertex testing its edges from the samples in every
// pass (two counts of 0.93 ms, an emission of 2.28 ms bound by its index
// divisions and idle lanes, two one-block scans of 524,288 counts).
__global__ void __launch_bounds__(256) iso_sides_kernel(IsoArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
  if (w0 >= a.nwords) return;
  float f[32];
#pragma unroll
  for (int j = 0; j < 32; j++) {
    const int64_t v = 32 * (w0 + j) + lane;
    f[j] = v < a.nverts ? __ldcs(a.vol + v) : 0.f;
  }
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < 32; j++) {
    const uint32_t m = __ballot_sync(0xffffffffu, 32 * (w0 + j) + lane < a.nverts && f[j] >= a.iso);
    mine = lane == j ? m : mine;
  }
  if (w0 + lane < a.nwords) a.sides[w0 + lane] = mine;
}

// Crossings per block of WORDS words, from the side bits alone.
template <int WORDS>
__global__ void __launch_bounds__(kIsoThreads) iso_count_kernel(IsoArgs a) {
  __shared__ uint32_t warp_tot[kIsoThreads / 32];
  uint32_t c = 0;
#pragma unroll
  for (int k = threadIdx.x; k < WORDS; k += kIsoThreads) {
    const int64_t w = (int64_t)blockIdx.x * WORDS + k;
    if (w < a.nwords) {
      uint32_t ex, ey, ez;
      crossing_masks(a, w, ex, ey, ez);
      c += __popc(ex) + __popc(ey) + __popc(ez);
    }
  }
  uint32_t tot;
  block_excl_scan(c, warp_tot, &tot);
  if (threadIdx.x == 0) a.block_counts[blockIdx.x] = tot;
}

// Points and normals of the crossings, in vertex order (per vertex +x, +y,
// +z).  The block lists its words' masks and first crossings in shared
// memory and its threads take the crossings one by one: crossing o finds its
// word by bisection over the first crossings and its vertex by bisection
// over the word's bits, so that no lane waits for words without crossings.
template <int WORDS>
__global__ void __launch_bounds__(kIsoThreads) iso_emit_kernel(IsoArgs a) {
  constexpr int kItems = WORDS > kIsoThreads ? WORDS / kIsoThreads : 1;  // words per thread (of the first WORDS threads)
  __shared__ uint32_t warp_tot[kIsoThreads / 32];
  __shared__ uint32_t s_first[WORDS];
  __shared__ uint32_t s_mask[3][WORDS];
  const int64_t word0 = (int64_t)blockIdx.x * WORDS;
  uint32_t c[kItems], sum = 0;
#pragma unroll
  for (int i = 0; i < kItems; i++) {
    const int k = threadIdx.x * kItems + i;
    uint32_t ex = 0, ey = 0, ez = 0;
    if (k < WORDS && word0 + k < a.nwords) crossing_masks(a, word0 + k, ex, ey, ez);
    if (k < WORDS) {
      s_mask[0][k] = ex;
      s_mask[1][k] = ey;
      s_mask[2][k] = ez;
    }
    c[i] = __popc(ex) + __popc(ey) + __popc(ez);
    sum += c[i];
  }
  uint32_t total;
  uint32_t run = block_excl_scan(sum, warp_tot, &total);
#pragma unroll
  for (int i = 0; i < kItems; i++) {
    if (threadIdx.x * kItems + i < WORDS) s_first[threadIdx.x * kItems + i] = run;
    run += c[i];
  }
  __syncthreads();
  const int64_t base = a.block_offsets[blockIdx.x];
  const int64_t plane = (int64_t)a.nx * a.ny;
  for (uint32_t q = threadIdx.x; q < total; q += kIsoThreads) {
    // the last word whose first crossing is at most q (words without
    // crossings share their successor's first crossing and are passed over)
    int k = 0;
#pragma unroll
    for (int step = WORDS / 2; step > 0; step >>= 1)
      if (s_first[k + step] <= q) k += step;
    const uint32_t ex = s_mask[0][k], ey = s_mask[1][k], ez = s_mask[2][k];
    uint32_t r = q - s_first[k];
    // the vertex holding the word's r-th crossing
    int b = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const uint32_t m = ((1u << step) - 1u) << b;
      const uint32_t n = __popc(ex & m) + __popc(ey & m) + __popc(ez & m);
      if (n <= r) {
        r -= n;
        b += step;
      }
    }
    const uint32_t e = ((ex >> b) & 1u) | (((ey >> b) & 1u) << 1) | (((ez >> b) & 1u) << 2);
    // direction: the r-th set bit of e
    int d = __ffs(e) - 1;
    for (; r > 0; r--) d = __ffs(e & (0xfffffffeu << d)) - 1;
    const int64_t o = base + q;
    if (o >= a.capacity) {
      atomicOr(a.status, kStatusCapacity);
      return;
    }
    const int64_t v = 32 * (word0 + k) + b;
    const int64_t vp = vert_mod(a, v, plane);
    const int z = a.nverts <= 0xffffffffll ? (int)((uint32_t)v / (uint32_t)plane) : (int)(v / plane);
    const int y = plane <= 0xffffffffll ? (int)((uint32_t)vp / (uint32_t)a.nx) : (int)(vp / a.nx);
    const int x = (int)(vp - (int64_t)y * a.nx);
    const float fa = vol_at(a, x, y, z);
    const float3 ga = vol_grad(a, x, y, z);
    const int x2 = x + (d == 0), y2 = y + (d == 1), z2 = z + (d == 2);
    const float fb = vol_at(a, x2, y2, z2);
    const float t = (a.iso - fa) / (fb - fa);
    const float3 gb = vol_grad(a, x2, y2, z2);
    float* p = a.points + 3 * o;
    p[0] = a.origin[0] + a.h[0] * ((float)x + (d == 0 ? t : 0.f));
    p[1] = a.origin[1] + a.h[1] * ((float)y + (d == 1 ? t : 0.f));
    p[2] = a.origin[2] + a.h[2] * ((float)z + (d == 2 ? t : 0.f));
    float nx = fmaf(t, gb.x - ga.x, ga.x), ny = fmaf(t, gb.y - ga.y, ga.y), nz = fmaf(t, gb.z - ga.z, ga.z);
    const float len = sqrtf(nx * nx + ny * ny + nz * nz);
    const float inv = len > 0.f ? 1.f / len : 0.f;
    float* nm = a.normals + 3 * o;
    nm[0] = nx * inv;
    nm[1] = ny * inv;
    nm[2] = len > 0.f ? nz * inv : 1.f;
  }
}

int64_t iso_words(int64_t nverts) { return (nverts + 31) / 32; }
static int iso_block_words(int64_t nverts) { return iso_words(nverts) < kIsoFewBelow ? kIsoFew : kIsoMany; }
int64_t iso_blocks(int64_t nverts) {
  const int words = iso_block_words(nverts);
  return (iso_words(nverts) + words - 1) / words;
}

void launch_iso_count(const IsoArgs& a, cudaStream_t s) {
  const int64_t warps = (a.nwords + 31) / 32;
  iso_sides_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(a);
  const unsigned blocks = (unsigned)iso_blocks(a.nverts);
  if (iso_block_words(a.nverts) == kIsoMany) iso_count_kernel<kIsoMany><<<blocks, kIsoThreads, 0, s>>>(a);
  else iso_count_kernel<kIsoFew><<<blocks, kIsoThreads, 0, s>>>(a);
}

void launch_iso_emit(const IsoArgs& a, cudaStream_t s) {
  const unsigned blocks = (unsigned)iso_blocks(a.nverts);
  if (iso_block_words(a.nverts) == kIsoMany) iso_emit_kernel<kIsoMany><<<blocks, kIsoThreads, 0, s>>>(a);
  else iso_emit_kernel<kIsoFew><<<blocks, kIsoThreads, 0, s>>>(a);
}

// ---------------------------------------------------------------- k nearest neighbours

// Per-block bounds of the (selected) points (6 floats: min xyz, max xyz), then
// one block combines them.
__global__ void __launch_bounds__(256) knn_bounds_kernel(const float* __restrict__ pts,
                                                         const int64_t* __restrict__ sel, int64_t n,
                                                         float* __restrict__ part) {
  __shared__ float red[6][8];
  float b[6] = {3.0e38f, 3.0e38f, 3.0e38f, -3.0e38f, -3.0e38f, -3.0e38f};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = sel ? sel[i] : i;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const float v = pts[3 * src + d];
      b[d] = fminf(b[d], v);
      b[3 + d] = fmaxf(b[3 + d], v);
    }
  }
#pragma unroll
  for (int d = 0; d < 6; d++) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float o = __shfl_down_sync(0xffffffffu, b[d], off);
      b[d] = d < 3 ? fminf(b[d], o) : fmaxf(b[d], o);
    }
    if ((threadIdx.x & 31) == 0) red[d][threadIdx.x >> 5] = b[d];
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int d = threadIdx.x;
    float v = red[d][0];
    for (int w = 1; w < 8; w++) v = d < 3 ? fminf(v, red[d][w]) : fmaxf(v, red[d][w]);
    part[6 * (int64_t)blockIdx.x + d] = v;
  }
}

__global__ void __launch_bounds__(192) knn_bounds_finish_kernel(const float* __restrict__ part, int nparts,
                                                                float* __restrict__ out) {
  const int d = threadIdx.x >> 5, lane = threadIdx.x & 31;  // a warp per bound
  float v = part[d];
  for (int b = lane; b < nparts; b += 32) v = d < 3 ? fminf(v, part[6 * b + d]) : fmaxf(v, part[6 * b + d]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float o = __shfl_down_sync(0xffffffffu, v, off);
    v = d < 3 ? fminf(v, o) : fmaxf(v, o);
  }
  if (lane == 0) out[d] = v;
}

namespace {

// A point's key is the Morton code of its finest cell, so that one sort orders
// the points by cell at every level l (cubes of 2^l finest cells along each
// axis), and a cell of any level is a run of the sorted points.  The finest
// cells are cubes too, 2^10 to 2^16 along the longest side of the bounding
// box: as many as 30 key bits allow, for a side of the box takes only the bits
// that its cells need.  A box with three long sides has 2^10, a flat one up to
// 2^15, a line 2^16 (a position's rounding, in finest cells, allows no more).
// With 2^10 for every box a line's finest cells hold thousands of points: 4M
// points on a line, whole call 21.5 ms (1.1 ms like this), on a ribbon 7.0 ms
// (1.2 ms).
//
// Bit order of a key: with a <= b <= c bits along the axes, the low a bits of
// all three interleaved, the next b - a of the two longer, the last of the
// longest; the bits of a level's cell are the key without its low
// min(l, a) + min(l, b) + min(l, c) ones.
constexpr int kMaxLevels = 16, kKeyBits = 30;
constexpr float kKnnMargin = 2e-3f;  // of a position in finest cells, 2^10 along the longest side

__device__ __forceinline__ uint32_t spread2(uint32_t x) {  // bit i -> bit 2 i
  x = (x | (x << 8)) & 0x00ff00ffu;
  x = (x | (x << 4)) & 0x0f0f0f0fu;
  x = (x | (x << 2)) & 0x33333333u;
  x = (x | (x << 1)) & 0x55555555u;
  return x;
}
__device__ __forceinline__ uint32_t spread3(uint32_t x) {  // bit i -> bit 3 i
  x &= 0x3ffu;
  x = (x | (x << 16)) & 0x030000ffu;
  x = (x | (x << 8)) & 0x0300f00fu;
  x = (x | (x << 4)) & 0x030c30c3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

// Key of the cell (x, y, z) of a level (coordinates in the order of a.bits).
// EVEN, here and below: the same bits along every axis, which are 10 then (the
// common box; by the general code the query takes 5 % longer there).
template <bool EVEN = false>
__device__ __forceinline__ uint32_t cell_key(const KnnArgs& a, uint32_t x, uint32_t y, uint32_t z, int level) {
  if constexpr (EVEN) return spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
  const int ba = max(a.bits[0] - level, 0), bb = max(a.bits[1] - level, 0);
  const uint32_t low = (1u << ba) - 1u;
  uint32_t k = spread3(x) | (spread3(y & low) << 1) | (spread3(z & low) << 2);
  if (a.bits[0] != a.bits[2]) {
    y >>= ba;
    z >>= ba;
    k |= (spread2(y) | (spread2(z & ((1u << (bb - ba)) - 1u)) << 1)) << (3 * ba);
    k |= (z >> (bb - ba)) << (ba + 2 * bb);
  }
  return k;
}

// Low bits of a key that a level's cells leave out.
__device__ __forceinline__ int level_shift(const KnnArgs& a, int level) {
  return min(level, a.bits[0]) + min(level, a.bits[1]) + min(level, a.bits[2]);
}

// The coarsest level at which two keys whose highest different bit is `bit` are
// of different cells.
__device__ __forceinline__ int level_of_bit(const KnnArgs& a, int bit) {
  const int ba = a.bits[0], bb = a.bits[1];
  return bit < 3 * ba ? bit / 3 : bit < ba + 2 * bb ? ba + (bit - 3 * ba) / 2 : bit - ba - bb;
}

template <bool EVEN = false>
__device__ __forceinline__ int cells_along(const KnnArgs& a, int k, int level) {
  return 1 << (EVEN ? kKeyBits / 3 - level : max(a.bits[k] - level, 0));
}

// A point's position in cells of a level, and its cell.
template <bool EVEN = false>
struct CellPos {
  float f[3];
  int c[3];
  __device__ __forceinline__ CellPos(const KnnArgs& a, float x, float y, float z, int level) {
    const float scale = 1.f / (float)(1 << level);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const int axis = EVEN ? k : a.axis[k];
      const float v = axis == 0 ? x : axis == 1 ? y : z;
      const float u = (v - a.lo[k]) * a.inv_cell;
      c[k] = min(max((int)u, 0), (1 << (EVEN ? kKeyBits / 3 : a.bits[k])) - 1) >> level;
      f[k] = u * scale;
    }
  }
};

// Margin of a position in cells of a level.
template <bool EVEN = false>
__device__ __forceinline__ float cell_margin(const KnnArgs& a, int level) {
  return EVEN ? kKnnMargin : fmaxf(kKnnMargin, a.margin / (float)(1 << level));
}

// First slot of a cell: the 8 cells of a cube of the next level share a line.
__device__ __forceinline__ uint32_t slot_of(uint32_t key, int bits) {
  return (((key >> 3) * 0x9E3779B1u) >> (35 - bits)) << 3 | (key & 7u);
}

// Table entry of a cell: its code, the first sorted point of its run and the
// run's length, 7 for longer ones.
constexpr unsigned long long kEmptySlot = ~0ull;
__device__ __forceinline__ unsigned long long cell_entry(uint32_t key, int64_t start, int64_t length) {
  return (unsigned long long)key << 34 | (unsigned long long)start << 3 | (unsigned long long)min(length, (int64_t)7);
}

// The level whose occupied cells hold kCellPoints points or more on average
// (the finest such one).  heads[l]: sorted points whose cell at level l, but
// not at l + 1, differs from their predecessor's; a level has one cell more
// than the heads at it and above.  (From 1 on the finer level made a surface's
// look-ups cheaper but left a fifth of a 4M set to the warps of the second
// kernel: 6.6 ms against 2.0 ms.)
constexpr int64_t kCellPoints = 2;
__device__ __forceinline__ int pick_level(const KnnArgs& a) {
  // (all words in flight at once; they are 0 from the coarsest level up)
  uint4 h[kMaxLevels / 4];
#pragma unroll
  for (int i = 0; i < kMaxLevels / 4; i++) h[i] = *reinterpret_cast<const uint4*>(a.heads + 4 * i);
  int64_t cells = 1;
  int level = kMaxLevels;
#pragma unroll
  for (int l = kMaxLevels - 1; l >= 0; l--) {
    const uint4 q = h[l / 4];
    cells += l % 4 == 0 ? q.x : l % 4 == 1 ? q.y : l % 4 == 2 ? q.z : q.w;
    level -= cells * kCellPoints <= a.n ? 1 : 0;  // (grows with every level: those that fit come first)
  }
  return min(level, a.bits[2]);
}

__device__ __forceinline__ const uint32_t* sorted_keys(const KnnArgs& a) {
  return (a.sort_ctrl[a.sort_passes] & 1u) ? a.keys[1] : a.keys[0];
}

// The sort's other value buffer: free after the sort.
__device__ __forceinline__ uint32_t* spare_vals(const KnnArgs& a) {
  return (a.sort_ctrl[a.sort_passes] & 1u) ? a.vals[0] : a.vals[1];
}
constexpr int kTodo = kKnnWords - 1;  // word of `heads` that counts the points left to the warps
static_assert(kTodo >= kMaxLevels, "a word per level before it");

// First sorted position in [lo, n) whose key is at least `key`.
__device__ __forceinline__ int64_t lower_bound(const uint32_t* keys, int64_t lo, int64_t n, uint64_t key) {
  int64_t hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((uint64_t)keys[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The run of sorted points of a cell of the given level (empty when no point
// lies in it).
__device__ __forceinline__ uint2 cell_run(const KnnArgs& a, const uint32_t* keys, uint32_t cell, int level) {
  const uint32_t mask = (uint32_t)((1ull << a.table_bits) - 1ull);
  for (uint32_t s = slot_of(cell, a.table_bits), probes = 0; probes <= mask; s = (s + 1) & mask, probes++) {
    const unsigned long long e = a.table[s];
    if (e == kEmptySlot) break;
    if ((uint32_t)(e >> 34) == cell) {
      const uint32_t start = (uint32_t)(e >> 3) & 0x7fffffffu, length = (uint32_t)e & 7u;
      if (length < 7u) return make_uint2(start, start + length);
      return make_uint2(start, (uint32_t)lower_bound(keys, (int64_t)start + 7, a.n, ((uint64_t)cell + 1) << level_shift(a, level)));
    }
  }
  return make_uint2(0u, 0u);
}

// Insert the squared distance of sorted point j into the sorted list of the
// three smallest.
__device__ __forceinline__ void near_point(const KnnArgs& a, int64_t j, float px, float py, float pz,
                                           float (&best)[3]) {
  const float4 q = a.sorted[j];
  const float ex = q.x - px, ey = q.y - py, ez = q.z - pz;
  const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
  if (d2 < best[2]) {
    best[2] = d2 < best[1] ? best[1] : d2;
    best[1] = d2 < best[0] ? best[0] : fminf(d2, best[1]);
    best[0] = fminf(d2, best[0]);
  }
}

// One axis of the 3^3 cells around a point's cell c (of dim cells; f: the
// point's fraction of it): per neighbour the squared distance to it (3e38
// outside the grid), less a margin for the rounding of f.  *border: distance to
// the nearer side of the cell.
struct CellAxis {
  int c;
  float gap2[3];
};
__device__ __forceinline__ CellAxis cell_axis(int c, int dim, float f, float margin, float cell, float* border) {
  CellAxis x;
  const float lo = fmaxf(f - margin, 0.f) * cell, hi = fmaxf(1.f - f - margin, 0.f) * cell;
  x.c = c;
  x.gap2[0] = c > 0 ? lo * lo * 0.999f : 3.0e38f;
  x.gap2[1] = 0.f;
  x.gap2[2] = c + 1 < dim ? hi * hi * 0.999f : 3.0e38f;
  *border = fminf(*border, fminf(f, 1.f - f));
  return x;
}

}  // namespace

__global__ void __launch_bounds__(256) knn_keys_kernel(KnnArgs a) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = a.sel ? a.sel[i] : i;
    const CellPos<> p(a, a.pts[3 * src], a.pts[3 * src + 1], a.pts[3 * src + 2], 0);
    a.keys[0][i] = cell_key(a, (uint32_t)p.c[0], (uint32_t)p.c[1], (uint32_t)p.c[2], 0);
    a.vals[0][i] = (uint32_t)i;
  }
}

// The points in sorted order (position and output index in one float4), and
// the heads per level.
__global__ void __launch_bounds__(256) knn_sorted_points_kernel(KnnArgs a) {
  __shared__ uint32_t s_heads[kMaxLevels];
  if (threadIdx.x < kMaxLevels) s_heads[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t* keys = sorted_keys(a);
  const uint32_t* vals = keys == a.keys[1] ? a.vals[1] : a.vals[0];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t o = vals[i];
    if ((int64_t)o >= a.n) continue;  // (only after a sort that gave up)
    const int64_t src = a.sel ? a.sel[o] : (int64_t)o;
    a.sorted[i] = make_float4(a.pts[3 * src], a.pts[3 * src + 1], a.pts[3 * src + 2], __uint_as_float(o));
    const uint32_t diff = i > 0 ? keys[i] ^ keys[i - 1] : 0u;
    if (diff) atomicAdd(&s_heads[min(level_of_bit(a, 31 - __clz(diff)), kMaxLevels - 1)], 1u);
  }
  __syncthreads();
  if (threadIdx.x < kMaxLevels && s_heads[threadIdx.x]) atomicAdd(a.heads + threadIdx.x, s_heads[threadIdx.x]);
}

// Insert every cell of the chosen level with its run of sorted points.
__global__ void __launch_bounds__(256) knn_table_kernel(KnnArgs a) {
  const int sh = level_shift(a, pick_level(a));
  const uint32_t* keys = sorted_keys(a);
  const uint32_t mask = (uint32_t)((1ull << a.table_bits) - 1ull);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t cell = keys[i] >> sh;
    if (i > 0 && keys[i - 1] >> sh == cell) continue;
    int length = 1;
    while (length < 7 && i + length < a.n && keys[i + length] >> sh == cell) length++;
    const unsigned long long entry = cell_entry(cell, i, length);
    for (uint32_t s = slot_of(cell, a.table_bits), probes = 0; probes <= mask; s = (s + 1) & mask, probes++)
      if (atomicCAS(a.table + s, kEmptySlot, entry) == kEmptySlot) break;
  }
}

__device__ __forceinline__ void write_scale(const KnnArgs& a, const float4& me, const float (&best)[3]) {
  float sum = 0.f;
#pragma unroll
  for (int k = 0; k < 3; k++) sum += best[k];
  const uint32_t o = __float_as_uint(me.w);
  if ((int64_t)o < a.n) a.out[o] = 0.5f * logf(fmaxf(sum / 3.f, 1e-14f));
}

// The cells around a sorted point at one level.
struct CellCube {
  CellAxis x, y, z;
  float border, margin;
  __device__ __forceinline__ CellCube(const KnnArgs& a, const float4& me, int l) {
    const float cell = a.cell * (float)(1 << l);
    const CellPos<> p(a, me.x, me.y, me.z, l);
    border = 1.f;
    margin = cell_margin(a, l);
    x = cell_axis(p.c[0], cells_along(a, 0, l), p.f[0] - (float)p.c[0], margin, cell, &border);
    y = cell_axis(p.c[1], cells_along(a, 1, l), p.f[1] - (float)p.c[1], margin, cell, &border);
    z = cell_axis(p.c[2], cells_along(a, 2, l), p.f[2] - (float)p.c[2], margin, cell, &border);
  }
  // squared distance within which every point lies in the cube
  __device__ __forceinline__ float reach2(const KnnArgs& a, int l) const {
    const float r = (1.f + border - margin) * a.cell * (float)(1 << l) * 0.999f;
    return r * r;
  }
};

// Distance in cells, along an axis, from a point at f to cell c, less a margin
// for the rounding of f.
__device__ __forceinline__ float cell_gap(float f, int c, float margin) {
  return fmaxf(fmaxf((float)c - f, f - (float)(c + 1)) - margin, 0.f);
}

// A warp takes 32 consecutive points in Morton order: the 3 smallest squared
// distances of each to other points, then out[point] = 0.5 log(max(1e-14,
// mean)).  The points next to a point in sorted order bound its third distance.
// The lanes whose cells are near the first lane's (nearly always all; the rest
// follow in further rounds, where the Morton order jumps) share a box: its
// cells, and one more on each side, are looked up 32 at a time, and the points
// of a cell that some lane's bound reaches are compared by all lanes at once,
// each read once per warp, so that no lane waits for another's list.  (4M points
// of a surface, whole initialisation: 8.8 ms with a loop over its own 27 cells
// per thread and a cell size by the bounding box's volume; 2.85 ms with a list
// of its cells' runs per thread; 2.03 ms like
// this.)  A point whose third
// distance is not inside the cells next to its own goes on the list of the next
// kernel.
constexpr int kQueryThreads = 128;
constexpr int kQuerySpan = 5;  // cells between a lane's and the first lane's, along an axis
template <bool EVEN>
__global__ void __launch_bounds__(kQueryThreads) knn_query_kernel(KnnArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t first = (((int64_t)blockIdx.x * kQueryThreads + threadIdx.x) >> 5) * 32;
  if (first >= a.n) return;
  const bool mine = first + lane < a.n;
  const int64_t i = min(first + lane, a.n - 1);
  const int level = pick_level(a);
  const uint32_t* keys = sorted_keys(a);
  const float4 me = a.sorted[i];
  float best[3] = {3.0e38f, 3.0e38f, 3.0e38f};
  for (int64_t j = max((int64_t)0, i - 4); j < min(a.n, i + 5); j++)
    if (j != i) near_point(a, j, me.x, me.y, me.z, best);
  const float bound = best[2];
  best[0] = best[1] = best[2] = 3.0e38f;  // (the cells hold these neighbours too)
  // the lane's cell and its position in cells; the warp's box
  const CellPos<EVEN> at(a, me.x, me.y, me.z, level);
  const float cell = a.cell * (float)(1 << level), margin = cell_margin<EVEN>(a, level);
  const float fx = at.f[0], fy = at.f[1], fz = at.f[2];
  const int cx = at.c[0], cy = at.c[1], cz = at.c[2];
  for (uint32_t todo = __ballot_sync(0xffffffffu, mine); todo;) {
    const int lead = __ffs((int)todo) - 1;
    // (every lane takes part in the exchanges)
    const int lx = __shfl_sync(0xffffffffu, cx, lead), ly = __shfl_sync(0xffffffffu, cy, lead);
    const int lz = __shfl_sync(0xffffffffu, cz, lead);
    const bool in = ((todo >> lane) & 1u) != 0u && max(abs(cx - lx), max(abs(cy - ly), abs(cz - lz))) <= kQuerySpan;
    todo &= ~__ballot_sync(0xffffffffu, in);
    // the box of the lanes taken
    auto low = [&](int c) { return max(__reduce_min_sync(0xffffffffu, in ? c : 1 << kMaxLevels) - 1, 0); };
    auto high = [&](int c, int k) {
      return min(__reduce_max_sync(0xffffffffu, in ? c : 0) + 1, cells_along<EVEN>(a, k, level) - 1);
    };
    const int x0 = low(cx), y0 = low(cy), z0 = low(cz);
    const int ex = high(cx, 0) - x0 + 1, exy = ex * (high(cy, 1) - y0 + 1), cells = exy * (high(cz, 2) - z0 + 1);
    const float cap = in ? 3.0e38f : 0.f, reach = in ? bound : -1.f;  // (the other lanes take nothing)
    for (int c0 = 0; c0 < cells; c0 += 32) {
      const int c = c0 + lane;
      const int z = z0 + c / exy, y = y0 + c % exy / ex, x = x0 + c % exy % ex;
      uint2 run = make_uint2(0u, 0u);
      if (c < cells) run = cell_run(a, keys, cell_key<EVEN>(a, (uint32_t)x, (uint32_t)y, (uint32_t)z, level), level);
      // the cell in 10 bits per axis: in the grid, or, where that may take more, in the box
      const int bx = EVEN ? 0 : x0, by = EVEN ? 0 : y0, bz = EVEN ? 0 : z0;
      const uint32_t pos = (uint32_t)((x - bx) | ((y - by) << 10) | ((z - bz) << 20));
      for (uint32_t m = __ballot_sync(0xffffffffu, run.y > run.x); m; m &= m - 1u) {
        const int src = __ffs((int)m) - 1;
        const uint32_t s0 = __shfl_sync(0xffffffffu, run.x, src), s1 = __shfl_sync(0xffffffffu, run.y, src);
        const uint32_t p = __shfl_sync(0xffffffffu, pos, src);
        const float gx = cell_gap(fx, bx + (int)(p & 0x3ffu), margin), gy = cell_gap(fy, by + (int)((p >> 10) & 0x3ffu), margin);
        const float gz = cell_gap(fz, bz + (int)(p >> 20), margin);
        const float gap2 = (gx * gx + gy * gy + gz * gz) * (cell * cell) * 0.999f;
        if (!__any_sync(0xffffffffu, !(gap2 > fminf(best[2], reach)))) continue;
#pragma unroll 4
        for (uint32_t j = s0; j < s1; j++) {
          const float4 q = __ldg(a.sorted + j);
          const float dx = q.x - me.x, dy = q.y - me.y, dz = q.z - me.z;
          float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
          // (not the point itself, and nothing at a NaN)
          d2 = (int64_t)j != i && d2 < cap ? d2 : 3.0e38f;
          best[2] = fminf(best[2], fmaxf(best[1], d2));
          best[1] = fminf(best[1], fmaxf(best[0], d2));
          best[0] = fminf(best[0], d2);
        }
      }
    }
  }
  // every point within this distance lies in the cells next to the lane's
  float border = 1.f;
  border = fminf(border, fminf(fx - (float)cx, 1.f - (fx - (float)cx)));
  border = fminf(border, fminf(fy - (float)cy, 1.f - (fy - (float)cy)));
  border = fminf(border, fminf(fz - (float)cz, 1.f - (fz - (float)cz)));
  const float reach = (1.f + border - margin) * cell * 0.999f;
  if (!mine) return;
  if (best[2] <= reach * reach) write_scale(a, me, best);
  else spare_vals(a)[atomicAdd(a.heads + kTodo, 1u)] = (uint32_t)i;
}

// The points left over (a few in a hundred; isolated ones among them need cubes that hold thousands of others): one warp each, over the
// cubes of 3^3 cells of coarser and coarser levels until the third distance is
// inside.  Lanes find the 27 runs by bisection, share the points of the runs,
// and merge their three best.
__global__ void __launch_bounds__(256) knn_far_kernel(KnnArgs a) {
  const int level = pick_level(a), lane = threadIdx.x & 31;
  const uint32_t* keys = sorted_keys(a);
  const int64_t todo = min((int64_t)a.heads[kTodo], a.n);
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < todo; t += warps) {
    const int64_t i = spare_vals(a)[t];
    const float4 me = a.sorted[i];
    float third[3] = {3.0e38f, 3.0e38f, 3.0e38f};
    for (int l = min(level + 1, a.bits[2]); l <= a.bits[2]; l++) {
      const CellCube c(a, me, l);
      const int shift = level_shift(a, l);
      const int x = lane % 3, y = lane / 3 % 3, z = lane / 9;
      uint32_t lo = 0, hi = 0;
      auto pick = [](const float (&g)[3], int k) { return k == 0 ? g[0] : k == 1 ? g[1] : g[2]; };
      if (lane < 27) {
        const float gap2 = pick(c.x.gap2, x) + pick(c.y.gap2, y) + pick(c.z.gap2, z);
        if (!(gap2 > third[2]) && gap2 < 3.0e38f) {
          const uint64_t k = cell_key(a, (uint32_t)(c.x.c + x - 1), (uint32_t)(c.y.c + y - 1), (uint32_t)(c.z.c + z - 1), l);
          lo = (uint32_t)lower_bound(keys, 0, a.n, k << shift);
          hi = (uint32_t)lower_bound(keys, lo, a.n, (k + 1) << shift);
        }
      }
      float best[3] = {3.0e38f, 3.0e38f, 3.0e38f};
      for (int q = 0; q < 27; q++) {
        const uint32_t s0 = __shfl_sync(0xffffffffu, lo, q), s1 = __shfl_sync(0xffffffffu, hi, q);
        for (uint32_t j = s0 + lane; j < s1; j += 32)
          if ((int64_t)j != i) near_point(a, j, me.x, me.y, me.z, best);
      }
      // the three smallest of the lanes' lists (distances order like their bits)
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const uint32_t m = __reduce_min_sync(0xffffffffu, __float_as_uint(best[0]));
        const uint32_t who = __ballot_sync(0xffffffffu, __float_as_uint(best[0]) == m);
        if (lane == __ffs((int)who) - 1) {
          best[0] = best[1];
          best[1] = best[2];
          best[2] = 3.0e38f;
        }
        third[k] = __uint_as_float(m);
      }
      if (third[2] <= c.reach2(a, l)) break;
    }
    if (lane == 0) write_scale(a, me, third);
  }
}

void launch_knn_bounds(const float* pts, const int64_t* sel, int64_t n, float* part, int nparts, float* out,
                       cudaStream_t s) {
  knn_bounds_kernel<<<nparts, 256, 0, s>>>(pts, sel, n, part);
  knn_bounds_finish_kernel<<<1, 192, 0, s>>>(part, nparts, out);
}

static unsigned knn_blocks(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 32));
}

void launch_knn_keys(const KnnArgs& a, cudaStream_t s) { knn_keys_kernel<<<knn_blocks(a.n), 256, 0, s>>>(a); }

int knn_grid(const float* lo, const float* hi, KnnArgs* a) {
  double ext[3], longest = 0.0;
  for (int d = 0; d < 3; d++) longest = std::max(longest, ext[d] = std::max((double)hi[d] - (double)lo[d], 0.0));
  // (at 2^10 the bits never exceed 30)
  for (int levels = kMaxLevels; levels >= kKeyBits / 3; levels--) {
    const double cell = longest / (double)(1 << levels);
    int bits[3], total = 0;
    for (int d = 0; d < 3; d++) {
      // bits of the last cell along the axis (the end of the longest side falls on the next one's border)
      const int last = (int)(ext[d] / cell * (1.0 + 1e-6));
      for (bits[d] = 0; bits[d] < levels && (last >> bits[d]) != 0;) bits[d]++;
      total += bits[d];
    }
    if (total > kKeyBits) continue;
    for (int k = 0; k < 3; k++) a->axis[k] = k;
    std::stable_sort(a->axis, a->axis + 3, [&](int x, int y) { return bits[x] < bits[y]; });
    for (int k = 0; k < 3; k++) {
      a->bits[k] = bits[a->axis[k]];
      a->lo[k] = lo[a->axis[k]];
    }
    a->cell = (float)cell;
    a->inv_cell = (float)(1.0 / cell);
    // ten times the rounding of a position at the far end (a difference and two roundings of the product)
    a->margin = kKnnMargin * (float)(1 << (levels - kKeyBits / 3));
    return total;
  }
  return 0;
}

void launch_knn_query(const KnnArgs& a, cudaStream_t s) {
  knn_sorted_points_kernel<<<knn_blocks(a.n), 256, 0, s>>>(a);
  knn_table_kernel<<<knn_blocks(a.n), 256, 0, s>>>(a);
  const unsigned queries = (unsigned)((a.n + kQueryThreads - 1) / kQueryThreads);
  if (a.bits[0] == a.bits[2]) knn_query_kernel<true><<<queries, kQueryThreads, 0, s>>>(a);
  else knn_query_kernel<false><<<queries, kQueryThreads, 0, s>>>(a);
  knn_far_kernel<<<knn_blocks(a.n), 256, 0, s>>>(a);
}

// ---------------------------------------------------------------- initial parameters

// Parameter planes of the initial Gaussians: mean = point, log-scales
// (s, s, s + log flatten), rotation taking +z onto the normal, the given
// opacity logit, SH DC of the Lambertian grey under the light (1,1,1)/sqrt 3,
// higher SH 0.  sel (optional) picks the points.
__global__ void __launch_bounds__(256) init_params_kernel(InitArgs a) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= a.n) return;
  const int64_t S = a.stride;
  float* P = a.params;
  const int64_t src = a.sel ? a.sel[g] : g;
  const float nx = a.normals[3 * src], ny = a.normals[3 * src + 1], nz = a.normals[3 * src + 2];
#pragma unroll
  for (int d = 0; d < 3; d++) P[d * S + g] = a.points[3 * src + d];
  const float s = a.log_scales[g];
  P[3 * S + g] = s;
  P[4 * S + g] = s;
  P[5 * S + g] = s + a.log_flatten;
  float qw = 1.f + nz, qx = -ny, qy = nx, qz = 0.f;
  if (qw < 1e-6f) {
    qw = 0.f;
    qx = 1.f;
    qy = 0.f;
  }
  const float inv = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
  P[6 * S + g] = qw * inv;
  P[7 * S + g] = qx * inv;
  P[8 * S + g] = qy * inv;
  P[9 * S + g] = qz * inv;
  P[10 * S + g] = a.opacity_logit;
  const float c = 0.1f + 0.9f * fmaxf(0.f, (nx + ny + nz) * 0.57735026918962576f);
  const float dc = (c - 0.5f) * 3.5449077018110318f;  // 2 sqrt(pi)
  for (int k = 0; k < a.planes - 11; k++) P[(11 + k) * S + g] = k < 3 ? dc : 0.f;
}

void launch_init_params(const InitArgs& a, cudaStream_t s) {
  if (a.n <= 0) return;
  init_params_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, s>>>(a);
}

}  // namespace gs
