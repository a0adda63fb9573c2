// Adaptive density control of 3D-GS: clone, split and prune Gaussians from
// the screen-space gradient statistic accumulated by the projection
// backward.
//
// The paper is silent on densification (N comes from the point cloud); this
// is 3D-GS's step: a Gaussian whose mean gradient, averaged over the views
// where it touches a tile, reaches the threshold is cloned when small
// (largest scale <= percent_dense x scene extent) and split into N samples
// of its own distribution (scales shrunk by 0.8 N) when large; Gaussians
// whose opacity is below the minimum are removed.  New Gaussians start with
// zero Adam moments.  The output keeps the input order, a Gaussian's outputs
// together: a counting pass (outputs per block of 256 or 1,024 Gaussians), the
// binning's block-sum scan, a pass that writes the source of every output
// (and the means of the split samples), and a copy of every plane that
// gathers by source and writes whole coalesced lines.
#include <algorithm>
#include <cmath>

#include "gs_internal.cuh"
#include "launch.h"

namespace gs {

namespace {

enum { kPrune = 0, kKeep = 1, kClone = 2, kSplit = 3 };

__device__ __forceinline__ int decide(const DensifyArgs& a, int64_t g) {
  const int64_t S = a.stride;
  const float o = a.p[10 * S + g];
  if (1.f / (1.f + expf(-o)) < a.min_opacity) return kPrune;
  const float c = a.count[g];
  const float avg = c > 0.f ? a.grad[g] / c : 0.f;
  if (!(avg >= a.tau)) return kKeep;
  const float smax = expf(fmaxf(a.p[3 * S + g], fmaxf(a.p[4 * S + g], a.p[5 * S + g])));
  return smax <= a.dense_extent ? kClone : kSplit;
}

__device__ __forceinline__ int outputs(int kind, int split_n) {
  return kind == kPrune ? 0 : kind == kKeep ? 1 : kind == kClone ? 2 : split_n;
}

__device__ __forceinline__ uint32_t block_prefix(uint32_t c, uint32_t* warp_tot, uint32_t* total) {
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

}  // namespace

// Gaussians per thread of the counting and source passes: 4, or 1 below 5 blocks
// of 1,024 per SM (a thread's splits are a chain).  Whole call, 1 / 4 per thread:
// 5,000 Gaussians of degree 0 51 / 63 us, 160,000 of degree 3 92 / 98, 700,000 231 /
// 235, 1M 313 / 305, 4M 1120 / 1080.
constexpr int kDensifyMany = 4, kDensifyFew = 1;
static int densify_items(int64_t n) {
  return n >= (int64_t)5 * 256 * kDensifyMany * sm_count() ? kDensifyMany : kDensifyFew;
}
// Source word of an output: its input Gaussian (n below 2^31), and the top
// bit when its moments start at zero.  A clone's copy follows its original,
// whose word is the bare Gaussian; a fresh output that does not is a split
// sample.
constexpr uint32_t kSrcFresh = 1u << 31;

// Thread t takes ITEMS consecutive Gaussians of the block's 256 ITEMS, so that
// one block scan of the threads' sums keeps the input order.
template <int ITEMS>
__global__ void __launch_bounds__(256) densify_count_kernel(DensifyArgs a) {
  __shared__ uint32_t warp_tot[8];
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int64_t g = (int64_t)blockIdx.x * (256 * ITEMS) + threadIdx.x * ITEMS + i;
    if (g < a.n) c += (uint32_t)outputs(decide(a, g), a.split_n);
  }
  uint32_t tot;
  block_prefix(c, warp_tot, &tot);
  if (threadIdx.x == 0) a.block_counts[blockIdx.x] = tot;
}

template <int ITEMS>
__global__ void __launch_bounds__(256) densify_source_kernel(DensifyArgs a) {
  __shared__ uint32_t warp_tot[8];
  const int64_t g0 = (int64_t)blockIdx.x * (256 * ITEMS) + threadIdx.x * ITEMS;
  int kind[ITEMS];
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    kind[i] = g0 + i < a.n ? decide(a, g0 + i) : kPrune;
    c += (uint32_t)outputs(kind[i], a.split_n);
  }
  uint32_t tot;
  int64_t o = block_prefix(c, warp_tot, &tot);
  o += a.block_offsets[blockIdx.x];
  const int64_t S = a.stride, OS = a.out_stride;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const int64_t g = g0 + i;
    if (kind[i] == kKeep || kind[i] == kClone) {
      a.source[o++] = (uint32_t)g;
      if (kind[i] == kClone) a.source[o++] = (uint32_t)g | kSrcFresh;
    } else if (kind[i] == kSplit) {
      // N samples of the Gaussian's own distribution, mean + R (s * z)
      const float w0 = a.p[6 * S + g], x0 = a.p[7 * S + g], y0 = a.p[8 * S + g], z0 = a.p[9 * S + g];
      const float iq = rsqrtf(w0 * w0 + x0 * x0 + y0 * y0 + z0 * z0);
      const float w = w0 * iq, x = x0 * iq, y = y0 * iq, z = z0 * iq;
      const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z),       2.f * (x * z + w * y),
                          2.f * (x * y + w * z),       1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                          2.f * (x * z - w * y),       2.f * (y * z + w * x),       1.f - 2.f * (x * x + y * y)};
      float sc[3];
#pragma unroll
      for (int d = 0; d < 3; d++) sc[d] = expf(a.p[(3 + d) * S + g]);
      for (int k = 0; k < a.split_n; k++, o++) {
        const float* zz = a.noise + 3 * ((int64_t)g * a.split_n + k);
        const float u0 = sc[0] * zz[0], u1 = sc[1] * zz[1], u2 = sc[2] * zz[2];
#pragma unroll
        for (int d = 0; d < 3; d++)
          a.po[d * OS + o] = a.p[d * S + g] + (R[3 * d] * u0 + R[3 * d + 1] * u1 + R[3 * d + 2] * u2);
        a.source[o] = (uint32_t)g | kSrcFresh;
      }
    }
  }
}

// Parameters and moments of the outputs: a block takes 1,024 consecutive
// outputs and a range of planes (blockIdx.y); a thread keeps the sources of 4
// outputs, 256 apart, and has the 12 loads of a plane of the three sets in
// flight.  Bound by HBM: sources are increasing, so a warp's gathers fall in
// one or two lines, and every store is a whole line.
__global__ void __launch_bounds__(256) densify_copy_kernel(DensifyArgs a, int64_t n_out, int planes_per_block) {
  constexpr int U = 4;
  const int64_t o0 = (int64_t)blockIdx.x * (256 * U) + threadIdx.x;
  uint32_t src[U];
  bool fresh[U], split[U];
#pragma unroll
  for (int u = 0; u < U; u++) {
    const int64_t o = o0 + 256 * u;
    const uint32_t w = o < n_out ? a.source[o] : 0u;
    const uint32_t before = o > 0 && o < n_out ? a.source[o - 1] : ~0u;
    src[u] = w & ~kSrcFresh;
    fresh[u] = (w & kSrcFresh) != 0u;
    split[u] = fresh[u] && before != src[u];
  }
  const int pl1 = min(a.planes, ((int)blockIdx.y + 1) * planes_per_block);
  for (int pl = (int)blockIdx.y * planes_per_block; pl < pl1; pl++) {
    const float* p = a.p + pl * a.stride;
    const float* m = a.m + pl * a.stride;
    const float* v = a.v + pl * a.stride;
    float pv[U], mv[U], vv[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      pv[u] = __ldg(p + src[u]);
      mv[u] = fresh[u] ? 0.f : __ldg(m + src[u]);
      vv[u] = fresh[u] ? 0.f : __ldg(v + src[u]);
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int64_t o = o0 + 256 * u;
      if (o >= n_out) continue;
      if (!(split[u] && pl < 3))  // the split samples' means are written already
        a.po[pl * a.out_stride + o] = split[u] && pl < 6 ? pv[u] - a.log_shrink : pv[u];
      a.mo[pl * a.out_stride + o] = mv[u];
      a.vo[pl * a.out_stride + o] = vv[u];
    }
  }
}

int64_t densify_blocks(int64_t n) {
  const int block = 256 * densify_items(n);
  return (n + block - 1) / block;
}

void launch_densify_count(const DensifyArgs& a, cudaStream_t s) {
  const unsigned blocks = (unsigned)densify_blocks(a.n);
  if (densify_items(a.n) == kDensifyMany) densify_count_kernel<kDensifyMany><<<blocks, 256, 0, s>>>(a);
  else densify_count_kernel<kDensifyFew><<<blocks, 256, 0, s>>>(a);
}

void launch_densify_emit(const DensifyArgs& a, int64_t n_out, cudaStream_t s) {
  if (n_out <= 0) return;
  const unsigned in_blocks = (unsigned)densify_blocks(a.n);
  if (densify_items(a.n) == kDensifyMany) densify_source_kernel<kDensifyMany><<<in_blocks, 256, 0, s>>>(a);
  else densify_source_kernel<kDensifyFew><<<in_blocks, 256, 0, s>>>(a);
  // planes per block: a quarter of degree 3's 59, fewer where that leaves less
  // than 4 blocks per SM (a block's planes are a chain of load latencies: 5,000
  // Gaussians, whole call, 63 us with 15 planes, 55 with 1)
  const int64_t blocks = (n_out + 1023) / 1024;
  const int planes = (int)std::clamp<int64_t>(a.planes * blocks / ((int64_t)sm_count() * 4), 1, 15);
  densify_copy_kernel<<<dim3((unsigned)blocks, (a.planes + planes - 1) / planes), 256, 0, s>>>(a, n_out, planes);
}

}  // namespace gs
