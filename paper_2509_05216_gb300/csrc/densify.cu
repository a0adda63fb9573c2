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
// together: a counting pass (outputs per block of 1,024 Gaussians), the
// binning's block-sum scan, a pass that writes the source of every output
// (and the means of the split samples), and a copy of every plane that
// gathers by source and writes whole coalesced lines.
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

constexpr int kDensifyItems = 4;  // Gaussians per thread of the counting and source passes
constexpr int kDensifyBlock = 256 * kDensifyItems;
// Source word of an output: its input Gaussian (n below 2^31), and the top
// bit when its moments start at zero.  A clone's copy follows its original,
// whose word is the bare Gaussian; a fresh output that does not is a split
// sample.
constexpr uint32_t kSrcFresh = 1u << 31;

// Thread t takes Gaussians 4 t .. 4 t + 3 of the block's 1,024, so that one
// block scan of the threads' sums keeps the input order.
__global__ void __launch_bounds__(256) densify_count_kernel(DensifyArgs a) {
  __shared__ uint32_t warp_tot[8];
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < kDensifyItems; i++) {
    const int64_t g = (int64_t)blockIdx.x * kDensifyBlock + threadIdx.x * kDensifyItems + i;
    if (g < a.n) c += (uint32_t)outputs(decide(a, g), a.split_n);
  }
  uint32_t tot;
  block_prefix(c, warp_tot, &tot);
  if (threadIdx.x == 0) a.block_counts[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(256) densify_source_kernel(DensifyArgs a) {
  __shared__ uint32_t warp_tot[8];
  const int64_t g0 = (int64_t)blockIdx.x * kDensifyBlock + threadIdx.x * kDensifyItems;
  int kind[kDensifyItems];
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < kDensifyItems; i++) {
    kind[i] = g0 + i < a.n ? decide(a, g0 + i) : kPrune;
    c += (uint32_t)outputs(kind[i], a.split_n);
  }
  uint32_t tot;
  int64_t o = block_prefix(c, warp_tot, &tot);
  o += a.block_offsets[blockIdx.x];
  const int64_t S = a.stride, OS = a.out_stride;
#pragma unroll
  for (int i = 0; i < kDensifyItems; i++) {
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

int64_t densify_blocks(int64_t n) { return (n + kDensifyBlock - 1) / kDensifyBlock; }

void launch_densify_count(const DensifyArgs& a, cudaStream_t s) {
  densify_count_kernel<<<(unsigned)densify_blocks(a.n), 256, 0, s>>>(a);
}

void launch_densify_emit(const DensifyArgs& a, int64_t n_out, cudaStream_t s) {
  if (n_out <= 0) return;
  densify_source_kernel<<<(unsigned)densify_blocks(a.n), 256, 0, s>>>(a);
  constexpr int kPlanes = 15;  // planes per block: a quarter of degree 3's 59
  densify_copy_kernel<<<dim3((unsigned)((n_out + 1023) / 1024), (a.planes + kPlanes - 1) / kPlanes), 256, 0, s>>>(
      a, n_out, kPlanes);
}

}  // namespace gs
