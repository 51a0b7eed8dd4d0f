// The encoding of one reference window by direct summation (§2.1-§2.3, FP32),
// one warp per window: what the re-scoring and the reranker's features use.
//
// Lane l owns entries g = l, l + 32, ... of the D complex entries in registers.
// Locations are taken 32 at a time, one per lane; ballots over the bits of
// their bins tell a lane which of them fall in its entries' bins, and it adds
// their phases (staged in shared memory, loaded a chunk ahead) in increasing
// order: every entry is its location-order sum, the same bits as adding one
// location after another. A chunk costs the warp a few ballots and about the
// largest bin's count of additions (5-6 of 32), where walking the locations
// costs 32 dependent shared-memory updates by m lanes.
#pragma once

#include "rope_common.cuh"

namespace rope {

constexpr int kSumMaxBands = 8;
constexpr int kSumMaxPerLane = kMaxScanDim / 32;
constexpr int kSumMaxBinBits = 8;  // bins per band up to 256

// float2 entries of shared memory a warp needs: 32 phases per band (up to
// kMaxScanDim entries), then the D sums
__host__ __device__ constexpr int window_sum_stage(int m, int D) { return D <= kMaxScanDim ? 32 * m : 0; }
__host__ __device__ constexpr int window_sum_smem(int m, int D) { return window_sum_stage(m, D) + D; }

// c(w0) into the D sums behind the warp's staged phases, which it returns.
__device__ __forceinline__ float2* window_direct_sum(const DevIndex& ix, int64_t w0, float2* stage) {
  const int lane = threadIdx.x & 31;
  const int n_loc = ix.N - ix.s + 1;
  float2* acc = stage + window_sum_stage(ix.m, ix.D);
  if (ix.D > kMaxScanDim) {
    // wider encodings (a materialised index's): one location after another,
    // the lanes k < m adding to their band's entry
    for (int g = lane; g < ix.D; g += 32) acc[g] = make_float2(0.f, 0.f);
    __syncwarp();
    for (int loc0 = 0; loc0 < n_loc; loc0 += 32) {
      const int loc = loc0 + lane;
      const uint32_t b = loc < n_loc ? bin_at(ix.packed, w0 + loc, ix.s, ix.map_lsb) : 0u;
      const int cnt = min(32, n_loc - loc0);
      for (int jj = 0; jj < cnt; ++jj) {
        const uint32_t bj = __shfl_sync(0xffffffffu, b, jj);
        if (lane < ix.m) {
          const float2 p = ix.phase[lane * n_loc + loc0 + jj];
          float2& v = acc[lane * ix.nb + bj];
          v.x += p.x;
          v.y += p.y;
        }
        __syncwarp();
      }
    }
    return acc;
  }
  const int bits = 32 - __clz(ix.nb > 1 ? ix.nb - 1 : 1);
  float ar[kSumMaxPerLane], ai[kSumMaxPerLane];
#pragma unroll
  for (int e = 0; e < kSumMaxPerLane; ++e) ar[e] = ai[e] = 0.f;
  uint32_t b = 0;
  float2 ph[kSumMaxBands];
  auto fetch = [&](int loc) {
    if (loc >= n_loc) return;
    b = bin_at(ix.packed, w0 + loc, ix.s, ix.map_lsb);
#pragma unroll
    for (int k = 0; k < kSumMaxBands; ++k)
      if (k < ix.m) ph[k] = __ldg(ix.phase + (size_t)k * n_loc + loc);
  };
  fetch(lane);
  for (int loc0 = 0; loc0 < n_loc; loc0 += 32) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kSumMaxBands; ++k)
      if (k < ix.m) stage[k * 32 + lane] = ph[k];
    __syncwarp();
    const uint32_t cur = b;
    const uint32_t valid = n_loc - loc0 >= 32 ? 0xffffffffu : (1u << (n_loc - loc0)) - 1u;
    fetch(loc0 + 32 + lane);
    uint32_t plane[kSumMaxBinBits];
#pragma unroll
    for (int i = 0; i < kSumMaxBinBits; ++i) plane[i] = i < bits ? __ballot_sync(0xffffffffu, (cur >> i) & 1u) : 0u;
#pragma unroll
    for (int e = 0; e < kSumMaxPerLane; ++e) {
      const int g = lane + 32 * e;
      if (32 * e >= ix.D || g >= ix.D) continue;
      const int band = g / ix.nb, bin = g - band * ix.nb;
      uint32_t hit = valid;
#pragma unroll
      for (int i = 0; i < kSumMaxBinBits; ++i)
        if (i < bits) hit &= ((bin >> i) & 1) ? plane[i] : ~plane[i];
      const float2* row = stage + band * 32;
      while (hit) {  // the matching locations in increasing order, up to four loads at a time
        const uint32_t h1 = hit & (hit - 1u), h2 = h1 & (h1 - 1u), h3 = h2 & (h2 - 1u);
        const float2 p0 = row[__ffs(hit) - 1];
        const float2 p1 = row[(__ffs(h1) - 1) & 31], p2 = row[(__ffs(h2) - 1) & 31], p3 = row[(__ffs(h3) - 1) & 31];
        ar[e] += p0.x;
        ai[e] += p0.y;
        if (h1) {
          ar[e] += p1.x;
          ai[e] += p1.y;
        }
        if (h2) {
          ar[e] += p2.x;
          ai[e] += p2.y;
        }
        if (h3) {
          ar[e] += p3.x;
          ai[e] += p3.y;
        }
        hit = h3 & (h3 - 1u);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < kSumMaxPerLane; ++e) {
    const int g = lane + 32 * e;
    if (g < ix.D) acc[g] = make_float2(ar[e], ai[e]);
  }
  __syncwarp();
  return acc;
}

}  // namespace rope
