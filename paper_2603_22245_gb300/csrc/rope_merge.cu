// Merge of the per-range candidate lists, optional FP32 re-scoring by direct
// summation, and the final per-read top-k (§3.5, generalised from top-1).
//
// Candidates are ordered by the 64-bit key (orderable score << 32 | ~window), so
// the best entry is the key maximum and ties in score go to the lower window.
// A block of eight warps takes rpb reads in three steps:
//   1. one warp per read keeps the best `depth` candidates, one per lane: the
//      keys of 512 entries at a time are held in registers, and the largest
//      left is taken until it no longer beats the worst kept (with sep > 0 at
//      most one per bucket, the best);
//   2. if re-scoring is on, the block's warps share the kept (read, window)
//      pairs: the window's encoding by direct summation (rope_window_sum.cuh)
//      or, in a materialised index, its stored row, against the read's FP32
//      encoding;
//   3. each read's kept entries are sorted across its warp (bitonic) and the
//      first k written.
// Bound by instruction latency (a few KB of candidates and letters per read);
// so small batches get one read per block, and the pairs of a read run side by
// side. Measured, merge with re-scoring of 16 candidates (one warp per read,
// 147 dependent updates per window before): 256 reads 199 -> 31 us, 4,096
// reads of 608 candidates 690 -> 304 us.
#include "rope_internal.h"
#include "rope_topk.cuh"
#include "rope_window_sum.cuh"

namespace rope {

__device__ __forceinline__ uint32_t ord_float(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unord_float(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
}
__device__ __forceinline__ uint64_t cand_key(float s, uint32_t w) {
  return ((uint64_t)ord_float(s) << 32) | (uint64_t)(0xFFFFFFFFu - w);
}

// largest of the warp's values, by its high and then its low word
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) { return ~warp_max_u64(~v); }

constexpr int kMergeWarps = 8;
constexpr int kMergeKeys = 16;  // candidate keys per lane held at a time

// Step 1: the best `depth` of the read's `total` candidates; entry i of the kept
// list in lane i's `mine` (unordered). Returns their number.
__device__ __forceinline__ int merge_select(const DevIndex& ix, const MergeArgs& a, const Candidate* cands, int total,
                                            int depth, uint64_t& mine) {
  const int lane = threadIdx.x & 31;
  mine = 0;
  int64_t my_bucket = -1;
  int n = 0;
  uint64_t worst = 0;  // smallest kept key once the list is full
  for (int base = 0; base < total; base += 32 * kMergeKeys) {
    uint64_t key[kMergeKeys], top = 0;
#pragma unroll
    for (int q = 0; q < kMergeKeys; ++q) {
      const int e = base + 32 * q + lane;
      key[q] = 0;
      if (e >= total) continue;
      const Candidate c = cands[e];
      if (c.win >= kUnusedWin) continue;  // empty entry, or the mark of an unused slot
      if (cands[e - e % a.cand_depth].win == kUnusedWin) continue;  // rest of an unused slot
      if (c.win >= ix.W) {
        // no scan writes a window past the index: a corrupt slot, never dereferenced
        set_status(a.status, kStatusBadArg);
        set_status(a.sticky_status, kStatusBadArg);
        continue;
      }
      key[q] = cand_key(c.score, c.win);
      top = key[q] > top ? key[q] : top;
    }
    while (true) {
      const uint64_t best = warp_max_u64(top);
      if (best == 0 || (n == depth && best <= worst)) break;
      if (top == best) {
        top = 0;
#pragma unroll
        for (int q = 0; q < kMergeKeys; ++q) {
          if (key[q] == best) key[q] = 0;
          top = key[q] > top ? key[q] : top;
        }
      }
      int slot = n;
      int64_t bucket = -1;
      if (a.sep > 0) {
        // a kept entry of the same bucket makes way if it is the worse one
        bucket = (int64_t)(0xFFFFFFFFu - (uint32_t)best) * ix.stride / a.sep;
        const uint32_t same = __ballot_sync(0xffffffffu, lane < n && my_bucket == bucket);
        if (same) {
          slot = __ffs(same) - 1;
          if (__shfl_sync(0xffffffffu, mine, slot) >= best) continue;
        }
      }
      if (slot == n) {
        if (n == depth) {
          slot = __ffs(__ballot_sync(0xffffffffu, lane < n && mine == worst)) - 1;
        } else {
          ++n;
        }
      }
      if (lane == slot) {
        mine = best;
        my_bucket = bucket;
      }
      if (n == depth) worst = warp_min_u64(lane < n ? mine : ~0ull);
    }
  }
  return n;
}

// Step 2: the FP32 fidelity of window jw against read r (warp-wide).
__device__ __forceinline__ float merge_rescore(const DevIndex& ix, const MergeArgs& a, int64_t r, uint32_t jw,
                                               float2* stage) {
  const int lane = threadIdx.x & 31;
  const int D = ix.D;
  const float* x = a.emb_f32 + (size_t)r * 2 * D;
  const float* nr = a.norms + (size_t)r * (1 + ix.m);
  auto warp_sum3 = [](float& u, float& v, float& w) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      u += __shfl_xor_sync(0xffffffffu, u, o);
      v += __shfl_xor_sync(0xffffffffu, v, o);
      w += __shfl_xor_sync(0xffffffffu, w, o);
    }
  };
  if (ix.win_f32) {
    // materialised index: the window's stored FP32 encoding (§2.1-§2.3
    // sums, built once) against the read's FP32 encoding
    const float* cw = ix.win_f32 + (size_t)jw * 2 * D;
    float re = 0.f, im = 0.f, C = 0.f;
#pragma unroll 8
    for (int g = lane; g < D; g += 32) {
      const float xr = __ldg(x + g), xi = __ldg(x + D + g);
      const float cr = __ldg(cw + g), ci = __ldg(cw + D + g);
      re = fmaf(xr, cr, fmaf(xi, ci, re));
      im = fmaf(xr, ci, fmaf(-xi, cr, im));
      C = fmaf(cr, cr, fmaf(ci, ci, C));
    }
    warp_sum3(re, im, C);
    const float X = nr[0];
    return (X > kZeroNorm2 && C > kZeroNorm2) ? fmaf(re, re, im * im) / (X * C) : 0.f;
  }
  const float2* acc = window_direct_sum(ix, (int64_t)jw * ix.stride, stage);
  float fid = 0.f;
  if (ix.score_mode == 0) {
    float re = 0.f, im = 0.f, C = 0.f;
    for (int g = lane; g < D; g += 32) {
      const float xr = x[g], xi = x[D + g];
      const float2 c = acc[g];
      re = fmaf(xr, c.x, fmaf(xi, c.y, re));
      im = fmaf(xr, c.y, fmaf(-xi, c.x, im));
      C = fmaf(c.x, c.x, fmaf(c.y, c.y, C));
    }
    warp_sum3(re, im, C);
    const float X = nr[0];
    fid = (X > kZeroNorm2 && C > kZeroNorm2) ? fmaf(re, re, im * im) / (X * C) : 0.f;
  } else {
    for (int k = 0; k < ix.m; ++k) {
      float re = 0.f, im = 0.f, C = 0.f;
      for (int b = lane; b < ix.nb; b += 32) {
        const int g = k * ix.nb + b;
        const float xr = x[g], xi = x[D + g];
        const float2 c = acc[g];
        re = fmaf(xr, c.x, fmaf(xi, c.y, re));
        im = fmaf(xr, c.y, fmaf(-xi, c.x, im));
        C = fmaf(c.x, c.x, fmaf(c.y, c.y, C));
      }
      warp_sum3(re, im, C);
      const float Xk = nr[1 + k];
      fid += (Xk > kZeroNorm2 && C > kZeroNorm2) ? fmaf(re, re, im * im) / (Xk * C) : 0.f;
    }
    fid /= ix.m;
  }
  __syncwarp();
  return fid;
}

__global__ void __launch_bounds__(32 * kMergeWarps, 3) merge_kernel(DevIndex ix, MergeArgs a, int rpb) {
  extern __shared__ float2 merge_smem[];
  __shared__ uint64_t keys[kMergeWarps][32];
  __shared__ int n_sel[kMergeWarps];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  float2* stage = merge_smem + (size_t)warp * window_sum_smem(ix.m, ix.D);
  const int total = a.n_ranges * a.cand_depth;
  const int depth = a.rescore ? a.rescore_depth : a.k;
  // the scan's lists are incomplete after a timeout: report nothing rather than part
  const int scan_bits = *reinterpret_cast<volatile int*>(a.status);
  const bool give_up = a.empty_on_timeout && (scan_bits & kStatusTimeout);
  if (a.sticky_status && blockIdx.x == 0 && threadIdx.x == 0 && scan_bits) atomicOr(a.sticky_status, scan_bits);

  for (int64_t r0 = (int64_t)blockIdx.x * rpb; r0 < a.n_reads; r0 += (int64_t)gridDim.x * rpb) {
    const int64_t r = r0 + warp;  // steps 1 and 3: this warp's read
    const bool own = warp < rpb && r < a.n_reads;
    if (own) {
      uint64_t mine = 0;
      const int n = give_up ? 0 : merge_select(ix, a, a.cand + (size_t)r * total, total, depth, mine);
      keys[warp][lane] = mine;
      if (lane == 0) n_sel[warp] = n;
    }
    __syncthreads();
    if (a.rescore) {
      const int n_here = (int)(a.n_reads - r0 < rpb ? a.n_reads - r0 : rpb);
      for (int q = 0; q < n_here; ++q)
        for (int i = warp; i < n_sel[q]; i += kMergeWarps) {
          const uint32_t jw = 0xFFFFFFFFu - (uint32_t)keys[q][i];
          const float fid = merge_rescore(ix, a, r0 + q, jw, stage);
          if (lane == 0) keys[q][i] = cand_key(fid, jw);
        }
      __syncthreads();
    }
    if (own) {
      uint64_t my_key = keys[warp][lane];
      // bitonic sort of the kept keys across the warp, descending
#pragma unroll
      for (int k2 = 2; k2 <= 32; k2 <<= 1) {
#pragma unroll
        for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
          const uint64_t other = __shfl_xor_sync(0xffffffffu, my_key, j2);
          const int p = lane ^ j2;
          const bool take_max = (((lane & k2) == 0) == (lane < p));
          my_key = take_max ? (other > my_key ? other : my_key) : (other < my_key ? other : my_key);
        }
      }
      if (lane < a.k) {
        int64_t ow = -1;
        float os = -INFINITY;
        if (lane < n_sel[warp] && my_key != 0) {
          ow = (int64_t)(0xFFFFFFFFu - (uint32_t)my_key) * ix.stride;
          os = unord_float((uint32_t)(my_key >> 32));
        }
        const int64_t orow = a.out_row ? a.out_row[r] : r;
        a.out_win[orow * a.k + lane] = ow;
        a.out_score[orow * a.k + lane] = os;
      }
    }
    __syncthreads();  // keys and counts are reused by the next reads
  }
}

cudaError_t launch_merge(const DevIndex& ix, const MergeArgs& a, cudaStream_t st) {
  if (a.n_reads <= 0) return cudaSuccess;
  // reads per block: one where the reads alone would not fill the chip (about
  // four blocks per SM), eight where every warp has a read of its own
  const int64_t want = a.n_reads / (4 * 152);
  const int rpb = (int)(want < 1 ? 1 : want > kMergeWarps ? kMergeWarps : want);
  int64_t blocks = (a.n_reads + rpb - 1) / rpb;
  if (blocks > 152 * 32) blocks = 152 * 32;
  const size_t smem = ix.win_f32 ? 0 : (size_t)kMergeWarps * window_sum_smem(ix.m, ix.D) * sizeof(float2);
  merge_kernel<<<(unsigned)blocks, 32 * kMergeWarps, smem, st>>>(ix, a, rpb);
  return cudaGetLastError();
}

}  // namespace rope

namespace rope {

// Two sorted top-k lists per read (forward row r, reverse row n + r, each by
// score descending and start ascending, missing entries (-1, -inf) last)
// merged into one: score descending, the forward strand first on equal
// scores, then the lower start.
__global__ void strand_merge_kernel(const int64_t* __restrict__ win2, const float* __restrict__ score2, int64_t n,
                                    int k, int64_t* __restrict__ out_win, float* __restrict__ out_score,
                                    int8_t* __restrict__ out_strand) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t* wf = win2 + r * k;
    const int64_t* wr = win2 + (n + r) * k;
    const float* sf = score2 + r * k;
    const float* sr = score2 + (n + r) * k;
    int i = 0, j = 0;
    for (int o = 0; o < k; ++o) {
      const bool okf = i < k && wf[i] >= 0, okr = j < k && wr[j] >= 0;
      int8_t strand = -1;
      if (okf && okr) {
        strand = sr[j] > sf[i] ? 1 : 0;  // equal scores: forward first
      } else if (okf) {
        strand = 0;
      } else if (okr) {
        strand = 1;
      }
      int64_t w = -1;
      float sc = -INFINITY;
      if (strand == 0) {
        w = wf[i];
        sc = sf[i++];
      } else if (strand == 1) {
        w = wr[j];
        sc = sr[j++];
      }
      out_win[r * k + o] = w;
      out_score[r * k + o] = sc;
      out_strand[r * k + o] = strand;
    }
  }
}

cudaError_t launch_strand_merge(const int64_t* win2, const float* score2, int64_t n, int k, int64_t* out_win,
                                float* out_score, int8_t* out_strand, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  strand_merge_kernel<<<(unsigned)blocks, 256, 0, st>>>(win2, score2, n, k, out_win, out_score, out_strand);
  return cudaGetLastError();
}

}  // namespace rope
