// Learned candidate reranker: exact Levenshtein labels, per-candidate
// features, a two-layer MLP (BF16 weights, FP32 arithmetic) with its forward,
// backward and AdamW kernels, and the pruning of each read's candidates to the
// ones with the smallest predicted edit distance.
//
// The paper has no reranker; it relates fidelity to Levenshtein distance (§1,
// §2.4 fitting curve) and thresholds fidelities per fragment (§3.3, §3.5).
// This network learns that relation from the scan's own score features.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "rope_internal.h"
#include "rope_window_sum.cuh"

namespace rope {

// ---------------------------------------------------------------- Levenshtein

// Global edit distance between the read head P (length N, letters from ASCII)
// and the reference window T (length N, from the 2-bit packed reference), by
// the bit-parallel recurrence of Myers (1999) in Hyyro's global form: bit i of
// Pv/Mv holds the vertical delta +1/-1 between rows i and i+1 of the DP
// column; for each text letter the column advances with one carry-propagating
// addition; the top row grows by one per column (global distance), so a 1 is
// shifted into the horizontal positive deltas. W 64-bit words hold N <= 64W.
template <int W>
__global__ void levenshtein_kernel(const uint32_t* __restrict__ packed, const uint8_t* __restrict__ seqs,
                                   const int64_t* __restrict__ offsets, const int64_t* __restrict__ read_idx,
                                   const int64_t* __restrict__ win_start, int64_t n_pairs, int N,
                                   int32_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_pairs; i += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t* P = seqs + offsets[read_idx[i]];
    const int64_t w = win_start[i];
    uint64_t peq[4][W];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int k = 0; k < W; ++k) peq[c][k] = 0;
    for (int p = 0; p < N; ++p) {
      const uint32_t c = letter_code(P[p]) & 3u;
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k == (p >> 6)) peq[c][k] |= 1ull << (p & 63);
    }
    uint64_t pv[W], mv[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
      pv[k] = ~0ull;
      mv[k] = 0;
    }
    const int top = N - 1 - 64 * (W - 1);  // bit of row N-1 in the last word
    int score = N;
    for (int j = 0; j < N; ++j) {
      const int64_t q = w + j;
      const uint32_t c = (packed[q >> 4] >> (2 * (q & 15))) & 3u;
      uint64_t carry = 0, hp_in = 1, hn_in = 0;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const uint64_t eq = peq[c][k];
        const uint64_t xv = eq | mv[k];
        const uint64_t a = eq & pv[k];
        const uint64_t s1 = a + pv[k];
        const uint64_t c1 = s1 < a;
        const uint64_t sum = s1 + carry;
        carry = c1 | (sum < s1);
        const uint64_t xh = (sum ^ pv[k]) | eq;
        uint64_t ph = mv[k] | ~(xh | pv[k]);
        uint64_t mh = pv[k] & xh;
        if (k == W - 1) {
          score += (int)((ph >> top) & 1ull) - (int)((mh >> top) & 1ull);
        }
        const uint64_t hp_out = ph >> 63, hn_out = mh >> 63;
        ph = (ph << 1) | hp_in;
        mh = (mh << 1) | hn_in;
        hp_in = hp_out;
        hn_in = hn_out;
        pv[k] = mh | ~(xv | ph);
        mv[k] = ph & xv;
      }
    }
    out[i] = score;
  }
}

cudaError_t launch_levenshtein(const uint32_t* packed, const uint8_t* seqs, const int64_t* offsets,
                               const int64_t* read_idx, const int64_t* win_start, int64_t n_pairs, int N, int32_t* out,
                               cudaStream_t st) {
  if (n_pairs <= 0) return cudaSuccess;
  const int threads = 128;
  int64_t blocks = (n_pairs + threads - 1) / threads;
  if (blocks > 152 * 64) blocks = 152 * 64;
  const int W = (N + 63) / 64;
  switch (W) {
    case 1: levenshtein_kernel<1><<<(unsigned)blocks, threads, 0, st>>>(packed, seqs, offsets, read_idx, win_start, n_pairs, N, out); break;
    case 2: levenshtein_kernel<2><<<(unsigned)blocks, threads, 0, st>>>(packed, seqs, offsets, read_idx, win_start, n_pairs, N, out); break;
    case 3: levenshtein_kernel<3><<<(unsigned)blocks, threads, 0, st>>>(packed, seqs, offsets, read_idx, win_start, n_pairs, N, out); break;
    case 4: levenshtein_kernel<4><<<(unsigned)blocks, threads, 0, st>>>(packed, seqs, offsets, read_idx, win_start, n_pairs, N, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- features

// Per (read, candidate) feature row, F = K + 2 + m (<= kMaxFeatures):
//   [0, K)       the read's K candidate scores, best first (missing -> 0)
//   K            this candidate's fidelity
//   K+1 .. K+m   this candidate's per-band fidelities |<x_k|c_k>|^2/(X_k C_k)
//   K+m+1        rank / K
// One warp per read; each candidate window is summed directly in FP32
// (location order), as the re-scoring does. Missing candidates get a zero row.
// letter (0..3) at reference position p, or 4 outside [0, L)
__device__ __forceinline__ uint32_t ref_letter(const uint32_t* __restrict__ packed, int64_t L, int64_t p) {
  return (p >= 0 && p < L) ? (packed[p >> 4] >> ((p & 15) * 2)) & 3u : 4u;
}

__global__ void features_kernel(DevIndex ix, const uint8_t* __restrict__ seqs, const int64_t* __restrict__ offsets,
                                const float* __restrict__ emb_f32, const float* __restrict__ norms,
                                const int64_t* __restrict__ cand_win, const float* __restrict__ cand_score,
                                int64_t n_reads, int K, int F, float* __restrict__ X) {
  extern __shared__ float2 feat_acc[];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  float2* stage = feat_acc + (size_t)warp * window_sum_smem(ix.m, ix.D);
  const int D = ix.D;
  for (int64_t r = (int64_t)blockIdx.x * wpb + warp; r < n_reads; r += (int64_t)gridDim.x * wpb) {
    const float* x = emb_f32 + (size_t)r * 2 * D;
    const float* nr = norms + (size_t)r * (1 + ix.m);
    for (int c = 0; c < K; ++c) {
      float* row = X + ((size_t)r * K + c) * F;
      const int64_t w0 = cand_win[r * K + c];
      if (w0 < 0) {
        for (int f = lane; f < F; f += 32) row[f] = 0.f;
        continue;
      }
      const float2* acc = window_direct_sum(ix, w0, stage);
      for (int k = 0; k < ix.m; ++k) {
        float re = 0.f, im = 0.f, C = 0.f;
        for (int b = lane; b < ix.nb; b += 32) {
          const int g = k * ix.nb + b;
          const float xr = x[g], xi = x[D + g];
          const float2 cc = acc[g];
          re = fmaf(xr, cc.x, fmaf(xi, cc.y, re));
          im = fmaf(xr, cc.y, fmaf(-xi, cc.x, im));
          C = fmaf(cc.x, cc.x, fmaf(cc.y, cc.y, C));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          re += __shfl_xor_sync(0xffffffffu, re, o);
          im += __shfl_xor_sync(0xffffffffu, im, o);
          C += __shfl_xor_sync(0xffffffffu, C, o);
        }
        const float Xk = nr[1 + k];
        if (lane == 0) row[K + 1 + k] = (Xk > kZeroNorm2 && C > kZeroNorm2) ? fmaf(re, re, im * im) / (Xk * C) : 0.f;
      }
      for (int f = lane; f < K; f += 32) {
        const float sc = cand_score[r * K + f];
        row[f] = cand_win[r * K + f] >= 0 ? sc : 0.f;
      }
      // Hamming fingerprint fidelities ((n - d) / n)^2 (§1) of the read head
      // against the window and the windows shifted by up to kShift letters
      // (letters outside the reference count as mismatches), and of the two
      // halves of the head at no shift
      {
        const uint8_t* head = seqs + offsets[r];
        const int N = ix.N, n1 = N / 2;
        int mm[2 * kShift + 1], mm1 = 0;
#pragma unroll
        for (int d = 0; d <= 2 * kShift; ++d) mm[d] = 0;
        for (int i = lane; i < N; i += 32) {
          const uint32_t q = letter_code(head[i]);
#pragma unroll
          for (int d = 0; d <= 2 * kShift; ++d) mm[d] += q != ref_letter(ix.packed, ix.L, w0 + i + d - kShift);
          if (i < n1) mm1 += q != ref_letter(ix.packed, ix.L, w0 + i);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
          for (int d = 0; d <= 2 * kShift; ++d) mm[d] += __shfl_xor_sync(0xffffffffu, mm[d], o);
          mm1 += __shfl_xor_sync(0xffffffffu, mm1, o);
        }
        if (lane == 0) {
          auto hf = [](int n, int d) {
            const float v = (float)(n - d) / (float)n;
            return v * v;
          };
          float best = 0.f;
#pragma unroll
          for (int d = 0; d <= 2 * kShift; ++d) best = fmaxf(best, hf(N, mm[d]));
          row[K] = cand_score[r * K + c];
          row[K + 1 + ix.m] = (float)c / (float)K;
          row[K + 2 + ix.m] = hf(N, mm[kShift]);
          row[K + 3 + ix.m] = best;
          row[K + 4 + ix.m] = hf(n1, mm1);
          row[K + 5 + ix.m] = hf(N - n1, mm[kShift] - mm1);
        }
      }
      for (int f = K + 6 + ix.m + lane; f < F; f += 32) row[f] = 0.f;
      __syncwarp();
    }
  }
}

cudaError_t launch_features(const DevIndex& ix, const uint8_t* seqs, const int64_t* offsets, const float* emb_f32,
                            const float* norms, const int64_t* cand_win, const float* cand_score, int64_t n_reads,
                            int K, int F, float* X, cudaStream_t st) {
  if (n_reads <= 0) return cudaSuccess;
  const int wpb = 8;
  int64_t blocks = (n_reads + wpb - 1) / wpb;
  if (blocks > 152 * 32) blocks = 152 * 32;
  features_kernel<<<(unsigned)blocks, wpb * 32, (size_t)wpb * window_sum_smem(ix.m, ix.D) * sizeof(float2), st>>>(
      ix, seqs, offsets, emb_f32, norms, cand_win, cand_score, n_reads, K, F, X);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- MLP

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// Forward: a block takes 32 samples, a lane per sample, and each of its warps a
// share of the hidden units; the BF16 weights are staged in shared memory as
// FP32 rows padded with zeros to FP (features rounded up to 8), read as float4
// broadcasts. pre[j][s] is stored when `pre` is non-null (training; unit-major,
// so stores here and loads in the backward pass are whole lines), and with
// targets the per-sample residual gradient dy = 2 (y - t) / B and squared error.
// Sample s of the batch is row idx[s] of X and t (row s when idx is null).
// A training batch (4,096 samples) is latency: with a thread per sample it ran
// on 32 SMs, 128 units one after another.
constexpr int kMlpWarps = 4;

template <int FP>
__global__ void __launch_bounds__(32 * kMlpWarps)
    mlp_forward_kernel(MlpWeights w, const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t B,
                       float* __restrict__ y, float* __restrict__ pre, const float* __restrict__ t,
                       float* __restrict__ dy, float* __restrict__ sq) {
  extern __shared__ __align__(16) float mlp_smem[];
  __shared__ float xt[32][FP + 1];
  __shared__ int64_t rows[32];
  __shared__ float part[kMlpWarps][32];
  float* W1 = mlp_smem;       // H x FP
  float* b1 = W1 + w.H * FP;  // H
  float* w2 = b1 + w.H;       // H
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < w.H * FP; i += blockDim.x) {
    const int j = i / FP, f = i - j * FP;
    W1[i] = f < w.F ? __bfloat162float(w.W1[j * w.F + f]) : 0.f;
  }
  for (int i = threadIdx.x; i < w.H; i += blockDim.x) {
    b1[i] = w.b1[i];
    w2[i] = __bfloat162float(w.w2[i]);
  }
  const float b2 = w.b2[0];
  const int j_lo = w.H * warp / kMlpWarps, j_hi = w.H * (warp + 1) / kMlpWarps;
  for (int64_t s0 = (int64_t)blockIdx.x * 32; s0 < B; s0 += (int64_t)gridDim.x * 32) {
    const int n = (int)min((int64_t)32, B - s0);
    if (threadIdx.x < 32) rows[lane] = lane < n ? (idx ? idx[s0 + lane] : s0 + lane) : 0;
    __syncthreads();  // (the weights too, the first time)
    for (int i = threadIdx.x; i < 32 * FP; i += blockDim.x) {
      const int q = i / FP, f = i - q * FP;
      xt[q][f] = q < n && f < w.F ? X[rows[q] * w.F + f] : 0.f;
    }
    __syncthreads();
    float xs[FP];
#pragma unroll
    for (int f = 0; f < FP; ++f) xs[f] = xt[lane][f];
    const int64_t s = s0 + lane;
    float acc = 0.f;
#pragma unroll 2
    for (int j = j_lo; j < j_hi; ++j) {
      const float4* row = reinterpret_cast<const float4*>(W1 + j * FP);
      float z = b1[j];
#pragma unroll
      for (int f = 0; f < FP; f += 4) {
        const float4 v = row[f / 4];
        z = fmaf(v.x, xs[f], z);
        z = fmaf(v.y, xs[f + 1], z);
        z = fmaf(v.z, xs[f + 2], z);
        z = fmaf(v.w, xs[f + 3], z);
      }
      if (pre && lane < n) pre[(int64_t)j * B + s] = z;
      acc = fmaf(w2[j], gelu_f(z), acc);
    }
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && lane < n) {
      float v = b2;
#pragma unroll
      for (int q = 0; q < kMlpWarps; ++q) v += part[q][lane];
      if (y) y[s] = v;
      if (t) {
        const float r = v - t[rows[lane]];
        dy[s] = 2.0f * r / (float)B;
        sq[s] = r * r;
      }
    }
    __syncthreads();  // rows, xt and part are free for the next samples
  }
}

// Backward:
//   dW1[j][f] = sum_s dy_s w2_j GELU'(pre_js) x_sf,  db1[j] = sum_s dy_s w2_j GELU'(pre_js)
//   dw2[j]    = sum_s dy_s GELU(pre_js);  db2 = sum_s dy_s, and the loss.
// A cluster of kBwdSplit blocks takes kBwdUnits hidden units, its blocks every
// kBwdSplit-th tile of 32 samples: per tile the block forms dz (a warp per unit,
// a lane per sample) and stages the samples' rows, then each warp adds 4 units x
// FP/4 features with a lane per sample; the next tile's loads are in flight
// meanwhile. Lanes, then the cluster's blocks (through distributed shared
// memory, in FP64), are summed in a fixed order: deterministic. A block per unit read
// every row for one unit and ended in F + 2 block-wide trees.
// `loss` receives the batch mean squared error, or has it added when
// accumulate != 0.
// Forward and backward of 4,096 samples (F = 24, H = 128): 125 -> 43 us.
constexpr int kBwdUnits = 8, kBwdSplit = 8;

template <int FP>
__global__ void __cluster_dims__(kBwdSplit, 1, 1) __launch_bounds__(32 * kBwdUnits)
    mlp_backward_kernel(MlpWeights w, const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t B,
                        const float* __restrict__ pre, const float* __restrict__ dy, const float* __restrict__ sq,
                        float* __restrict__ grad, float* __restrict__ loss, int accumulate) {
  namespace cg = cooperative_groups;
  constexpr int FQ = FP / 4;                               // features per warp
  constexpr int XPT = (32 * FP) / (32 * kBwdUnits);        // staged features per thread
  __shared__ float xt[32][FP + 1];
  __shared__ float dzs[kBwdUnits][32];
  __shared__ float part[kBwdUnits][FP + 2];  // dW1 row, db1, dw2
  __shared__ double part2[2];                // sum of dy, sum of squared errors
  cg::cluster_group cluster = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = (int)cluster.block_rank();
  const int j0 = (int)(blockIdx.x / kBwdSplit) * kBwdUnits;
  const int j = j0 + warp;
  const bool unit = j < w.H;
  const float w2j = unit ? __bfloat162float(w.w2[j]) : 0.f;
  const int u0 = (warp >> 2) * 4, f0 = (warp & 3) * FQ;
  float acc[4][FQ];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int f = 0; f < FQ; ++f) acc[q][f] = 0.f;
  float gb1 = 0.f, gw2 = 0.f;
  double sdy = 0.0, ssq = 0.0;  // (the warp of unit 0 alone)
  float z = 0.f, d = 0.f, e2 = 0.f, xr[XPT];
  auto fetch = [&](int64_t s0) {
    const int64_t s = s0 + lane;
    const bool in = s < B;
    z = in && unit ? pre[(int64_t)j * B + s] : 0.f;
    d = in ? dy[s] : 0.f;
    e2 = in && j == 0 ? sq[s] : 0.f;
#pragma unroll
    for (int q = 0; q < XPT; ++q) {
      const int i = threadIdx.x + q * 32 * kBwdUnits;
      const int r = i / FP, f = i - r * FP;
      xr[q] = 0.f;
      if (s0 + r < B && f < w.F) xr[q] = X[(idx ? idx[s0 + r] : s0 + r) * w.F + f];
    }
  };
  const int64_t step = 32 * kBwdSplit;
  fetch(32 * rank);
  for (int64_t s0 = 32 * rank; s0 < B; s0 += step) {
    const float dz = d * w2j * gelu_grad_f(z);
    gb1 += dz;
    gw2 = fmaf(d, gelu_f(z), gw2);
    if (j == 0) {
      sdy += d;
      ssq += e2;
    }
    dzs[warp][lane] = dz;
#pragma unroll
    for (int q = 0; q < XPT; ++q) {
      const int i = threadIdx.x + q * 32 * kBwdUnits;
      xt[i / FP][i % FP] = xr[q];
    }
    __syncthreads();
    if (s0 + step < B) fetch(s0 + step);
    float g[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) g[q] = dzs[u0 + q][lane];
#pragma unroll
    for (int f = 0; f < FQ; ++f) {
      const float x = xt[lane][f0 + f];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q][f] = fmaf(g[q], x, acc[q][f]);
    }
    __syncthreads();
  }
  auto lanes = [](auto v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int f = 0; f < FQ; ++f) {
      const float v = lanes(acc[q][f]);
      if (lane == 0) part[u0 + q][f0 + f] = v;
    }
  gb1 = lanes(gb1);
  gw2 = lanes(gw2);
  if (j == 0) {
    sdy = lanes(sdy);
    ssq = lanes(ssq);
  }
  if (lane == 0) {
    part[warp][FP] = gb1;
    part[warp][FP + 1] = gw2;
    if (warp == 0) {
      part2[0] = sdy;
      part2[1] = ssq;
    }
  }
  cluster.sync();
  // block `rank` adds up unit j0 + rank, in block order
  const int jr = j0 + rank, f = threadIdx.x;
  static_assert(kBwdUnits == kBwdSplit && FP + 2 <= 32 * kBwdUnits, "one unit per block, one entry per thread");
  if (jr < w.H && f < FP + 2) {
    double sum = 0.0;
    for (int q = 0; q < kBwdSplit; ++q) sum += cluster.map_shared_rank(&part[0][0], q)[rank * (FP + 2) + f];
    const float v = (float)sum;
    if (f < w.F) grad[jr * w.F + f] = v;
    else if (f == FP) grad[w.H * w.F + jr] = v;
    else if (f == FP + 1) grad[w.H * w.F + w.H + jr] = v;
  }
  if (jr == 0 && f < 2) {
    double sum = 0.0;
    for (int q = 0; q < kBwdSplit; ++q) sum += cluster.map_shared_rank(part2, q)[f];
    if (f == 0) grad[w.H * w.F + 2 * w.H] = (float)sum;
    else if (loss) loss[0] = (accumulate ? loss[0] : 0.f) + (float)(sum / (double)B);
  }
  cluster.sync();  // the other blocks' sums stay readable until all are done
}

// AdamW on the FP32 master parameters (flat: W1, b1, w2, b2), then the BF16
// copies of W1 and w2 the forward reads.
__global__ void adamw_kernel(MlpWeights w, const float* __restrict__ grad, float* __restrict__ master,
                             float* __restrict__ m1, float* __restrict__ m2, int64_t step, float lr, float beta1,
                             float beta2, float eps, float wd) {
  const int P = w.H * w.F + 2 * w.H + 1;
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    const float g = grad[i];
    const float a = beta1 * m1[i] + (1.0f - beta1) * g;
    const float b = beta2 * m2[i] + (1.0f - beta2) * g * g;
    m1[i] = a;
    m2[i] = b;
    const float p = master[i] * (1.0f - lr * wd) - lr * (a / c1) / (sqrtf(b / c2) + eps);
    master[i] = p;
    if (i < w.H * w.F) w.W1[i] = __float2bfloat16_rn(p);
    else if (i < w.H * w.F + w.H) w.b1[i - w.H * w.F] = p;
    else if (i < w.H * w.F + 2 * w.H) w.w2[i - w.H * w.F - w.H] = __float2bfloat16_rn(p);
    else w.b2[0] = p;
  }
}

// the kernels by the number of features rounded up to 8
template <class Fn>
static cudaError_t by_features(int F, Fn&& go) {
  static_assert(kMaxFeatures == 32, "padded feature counts");
  if (F <= 8) return go(std::integral_constant<int, 8>());
  if (F <= 16) return go(std::integral_constant<int, 16>());
  if (F <= 24) return go(std::integral_constant<int, 24>());
  if (F <= 32) return go(std::integral_constant<int, 32>());
  return cudaErrorInvalidValue;
}

cudaError_t launch_mlp_forward(const MlpWeights& w, const float* X, const int64_t* idx, int64_t B, float* y, float* pre,
                               const float* t, float* dy, float* sq, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  // the widest network: its weights, unpadded, in 48 KB
  if ((size_t)(w.H * w.F + 2 * w.H) * sizeof(float) > 48 * 1024) return cudaErrorInvalidValue;
  int64_t blocks = (B + 31) / 32;
  if (blocks > 152 * 8) blocks = 152 * 8;
  return by_features(w.F, [&](auto fp) -> cudaError_t {
    constexpr int FP = decltype(fp)::value;
    const size_t smem = (size_t)(w.H * FP + 2 * w.H) * sizeof(float);
    auto kern = mlp_forward_kernel<FP>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)blocks, 32 * kMlpWarps, smem, st>>>(w, X, idx, B, y, pre, t, dy, sq);
    return cudaGetLastError();
  });
}

cudaError_t launch_mlp_backward(const MlpWeights& w, const float* X, const int64_t* idx, int64_t B, const float* pre,
                                const float* dy, const float* sq, float* grad, float* loss, int accumulate,
                                cudaStream_t st) {
  return by_features(w.F, [&](auto fp) -> cudaError_t {
    constexpr int FP = decltype(fp)::value;
    const int clusters = (w.H + kBwdUnits - 1) / kBwdUnits;
    mlp_backward_kernel<FP><<<clusters * kBwdSplit, 32 * kBwdUnits, 0, st>>>(w, X, idx, B, pre, dy, sq, grad, loss,
                                                                              accumulate);
    return cudaGetLastError();
  });
}

cudaError_t launch_adamw(const MlpWeights& w, const float* grad, float* master, float* m1, float* m2, int64_t step,
                         float lr, float beta1, float beta2, float eps, float wd, cudaStream_t st) {
  const int P = w.H * w.F + 2 * w.H + 1;
  adamw_kernel<<<(P + 255) / 256, 256, 0, st>>>(w, grad, master, m1, m2, step, lr, beta1, beta2, eps, wd);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- pruning

// Per read, keep the `keep` candidates with the smallest predicted distance
// (ties: better scan score, then lower start). Missing candidates are skipped.
__global__ void prune_kernel(const int64_t* __restrict__ cand_win, const float* __restrict__ cand_score,
                             const float* __restrict__ pred, int64_t n_reads, int K, int keep,
                             int64_t* __restrict__ out_win, float* __restrict__ out_score,
                             float* __restrict__ out_pred) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n_reads; r += (int64_t)gridDim.x * blockDim.x) {
    uint64_t taken = 0;
    for (int q = 0; q < keep; ++q) {
      int best = -1;
      for (int c = 0; c < K; ++c) {
        if ((taken >> c) & 1ull) continue;
        const int64_t wc = cand_win[r * K + c];
        if (wc < 0) continue;
        if (best < 0) {
          best = c;
          continue;
        }
        const float pc = pred[r * K + c], pb = pred[r * K + best];
        const float sc = cand_score[r * K + c], sb = cand_score[r * K + best];
        if (pc < pb || (pc == pb && (sc > sb || (sc == sb && wc < cand_win[r * K + best])))) best = c;
      }
      if (best >= 0) {
        taken |= 1ull << best;
        out_win[r * keep + q] = cand_win[r * K + best];
        out_score[r * keep + q] = cand_score[r * K + best];
        if (out_pred) out_pred[r * keep + q] = pred[r * K + best];
      } else {
        out_win[r * keep + q] = -1;
        out_score[r * keep + q] = -INFINITY;
        if (out_pred) out_pred[r * keep + q] = INFINITY;
      }
    }
  }
}

cudaError_t launch_prune(const int64_t* cand_win, const float* cand_score, const float* pred, int64_t n_reads, int K,
                         int keep, int64_t* out_win, float* out_score, float* out_pred, cudaStream_t st) {
  if (n_reads <= 0) return cudaSuccess;
  int64_t blocks = (n_reads + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  prune_kernel<<<(unsigned)blocks, 256, 0, st>>>(cand_win, cand_score, pred, n_reads, K, keep, out_win, out_score,
                                                  out_pred);
  return cudaGetLastError();
}

}  // namespace rope

namespace rope {

__global__ void ld_fraction_kernel(const int32_t* __restrict__ ld, int64_t n, float inv_n, float* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (float)ld[i] * inv_n;
}

cudaError_t launch_ld_fraction(const int32_t* ld, int64_t n, int N, float* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  ld_fraction_kernel<<<(unsigned)blocks, 256, 0, st>>>(ld, n, 1.0f / (float)N, out);
  return cudaGetLastError();
}

// The fallback without a network: candidate c of every read is given the
// "prediction" c, so pruning keeps the scan's own ranking.
__global__ void rank_prediction_kernel(int64_t n_reads, int K, float* __restrict__ pred) {
  const int64_t n = n_reads * K;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    pred[i] = (float)(i % K);
}

cudaError_t launch_rank_as_prediction(int64_t n_reads, int K, float* pred, cudaStream_t st) {
  const int64_t n = n_reads * K;
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  rank_prediction_kernel<<<(unsigned)blocks, 256, 0, st>>>(n_reads, K, pred);
  return cudaGetLastError();
}

}  // namespace rope
