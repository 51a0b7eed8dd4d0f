// FP32 CUDA-core scan ("plain" path).
//
// A thread holds one or two reads' normalised vectors in registers; the
// block's eight warps generate tiles of window vectors on chip (chains of D/4
// lanes running the §3.4 recurrence from exact anchors), normalise them by the
// stored 1/sqrt(C_j) and stage them in shared memory; every thread then forms
// Re and Im of <x|c> for each window (the §4 real identity) and the fidelity
// Re^2 + Im^2, keeping its reads' best windows in shared-memory lists.
//
// Bounds: 4D multiply-adds per read and window on the FP32 units, and the
// windows' rows as broadcasts from shared memory (a 16-byte load takes four of
// the SM's 128-byte cycles whether its lanes agree or not): with one read per
// thread the loads take twice the multiply-adds' time, with two the same. The
// multiply-adds run as pairs (fma.rn.f32x2 over consecutive entries: the bits of
// separate sums over even and odd entries), four windows at a time.
// 500 reads x 2 M windows (d = 64, 8 candidates): 10.4 ms with one read per
// thread and unbounded lists, 9.7 ms with two, 8.0 ms with bounded lists; what
// is left beside the multiply-adds is the updates of each list's first windows.
// Small calls have neither (256 reads or fewer keep one read per thread, and a
// block with a single item has no earlier list to bound it by): 256 reads x
// 500,000 windows 1.66 -> 1.40 ms, 64 reads x 20,000 0.89 -> 0.83 ms.
#include "rope_internal.h"
#include "rope_topk.cuh"

namespace rope {

constexpr int kF32Threads = 256;  // reads per group
constexpr int kF32Steps = 8;      // windows per chain per tile
constexpr int kF32Batch = 4;      // windows scored together
static_assert(kF32Steps % kF32Batch == 0, "a batch's windows belong to one chain");

constexpr uint64_t kNegPair = 0x8000000080000000ull;  // flips the signs of a pair

// two FP32 values in one 64-bit register, lo in the low half
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float f32x2_sum(uint64_t v) {
  return __uint_as_float((uint32_t)v) + __uint_as_float((uint32_t)(v >> 32));
}

template <int D>
struct F32Shape {
  static constexpr int LPC = D / 4;
  static constexpr int CPW = 32 / LPC;
  static constexpr int C = (kF32Threads / 32) * CPW;  // chains per block
  static constexpr int TW = C * kF32Steps;            // windows per tile
  static constexpr int SUP = C * kAnchorPeriod;       // windows per super-tile
  static constexpr size_t kTileBytes = (size_t)TW * 2 * D * sizeof(float);
};

// R reads per thread: read slots tid and tid + kF32Threads of the group
template <int D, int R, bool kDense, bool kPerBand>
__global__ void __launch_bounds__(kF32Threads) scan_fp32_kernel(DevIndex ix, ScanArgs a) {
  using Sh = F32Shape<D>;
  constexpr int kGroup = R * kF32Threads;
  // writing every score at few entries is bound by the stores: 300 reads x 500,000
  // windows at D = 4 3.5 ms by range, 4.0 ms by group; at D = 32 0.64 and 0.56 ms
  // (300 reads x 20,000)
  constexpr bool kByRange = kDense && D < 32;
  static_assert(R == 1 || !kPerBand, "per-band scores take one read per thread");
  extern __shared__ __align__(16) uint8_t f32_smem[];
  float* tile = reinterpret_cast<float*>(f32_smem);
  float* list_s = reinterpret_cast<float*>(f32_smem + Sh::kTileBytes);
  uint32_t* list_w = reinterpret_cast<uint32_t*>(list_s + (size_t)a.cand_depth * kGroup);

  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int lic = lane % Sh::LPC;
  const int chain = warp * Sh::CPW + lane / Sh::LPC;
  const int S = ix.stride;
  const int n_items = a.n_groups * a.n_ranges;

  ThreadList lst[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    lst[i].s = list_s + tid + i * kF32Threads;
    lst[i].w = list_w + tid + i * kF32Threads;
    lst[i].stride = kGroup;
    lst[i].depth = a.cand_depth;
  }

  Chain<D> ch;
  ch.setup(ix, lic);

  // A contiguous run of items per block. With one read per thread an SM holds two
  // blocks or more (but at D = 64), and the first blocks, which lie on SMs of their
  // own, take the items left over (4,000 reads x 100,000 windows at D = 16: 2.2 ms,
  // 2.8 ms with them spread over the blocks); with two it holds one block, and they
  // are spread (1,000 reads x 8 M at D = 32: 48.1 ms, 49.1 ms with the first blocks).
  // The items are in group-major order, so that most of a block's items share
  // their reads, or (kByRange) with the groups of a range side by side, so that
  // full and partly filled groups mix over the SMs.
  int it_lo, it_hi;
  if (R == 1) {
    const int per_block = n_items / (int)gridDim.x, left_over = n_items % (int)gridDim.x;
    it_lo = (int)blockIdx.x * per_block + min((int)blockIdx.x, left_over);
    it_hi = it_lo + per_block + ((int)blockIdx.x < left_over ? 1 : 0);
  } else {
    it_lo = (int)((int64_t)n_items * blockIdx.x / gridDim.x);
    it_hi = (int)((int64_t)n_items * (blockIdx.x + 1) / gridDim.x);
  }
  // Every range has lists of its own, and a list taking its first windows is
  // mostly updates. A list that two earlier lists of the read beat with all
  // their entries cannot add to the merge_depth best of the union, so a window
  // below the second-largest worst entry of the lists done so far is passed by
  // (with buckets, sep > 0, entries of two lists may be one: no bound).
  const bool bounded = !kDense && a.sep == 0 && 2 * a.cand_depth >= a.merge_depth;
  float first[R], bound[R];  // the two largest worst entries
  int prev_grp = -1;

  for (int item = it_lo; item < it_hi; ++item) {
    const int grp = kByRange ? item % a.n_groups : item / a.n_ranges;
    const int rng = kByRange ? item / a.n_groups : item % a.n_ranges;
    const int64_t r = (int64_t)grp * kGroup + tid;  // read of slot i: r + i * kF32Threads
    const bool have_read = r < a.n_reads;
    const int64_t st_begin = a.st0 + (int64_t)rng * a.range_len;
    const int64_t j_lo = max(st_begin, a.jb);
    const int64_t j_hi = min(st_begin + a.range_len, a.je);

    // the reads' vectors, normalised (per band in score mode 1)
    float xr[R][D], xi[R][D];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int64_t ri = r + i * kF32Threads;
      const bool have = ri < a.n_reads;
      const float* e = a.emb_f32 + (have ? ri : 0) * 2 * D;
      const float* nr = a.norms + (have ? ri : 0) * (1 + ix.m);
      float inv = 0.f;
      if (!kPerBand) {
        const float X = nr[0];
        inv = (have && X > kZeroNorm2) ? rsqrtf(X) : 0.f;
      }
#pragma unroll
      for (int g = 0; g < D; ++g) {
        float sc = inv;
        if (kPerBand) {
          const float Xk = nr[1 + g / ix.nb];
          sc = (have && Xk > kZeroNorm2) ? rsqrtf(Xk) : 0.f;
        }
        xr[i][g] = e[g] * sc;
        xi[i][g] = e[D + g] * sc;
      }
      if (!kDense) {
        if (grp != prev_grp) first[i] = bound[i] = -INFINITY;
        lst[i].reset();
        lst[i].thr = have ? bound[i] : INFINITY;  // a missing read's list takes nothing
      }
    }

    prev_grp = grp;

    for (int64_t st = st_begin; st < j_hi; st += Sh::SUP) {
      const int64_t a_idx = st / ix.A + chain;
      const bool chain_live = a_idx * ix.A < ix.W;
      if (chain_live) {
        ch.load(ix.anchors + a_idx * D, lic);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) ch.cr[i] = ch.ci[i] = 0.f;
      }
      for (int rd = 0; rd < kAnchorPeriod / kF32Steps; ++rd) {
        // ---- generate kF32Steps windows per chain into the tile
#pragma unroll 1
        for (int u = 0; u < kF32Steps; ++u) {
          const int64_t j = st + (int64_t)chain * ix.A + rd * kF32Steps + u;
          const bool live = chain_live && j < ix.W;
          float* row = tile + (size_t)(chain * kF32Steps + u) * 2 * D;
          float4 vr, vi;
          if (!kPerBand) {
            const float inv = live ? ix.inv_norm[j] : 0.f;
            vr = make_float4(ch.cr[0] * inv, ch.cr[1] * inv, ch.cr[2] * inv, ch.cr[3] * inv);
            vi = make_float4(ch.ci[0] * inv, ch.ci[1] * inv, ch.ci[2] * inv, ch.ci[3] * inv);
          } else {
            const float Ck = live ? ix.band_norm[j * ix.m + ch.band] : 0.f;
            const float inv = Ck > kZeroNorm2 ? rsqrtf(Ck) : 0.f;
            vr = make_float4(ch.cr[0] * inv, ch.cr[1] * inv, ch.cr[2] * inv, ch.cr[3] * inv);
            vi = make_float4(ch.ci[0] * inv, ch.ci[1] * inv, ch.ci[2] * inv, ch.ci[3] * inv);
          }
          reinterpret_cast<float4*>(row)[lic] = vr;
          reinterpret_cast<float4*>(row + D)[lic] = vi;
          if (live) {
            const int64_t w = j * S;
            if (S == 1) {
              ch.step1(bin_at(ix.packed, w, ix.s, ix.map_lsb),
                       bin_at(ix.packed, w + ix.N - ix.s + 1, ix.s, ix.map_lsb));
            } else {
              for (int q = 0; q < S; ++q) {
                ch.sub_at(bin_at(ix.packed, w + q, ix.s, ix.map_lsb), ix.eout[ch.band * S + q]);
                ch.add_at(bin_at(ix.packed, w + ix.N - ix.s + 1 + q, ix.s, ix.map_lsb), ix.ein[ch.band * S + q]);
              }
              ch.rotate();
            }
          }
        }
        __syncthreads();
        // ---- score every window of the tile against this thread's read
        if (have_read) {
#pragma unroll 1
          for (int q = 0; q < Sh::TW; q += kF32Batch) {
            float sc[R][kF32Batch];
            if (!kPerBand) {
              // Re and -Im of each window, even and odd entries in the halves of a pair
              const ulonglong2* c = reinterpret_cast<const ulonglong2*>(tile + (size_t)q * 2 * D);
              uint64_t re[R][kF32Batch], im[R][kF32Batch];
#pragma unroll
              for (int i = 0; i < R; ++i)
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) re[i][h] = im[i][h] = 0;
#pragma unroll
              for (int e4 = 0; e4 < D / 4; ++e4)
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) {
                  const ulonglong2 cr = c[h * (2 * D / 4) + e4], ci = c[h * (2 * D / 4) + D / 4 + e4];
                  const uint64_t nx = ci.x ^ kNegPair, ny = ci.y ^ kNegPair;
#pragma unroll
                  for (int i = 0; i < R; ++i) {
                    const uint64_t r0 = f32x2(xr[i][4 * e4], xr[i][4 * e4 + 1]), r1 = f32x2(xr[i][4 * e4 + 2], xr[i][4 * e4 + 3]);
                    const uint64_t i0 = f32x2(xi[i][4 * e4], xi[i][4 * e4 + 1]), i1 = f32x2(xi[i][4 * e4 + 2], xi[i][4 * e4 + 3]);
                    re[i][h] = fma_f32x2(r0, cr.x, fma_f32x2(i0, ci.x, re[i][h]));
                    im[i][h] = fma_f32x2(r0, nx, fma_f32x2(i0, cr.x, im[i][h]));
                    re[i][h] = fma_f32x2(r1, cr.y, fma_f32x2(i1, ci.y, re[i][h]));
                    im[i][h] = fma_f32x2(r1, ny, fma_f32x2(i1, cr.y, im[i][h]));
                  }
                }
#pragma unroll
              for (int i = 0; i < R; ++i)
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) {
                  const float vr = f32x2_sum(re[i][h]), vi = f32x2_sum(im[i][h]);
                  sc[i][h] = fmaf(vr, vr, vi * vi);
                }
            } else {
#pragma unroll
              for (int h = 0; h < kF32Batch; ++h) sc[0][h] = 0.f;
              const float* t0 = tile + (size_t)q * 2 * D;
              for (int k = 0; k < ix.m; ++k) {
                float re[kF32Batch], im[kF32Batch];
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) re[h] = im[h] = 0.f;
#pragma unroll
                for (int g = 0; g < D; ++g) {
                  if (g / ix.nb != k) continue;
#pragma unroll
                  for (int h = 0; h < kF32Batch; ++h) {
                    const float cr = t0[h * 2 * D + g], ci = t0[h * 2 * D + D + g];
                    re[h] = fmaf(xr[0][g], cr, fmaf(xi[0][g], ci, re[h]));
                    im[h] = fmaf(xr[0][g], ci, fmaf(-xi[0][g], cr, im[h]));
                  }
                }
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) sc[0][h] += fmaf(re[h], re[h], im[h] * im[h]);
              }
#pragma unroll
              for (int h = 0; h < kF32Batch; ++h) sc[0][h] /= ix.m;
            }
            // window numbers of tile slots q .. q+kF32Batch-1 (of one chain)
            const int64_t jq = st + (int64_t)(q / kF32Steps) * ix.A + rd * kF32Steps + (q % kF32Steps);
#pragma unroll
            for (int i = 0; i < R; ++i) {
              if (kDense) {
                const int64_t ri = r + i * kF32Threads;
                if (ri >= a.n_reads) continue;
#pragma unroll
                for (int h = 0; h < kF32Batch; ++h) {
                  const int64_t j = jq + h;
                  if (j >= j_lo && j < j_hi) a.dense[ri * (a.je - a.jb) + (j - a.jb)] = sc[i][h];
                }
              } else {
                float top = sc[i][0];
#pragma unroll
                for (int h = 1; h < kF32Batch; ++h) top = fmaxf(top, sc[i][h]);
                if (top < lst[i].thr) continue;
                // (with two reads the updates' code, eight times over, costs more than
                // picking each window's score: 8.8 against 8.0 ms at 500 reads x 2 M
                // windows; with one read unrolled is the faster, 0.83 against 0.97 ms
                // at 64 reads x 20,000, but per band, D = 64 and 700 reads x 500,000,
                // 31 against 26 ms)
#pragma unroll(R == 1 && !(kPerBand && D == 64) ? kF32Batch : 1)
                for (int h = 0; h < kF32Batch; ++h) {
                  const int64_t j = jq + h;
                  float v = sc[i][0];
#pragma unroll
                  for (int u = 1; u < kF32Batch; ++u) v = h == u ? sc[i][u] : v;
                  if (j >= j_lo && j < j_hi && v >= lst[i].thr) {
                    lst[i].insert(v, (uint32_t)j, a.sep, S);
                    lst[i].thr = fmaxf(lst[i].thr, bound[i]);
                  }
                }
              }
            }
          }
        }
        __syncthreads();
      }
    }
    if (!kDense) {
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int64_t ri = r + i * kF32Threads;
        if (ri >= a.n_reads) continue;
        Candidate* out = a.cand + ((size_t)ri * a.n_ranges + rng) * a.cand_depth;
        for (int e = 0; e < a.cand_depth; ++e) out[e] = Candidate{lst[i].S(e), lst[i].Wn(e)};
        const float worst = lst[i].S(lst[i].worst);  // -inf: not full
        if (bounded) {
          bound[i] = fmaxf(bound[i], fminf(first[i], worst));
          first[i] = fmaxf(first[i], worst);
        }
      }
    }
  }
}

int scan_fp32_supported(int D) { return D == 4 || D == 8 || D == 16 || D == 32 || D == 64; }

int64_t scan_fp32_super_tile(int D) {
  switch (D) {
    case 4: return F32Shape<4>::SUP;
    case 8: return F32Shape<8>::SUP;
    case 16: return F32Shape<16>::SUP;
    case 32: return F32Shape<32>::SUP;
    case 64: return F32Shape<64>::SUP;
  }
  return 0;
}

int scan_fp32_group() { return kF32Threads; }

// Two reads per thread (one generation of a window, and one read of it from
// shared memory, then serve 512 reads instead of 256) where that pays:
//   * at D = 32: with fewer entries it was 1.1 to 2.3 times slower almost
//     throughout, and at D = 64 two reads' vectors do not fit in registers;
//   * with four items per SM or more, to even out their ends: 500 reads x 1 M windows
//     (489 items) 5.1 ms against 4.4 with one read, 2,600 x 500,000 (738) 10.3 against
//     10.9, 500 x 2 M (977) 8.0 against 8.3. Writing every score there are no lists
//     to fill, and more groups of 256 times ranges than SMs are enough: 1,024 reads x
//     100,000 1.2 against 1.5 ms, 500 reads 0.95 against 0.57;
//   * with no half group idle, or a 12th at most: 700 reads x 2 M (three groups of
//     256) 13.9 against 11.1 ms, 1,100 reads (five) 20.2 against 17.3, 2,600 (eleven)
//     35.4 against 37.4.
int scan_fp32_reads_per_thread(const DevIndex& ix, int64_t n_reads, int n_ranges, int num_sms, bool dense) {
  if (ix.D != 32 || ix.score_mode != 0) return 1;
  const int64_t g1 = (n_reads + kF32Threads - 1) / kF32Threads, g2 = (g1 + 1) / 2;
  if (11 * 2 * g2 > 12 * g1) return 1;
  return (dense ? g1 * n_ranges > num_sms : g2 * n_ranges >= 4 * num_sms) ? 2 : 1;
}

template <int D, int R, bool kDense, bool kPerBand>
static cudaError_t launch_one(const DevIndex& ix, const ScanArgs& a, int num_sms, cudaStream_t st) {
  using Sh = F32Shape<D>;
  const size_t smem = Sh::kTileBytes + (kDense ? 0 : (size_t)a.cand_depth * kF32Threads * R * 8);
  auto kern = scan_fp32_kernel<D, R, kDense, kPerBand>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kF32Threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  const int n_items = a.n_groups * a.n_ranges;
  int grid = num_sms * per_sm;
  if (grid > n_items) grid = n_items;
  if (grid < 1) return cudaSuccess;
  kern<<<grid, kF32Threads, smem, st>>>(ix, a);
  return cudaGetLastError();
}

template <bool kDense, bool kPerBand>
static cudaError_t dispatch(const DevIndex& ix, const ScanArgs& a, int num_sms, cudaStream_t st) {
  switch (ix.D) {
    case 4: return launch_one<4, 1, kDense, kPerBand>(ix, a, num_sms, st);
    case 8: return launch_one<8, 1, kDense, kPerBand>(ix, a, num_sms, st);
    case 16: return launch_one<16, 1, kDense, kPerBand>(ix, a, num_sms, st);
    case 32:
      if constexpr (!kPerBand) {
        // fewer groups than of 256 reads each: the plan took two reads per thread
        if ((int64_t)a.n_groups * kF32Threads < a.n_reads) return launch_one<32, 2, kDense, kPerBand>(ix, a, num_sms, st);
      }
      return launch_one<32, 1, kDense, kPerBand>(ix, a, num_sms, st);
    case 64: return launch_one<64, 1, kDense, kPerBand>(ix, a, num_sms, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_scan_fp32(const DevIndex& ix, const ScanArgs& a, bool dense, int num_sms, cudaStream_t st) {
  const bool pb = ix.score_mode == 1;
  if (dense) return pb ? dispatch<true, true>(ix, a, num_sms, st) : dispatch<true, false>(ix, a, num_sms, st);
  return pb ? dispatch<false, true>(ix, a, num_sms, st) : dispatch<false, false>(ix, a, num_sms, st);
}

}  // namespace rope
