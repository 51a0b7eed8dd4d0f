// Encoding kernels: 2-bit packing, s-mer bins, read-head encodings (direct
// summation), the FP64 reference pre-pass (anchors and exact window norms) and
// the window-embedding inspection kernel.
#include <cuda_bf16.h>

#include <type_traits>

#include "rope_internal.h"

namespace rope {

// ---------------------------------------------------------------- a1: packing

// Four letters (one byte each) to four 2-bit codes in one byte, a word at a
// time. Bits 1-2 of an ASCII letter are 0,1,3,2 for A,C,G,T (either case), a
// Gray code: x ^ (x >> 1) turns them into 0,1,2,3. The letters are then
// checked by rebuilding each byte's lower-case letter from its code
// ('a' + {0, 2, 6, 19}) and comparing with the input folded to lower case;
// any difference, accumulated in `bad`, marks a letter outside ACGTacgt. The
// multiply gathers the byte-spaced codes into the top byte (the partial
// products of different bytes land in disjoint bits below it).
__device__ __forceinline__ uint32_t pack4(uint32_t x, uint32_t& bad) {
  const uint32_t g = (x >> 1) & 0x03030303u;
  const uint32_t code = g ^ ((g >> 1) & 0x01010101u);
  const uint32_t hi = (code >> 1) & 0x01010101u;           // code >= 2
  const uint32_t three = hi & code;                         // code == 3
  const uint32_t letter = 0x61616161u + ((code + hi) << 1) + three * 11u;
  bad |= (x | 0x20202020u) ^ letter;
  return (code * 0x01041040u) >> 24;
}

// One output word (16 letters) per thread; 16-byte vector loads when aligned.
// HBM-bound: 1 byte in and 1/4 byte out per letter.
// One thread packs kPackWords consecutive 16-letter words per step: their
// four 16-byte loads are issued together, so enough bytes are in flight to
// keep HBM busy; the ragged tail and unaligned inputs take the byte path.
constexpr int kPackWords = 4;

__device__ __forceinline__ uint32_t pack_bytes(const uint8_t* seq, int64_t base, int64_t len, uint32_t& bad) {
  uint32_t word = 0;
  for (int i = 0; i < 16 && base + i < len; ++i) {
    const uint32_t c = letter_code(seq[base + i]);
    bad |= (c > 3);
    word |= (c & 3u) << (2 * i);
  }
  return word;
}

__global__ void pack_kernel(const uint8_t* __restrict__ seq, int64_t len, uint32_t* __restrict__ out,
                            int64_t n_words, int* status) {
  // vector loads and stores need 16-byte aligned input and output
  const bool aligned = ((((uintptr_t)seq) | ((uintptr_t)out)) & 15u) == 0;
  uint32_t bad = 0;
  const int64_t n_groups = (n_words + kPackWords - 1) / kPackWords;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n_groups;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w0 = g * kPackWords;
    if (aligned && (w0 + kPackWords) * 16 <= len) {
      uint4 v[kPackWords];
#pragma unroll
      for (int q = 0; q < kPackWords; ++q) v[q] = __ldg(reinterpret_cast<const uint4*>(seq + (w0 + q) * 16));
      uint32_t wd[kPackWords];
#pragma unroll
      for (int q = 0; q < kPackWords; ++q)
        wd[q] = pack4(v[q].x, bad) | (pack4(v[q].y, bad) << 8) | (pack4(v[q].z, bad) << 16) |
                (pack4(v[q].w, bad) << 24);
      *reinterpret_cast<uint4*>(out + w0) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
    } else {
      for (int q = 0; q < kPackWords && w0 + q < n_words; ++q) out[w0 + q] = pack_bytes(seq, (w0 + q) * 16, len, bad);
    }
  }
  if (bad) set_status(status, kStatusBadBase);
}

cudaError_t launch_pack(const uint8_t* seq, int64_t len, uint32_t* out, int* status, cudaStream_t st) {
  const int64_t n_words = (len + 15) / 16;
  if (n_words == 0) return cudaSuccess;
  const int threads = 256;
  const int64_t n_groups = (n_words + kPackWords - 1) / kPackWords;
  int64_t blocks = (n_groups + threads - 1) / threads;
  if (blocks > 152 * 32) blocks = 152 * 32;
  pack_kernel<<<(unsigned)blocks, threads, 0, st>>>(seq, len, out, n_words, status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- a2: bins

__global__ void mer_bins_kernel(const uint32_t* __restrict__ packed, int64_t n_pos, int64_t n_words, int s,
                                const uint16_t* __restrict__ map_lsb, uint16_t* __restrict__ out) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n_pos; p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t wi = p >> 4;
    const uint32_t lo = packed[wi];
    const uint32_t hi = wi + 1 < n_words ? packed[wi + 1] : 0u;
    const uint64_t v = ((uint64_t)hi << 32) | lo;
    const uint32_t field = (uint32_t)(v >> ((p & 15) * 2)) & ((1u << (2 * s)) - 1u);
    out[p] = map_lsb[field];
  }
}

cudaError_t launch_mer_bins(const uint32_t* packed, int64_t len, int64_t n_words, int s, const uint16_t* map_lsb,
                            uint16_t* out, cudaStream_t st) {
  const int64_t n_pos = len - s + 1;
  if (n_pos <= 0) return cudaSuccess;
  int64_t blocks = (n_pos + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  mer_bins_kernel<<<(unsigned)blocks, 256, 0, st>>>(packed, n_pos, n_words, s, map_lsb, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- a3: read heads

// One warp per read. Locations are taken in order; for each location the
// lanes k < m add exp(2 pi i f_k loc / N) to entry (k, bin) of a per-warp
// shared accumulator, so every entry is summed in location order (the direct
// sum of §2.1-§2.3 in FP32, deterministic).
// Letter q (0..3, 4 if not ACGT) of the head of a read of length len: the read
// itself, or (rc) its reverse complement, whose head is the complement of the
// read's last letters read backwards.
__device__ __forceinline__ uint32_t head_letter(const uint8_t* seq, int64_t len, int q, bool rc) {
  if (!rc) return letter_code(seq[q]);
  const uint32_t c = letter_code(seq[len - 1 - q]);
  return c > 3 ? c : 3u - c;  // A<->T, C<->G
}

// One warp per read; lane l owns entries g = l, l + 32, ... of the D complex
// entries (band g / 4^t, bin g % 4^t) in registers. The locations are taken 32
// at a time, one per lane; warp ballots of the bits of their bins tell each
// lane which of the 32 locations fall in its entries' bins, and the lane adds
// e^{2 pi i f_k loc / N} (phase table staged in shared memory) for those
// locations in increasing order. Every entry is thus summed in location order
// (the direct sum of §2.1-§2.3 in FP32, deterministic), with a warp cost per
// 32 locations of a few ballots plus the largest bin's count.
constexpr int kEncMaxPerLane = kMaxScanDim / 32;
constexpr int kEncMaxBinBits = 8;  // bins per band up to 256

// rc: the heads of the reads' reverse complements. The strand belongs to the
// launch: chosen per read it sits in every letter's load, and 1,000,000 reads of
// 150 letters (d = 64) took 3.60 instead of 1.98 ms.
__global__ void encode_reads_kernel(EncTables tb, const uint8_t* __restrict__ seqs,
                                    const int64_t* __restrict__ offsets, int64_t n, float* __restrict__ emb_f32,
                                    __nv_bfloat16* __restrict__ emb_bf16, float* __restrict__ norms, int* status,
                                    const int64_t* __restrict__ perm, bool rc) {
  extern __shared__ float2 enc_phase[];  // [m * n_loc] phases, staged once per block
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const int n_loc = tb.N - tb.s + 1;
  const int E = (tb.D + 31) / 32;  // entries per lane
  const int bin_bits = 32 - __clz(tb.nb > 1 ? tb.nb - 1 : 1);
  for (int i = threadIdx.x; i < tb.m * n_loc; i += blockDim.x) enc_phase[i] = tb.phase[i];
  __syncthreads();
  int band[kEncMaxPerLane], bin[kEncMaxPerLane];
#pragma unroll
  for (int e = 0; e < kEncMaxPerLane; ++e) {
    const int g = lane + 32 * e;
    band[e] = g < tb.D ? g / tb.nb : 0;
    bin[e] = g < tb.D ? g % tb.nb : -1;  // -1: no entry
  }
  for (int64_t r = (int64_t)blockIdx.x * wpb + warp; r < n; r += (int64_t)gridDim.x * wpb) {
    const int64_t src = perm ? perm[r] : r;
    const int64_t start = offsets[src];
    const int64_t len = offsets[src + 1] - start;
    const uint8_t* seq = seqs + start;
    float ar[kEncMaxPerLane], ai[kEncMaxPerLane];
#pragma unroll
    for (int e = 0; e < kEncMaxPerLane; ++e) ar[e] = ai[e] = 0.f;
    bool ok = len >= tb.N;
    if (!ok) {
      if (lane == 0) set_status(status, kStatusShortRead);
    } else {
      int bad = 0;
      for (int i = lane; i < tb.N; i += 32) bad |= head_letter(seq, len, i, rc) > 3;
      if (__any_sync(0xffffffffu, bad)) {
        ok = false;
        if (lane == 0) set_status(status, kStatusBadBase);
      }
    }
    if (ok) {
      for (int loc0 = 0; loc0 < n_loc; loc0 += 32) {
        const int loc = loc0 + lane;
        uint32_t b = 0;
        if (loc < n_loc) {
          uint32_t code = 0;
          for (int i = 0; i < tb.s; ++i) code = code * 4u + (head_letter(seq, len, loc + i, rc) & 3u);
          b = (uint32_t)tb.map[code];
        }
        // bit planes of the 32 locations' bins: the locations whose bin is
        // B are the lanes that agree with B on every plane
        const uint32_t valid = __ballot_sync(0xffffffffu, loc < n_loc);
        uint32_t plane[kEncMaxBinBits];
#pragma unroll
        for (int i = 0; i < kEncMaxBinBits; ++i)
          plane[i] = i < bin_bits ? __ballot_sync(0xffffffffu, (b >> i) & 1u) : 0u;
#pragma unroll
        for (int e = 0; e < kEncMaxPerLane; ++e) {
          if (e >= E || bin[e] < 0) continue;
          uint32_t hit = valid;
#pragma unroll
          for (int i = 0; i < kEncMaxBinBits; ++i)
            if (i < bin_bits) hit &= ((bin[e] >> i) & 1) ? plane[i] : ~plane[i];
          const float2* ph_row = enc_phase + band[e] * n_loc + loc0;
          while (hit) {  // the matching locations in increasing order
            const int j = __ffs(hit) - 1;
            hit &= hit - 1u;
            const float2 ph = ph_row[j];
            ar[e] += ph.x;
            ai[e] += ph.y;
          }
        }
      }
    }
    // per-band squared norms, then the total
    float total = 0.f;
    for (int k = 0; k < tb.m; ++k) {
      float part = 0.f;
#pragma unroll
      for (int e = 0; e < kEncMaxPerLane; ++e)
        if (e < E && bin[e] >= 0 && band[e] == k) part = fmaf(ar[e], ar[e], fmaf(ai[e], ai[e], part));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lane == 0) norms[r * (1 + tb.m) + 1 + k] = part;
      total += part;
    }
    if (lane == 0) norms[r * (1 + tb.m)] = total;
    const float inv = total > kZeroNorm2 ? rsqrtf(total) : 0.f;
#pragma unroll
    for (int e = 0; e < kEncMaxPerLane; ++e) {
      const int g = lane + 32 * e;
      if (e >= E || g >= tb.D) continue;
      if (emb_f32) {
        emb_f32[r * 2 * tb.D + g] = ar[e];
        emb_f32[r * 2 * tb.D + tb.D + g] = ai[e];
      }
      if (emb_bf16) {
        emb_bf16[r * 2 * tb.D + g] = __float2bfloat16_rn(ar[e] * inv);
        emb_bf16[r * 2 * tb.D + tb.D + g] = __float2bfloat16_rn(ai[e] * inv);
      }
    }
  }
}

// Encodings wider than kMaxScanDim complex entries, or heads whose phase table
// exceeds what one block stages: one warp per read head, its D complex entries
// in shared memory. Locations are taken 32 at a time, one per lane; lanes whose
// locations fall in the same bin form a group (__match_any_sync), and the
// group's lowest lane (its first location) sums the group's phases in
// location order and adds that sum to the entry, so each entry receives one
// update per 32 locations, in location order (deterministic FP32 sums of the
// §2.1-§2.3 direct sum). The phases of kEncChunk locations are staged in
// shared memory once per block for all of its warps.
// A step of 32 locations is a chain (letters, s-mer codes, the bin table, which
// at 4^8 codes lies in L2, the group's sum), so letters are loaded three steps and
// bins one step ahead, codes come from bit planes of the letters, and only the
// groups' lowest lanes walk their group.
// 2,048 heads of 20,000 letters on both strands (s = 8, 4 bands of 256 bins)
// mapped against 30 Mbp, whole call: 3.75 ms with every lane following the
// largest group by shuffles and nothing loaded ahead, 2.49 ms so, and 1.89 ms
// with both strands in one launch and a block per SM that holds all of its heads.
constexpr int kEncChunk = 256;
constexpr int kEncWideWarps = 28;  // most warps of a block (72 registers a thread)

// bit i of v (i < 8) at bit 2i
__device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
  v = (v | (v << 4)) & 0x0F0Fu;
  v = (v | (v << 2)) & 0x3333u;
  return (v | (v << 1)) & 0x5555u;
}

__global__ void __launch_bounds__(32 * kEncWideWarps) encode_reads_wide_kernel(EncTables tb, const uint8_t* __restrict__ seqs,
                                    const int64_t* __restrict__ offsets, int64_t n, float* __restrict__ emb_f32,
                                    __nv_bfloat16* __restrict__ emb_bf16, float* __restrict__ norms, int* status,
                                    const int64_t* __restrict__ perm, int64_t n_fwd) {
  extern __shared__ float2 enc_sm[];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const int n_loc = tb.N - tb.s + 1;
  float2* ph = enc_sm;                                              // [m][kEncChunk]
  float2* acc = enc_sm + (size_t)tb.m * kEncChunk + (size_t)warp * tb.D;  // this warp's entries
  for (int64_t r0 = (int64_t)blockIdx.x * wpb; r0 < n; r0 += (int64_t)gridDim.x * wpb) {
    const int64_t r = r0 + warp;
    const bool live = r < n;
    const bool rc = live && r >= n_fwd;
    const int64_t src = !live ? 0 : rc ? r - n_fwd : perm ? perm[r] : r;
    const int64_t start = live ? offsets[src] : 0;
    const int64_t len = live ? offsets[src + 1] - start : 0;
    const uint8_t* seq = seqs + start;
    for (int g = lane; g < tb.D; g += 32) acc[g] = make_float2(0.f, 0.f);
    bool ok = live && len >= tb.N;
    if (live && !ok && lane == 0) set_status(status, kStatusShortRead);
    uint32_t bad = 0;
    auto letter = [&](int q) { return ok && q < tb.N ? head_letter(seq, len, q, rc) : 0u; };
    // bit planes of letters l0 .. l0+31 (lo) of the step whose bins come next;
    // those of the 32 letters behind come from `ahead`
    uint32_t ahead = letter(lane);
    bad |= ahead;
    uint32_t lo0 = __ballot_sync(0xffffffffu, ahead & 1u), lo1 = __ballot_sync(0xffffffffu, ahead & 2u);
    ahead = letter(32 + lane);
    uint32_t ahead2 = letter(64 + lane);
    // bin of location l0 + lane, called for l0 = 0, 32, ...
    auto next_bin = [&](int l0) -> uint32_t {
      bad |= ahead;
      const uint32_t hi0 = __ballot_sync(0xffffffffu, ahead & 1u), hi1 = __ballot_sync(0xffffffffu, ahead & 2u);
      ahead = ahead2;
      ahead2 = letter(l0 + 96 + lane);
      const uint32_t code = (spread_bits(__brev(__funnelshift_r(lo0, hi0, lane)) >> (32 - tb.s))) |
                            (spread_bits(__brev(__funnelshift_r(lo1, hi1, lane)) >> (32 - tb.s)) << 1);
      lo0 = hi0;
      lo1 = hi1;
      return l0 + lane < n_loc ? (uint32_t)__ldg(tb.map + code) : 0xFFFFFFFFu;
    };
    uint32_t bin = next_bin(0);
    for (int c0 = 0; c0 < n_loc; c0 += kEncChunk) {
      const int c1 = min(c0 + kEncChunk, n_loc);
      __syncthreads();  // every warp is done with the previous chunk's phases
      for (int i = threadIdx.x; i < tb.m * kEncChunk; i += blockDim.x) {
        const int k = i / kEncChunk, u = i - k * kEncChunk;
        if (c0 + u < c1) ph[i] = tb.phase[(size_t)k * n_loc + c0 + u];
      }
      __syncthreads();
      if (!ok) continue;
      for (int l0 = c0; l0 < c1; l0 += 32) {
        const uint32_t cur = bin;
        bin = next_bin(l0 + 32);
        const uint32_t grp = __match_any_sync(0xffffffffu, cur);
        if (cur != 0xFFFFFFFFu && (grp & ((1u << lane) - 1u)) == 0) {
          const float2* row = ph + (l0 - c0);
          for (int k0 = 0; k0 < tb.m; k0 += 4) {
            float2 sum[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[k] = make_float2(0.f, 0.f);
            for (uint32_t rest = grp; rest; rest &= rest - 1u) {  // the group's members in location order
              const int q = __ffs(rest) - 1;
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                if (k0 + k >= tb.m) continue;
                const float2 p = row[(k0 + k) * kEncChunk + q];
                sum[k].x += p.x;
                sum[k].y += p.y;
              }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (k0 + k >= tb.m) continue;
              float2& e = acc[(k0 + k) * tb.nb + cur];
              e.x += sum[k].x;
              e.y += sum[k].y;
            }
          }
        }
        __syncwarp();
      }
    }
    if (__any_sync(0xffffffffu, bad & 4u)) {  // a letter outside ACGT (code 4): an empty encoding
      if (lane == 0) set_status(status, kStatusBadBase);
      for (int g = lane; g < tb.D; g += 32) acc[g] = make_float2(0.f, 0.f);
    }
    __syncwarp();
    if (live) {
      // per-band squared norms, then the total
      float total = 0.f;
      for (int k = 0; k < tb.m; ++k) {
        float part = 0.f;
        for (int b = lane; b < tb.nb; b += 32) {
          const float2 a = acc[k * tb.nb + b];
          part = fmaf(a.x, a.x, fmaf(a.y, a.y, part));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) norms[r * (1 + tb.m) + 1 + k] = part;
        total += part;
      }
      if (lane == 0) norms[r * (1 + tb.m)] = total;
      const float inv = total > kZeroNorm2 ? rsqrtf(total) : 0.f;
      for (int g = lane; g < tb.D; g += 32) {
        const float2 a = acc[g];
        if (emb_f32) {
          emb_f32[r * 2 * tb.D + g] = a.x;
          emb_f32[r * 2 * tb.D + tb.D + g] = a.y;
        }
        if (emb_bf16) {
          emb_bf16[r * 2 * tb.D + g] = __float2bfloat16_rn(a.x * inv);
          emb_bf16[r * 2 * tb.D + tb.D + g] = __float2bfloat16_rn(a.y * inv);
        }
      }
    }
    __syncwarp();
  }
}

cudaError_t launch_encode_reads(const EncTables& tb, const uint8_t* seqs, const int64_t* offsets, int64_t n,
                                float* emb_f32, uint16_t* emb_bf16, float* norms, int* status, cudaStream_t st,
                                const int64_t* perm, int64_t n_rc) {
  if (n <= 0) return cudaSuccess;
  const size_t phase_bytes = (size_t)tb.m * (tb.N - tb.s + 1) * sizeof(float2);
  if (tb.D <= kMaxScanDim && phase_bytes <= 48 * 1024) {
    const int wpb = 8;
    auto grid = [](int64_t rows) {
      const int64_t blocks = (rows + wpb - 1) / wpb;
      return (unsigned)(blocks > 152 * 16 ? 152 * 16 : blocks);  // each block stages the phase table once
    };
    __nv_bfloat16* bf16 = reinterpret_cast<__nv_bfloat16*>(emb_bf16);
    encode_reads_kernel<<<grid(n), wpb * 32, phase_bytes, st>>>(tb, seqs, offsets, n, emb_f32, bf16, norms, status,
                                                                perm, false);
    if (n_rc > 0)
      encode_reads_kernel<<<grid(n_rc), wpb * 32, phase_bytes, st>>>(
          tb, seqs, offsets, n_rc, emb_f32 ? emb_f32 + n * 2 * tb.D : nullptr, bf16 ? bf16 + n * 2 * tb.D : nullptr,
          norms + n * (1 + tb.m), status, nullptr, true);
    return cudaGetLastError();
  }
  const int64_t n_fwd = n;
  n += n_rc;
  // A step is latency, so an SM wants as many heads at a time as it is going to
  // get: one block per SM with a warp for each of the SM's heads, or, where their
  // sums do not fit in its shared memory, an equal share in each wave.
  int dev = 0, sms = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  const size_t chunk_bytes = (size_t)tb.m * kEncChunk * sizeof(float2);
  int64_t most = ((size_t)optin - chunk_bytes) / (tb.D * sizeof(float2));
  if (most > kEncWideWarps) most = kEncWideWarps;
  if (most < 1) most = 1;
  const int64_t waves = (n + sms * most - 1) / (sms * most);
  const int wpb = (int)((n + sms * waves - 1) / (sms * waves));
  const size_t smem = chunk_bytes + (size_t)wpb * tb.D * sizeof(float2);
  e = allow_smem(encode_reads_wide_kernel, smem);
  if (e != cudaSuccess) return e;
  int64_t blocks = (n + wpb - 1) / wpb;
  if (blocks > 152 * 16) blocks = 152 * 16;
  encode_reads_wide_kernel<<<(unsigned)blocks, wpb * 32, smem, st>>>(tb, seqs, offsets, n, emb_f32,
                                                                       reinterpret_cast<__nv_bfloat16*>(emb_bf16),
                                                                       norms, status, perm, n_fwd);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- reference pre-pass

// Letters of the packed reference from position p on, one per step: the code of
// the s letters at the current position, the next word loaded a word ahead.
struct LetterCursor {
  const uint32_t* next;
  uint64_t v;
  uint32_t ahead;
  int have;  // letters in v
  __device__ __forceinline__ void start(const uint32_t* __restrict__ packed, int64_t p) {
    next = packed + (p >> 4);
    const int off = (int)(p & 15);
    v = __ldg(next) >> (2 * off);
    have = 16 - off;
    ahead = __ldg(next + 1);
    next += 2;
  }
  __device__ __forceinline__ uint32_t code(int s, uint32_t mask) {
    if (have < s) {
      v |= (uint64_t)ahead << (2 * have);
      have += 16;
      ahead = __ldg(next++);
    }
    const uint32_t c = (uint32_t)v & mask;
    v >>= 2;
    --have;
    return c;
  }
};

// 1/sqrt(x) rounded to FP32, x > 0 in FP32's range: an FP32 estimate and one
// third-order Householder step in FP64 (relative error about e^3 for an
// estimate's e < 2^-21), 5 FP64 operations where a division and a root take tens.
__device__ __forceinline__ float inv_sqrt_f64(double x) {
  const double r = (double)rsqrtf((float)x);
  const double e = fma(-x * r, r, 1.0);
  return (float)fma(r * e, fma(0.375, e, 0.5), r);
}

// Anchors and window norms, in FP64: a lane per (anchor chunk of A windows,
// band). In the frame of the chunk's first window, w0, a location at offset d
// adds w_k^d (w_k = e^{2 pi i f_k / N}) to its bin's sum S_{k,b} whatever window
// it is seen from: window j's entry is S_{k,b} times a unit phase (§3.4's
// rotation), so norms need no rotation, and sliding by a letter changes
// C_k = sum_b |S_{k,b}|^2 only through the leaving and the entering bin:
// |S -+ w|^2 = |S|^2 -+ 2 S.w + 1. A lane keeps its band's sums in shared memory,
// column = lane (no bank conflicts whatever the bins), sums the first window
// directly (§2.1-§2.3; stored in FP32, the anchor that seeds the on-chip FP32
// recurrence) and walks the chunk. The stored 1/sqrt(C_j) thus carries neither
// the FP32 recurrence's drift nor any rotation's rounding. A difference carries
// the rounding of the largest C it came through, though: four a slide, 256 S a
// chunk (S letters a window). So a chunk in which C falls by 2^18 / S or more (sums
// that nearly cancel) is walked a second time, with C formed from the sums wherever
// it has fallen so far: its relative error stays below 2^-27, an eighth of FP32's.
// Looking at that in every step of the one walk costs its latency (437 against 420
// us for 1 Mbp); noting it does not. Where it happens often (one-letter s-mers on a
// reference with tandem repeats, whose windows cancel wholly) the second walks cost
// a third more: 323 -> 419 us for 1 Mbp.
//
// Bound by the FP64 unit (2 results a cycle per SM): 11 operations a window and
// band, 2 a location of the first window. A warp per chunk that rotated all D
// entries and reduced their squares at every window took about 45 FP64
// instructions of a whole warp a window.
// Index of 10 Mbp (s = 4, m = t = 2, N = 150), whole call: 38.3 -> 1.74 ms, and
// 1.50 -> 1.31 ms by forming each root once instead of in every band's lane.
template <bool kUnit>  // stride 1: a window's letters four steps at a time
__global__ void prepass_kernel(DevIndex ix, PrepassTables pt, float2* __restrict__ anchors,
                               float* __restrict__ inv_norm, float* __restrict__ band_norm) {
  extern __shared__ double2 pre_acc[];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const int m = ix.m, nb = ix.nb, S = ix.stride, s = ix.s;
  double2* acc = pre_acc + (size_t)warp * nb * 32 + lane;  // entry b: acc[32 * b]
  const int64_t n_chunks = (ix.W + ix.A - 1) / ix.A;
  const int n_loc = ix.N - s + 1;
  const uint32_t mask = (1u << (2 * s)) - 1u;
  const int cpw = 32 / m;  // chunks per warp
  const int k = lane % m;  // this lane's band
  const int64_t a = ((int64_t)blockIdx.x * wpb + warp) * cpw + lane / m;
  const bool live = lane < cpw * m && a < n_chunks;
  // the other lanes walk the last chunk and store nothing
  const int64_t j0 = (live ? a : n_chunks - 1) * ix.A;
  const double2* ph = pt.phase + (size_t)k * pt.n_phase;
  const int group = lane - k;

  LetterCursor out, in;  // leaving and entering locations
  double C = 0.0;
  // high word (ordered as the value, if positive) of the largest C since C was last formed from the sums
  int peak = 0;
  const int drop = (18 - (S > 1 ? 32 - __clz(S - 1) : 0)) << 20;
  bool fallen = false;  // C fell that far below it
  auto bin = [&](LetterCursor& c) { return (uint32_t)__ldg(ix.map_lsb + c.code(s, mask)); };
  auto add = [&](uint32_t b, double2 w) {
    double2 v = acc[32 * b];
    v.x += w.x;
    v.y += w.y;
    acc[32 * b] = v;
  };
  auto first_window = [&]() {
    for (int b = 0; b < nb; ++b) acc[32 * b] = make_double2(0.0, 0.0);
    out.start(ix.packed, j0 * S);
    in.start(ix.packed, j0 * S);
    int d = 0;
    for (; d + 4 <= n_loc; d += 4) {
      uint32_t b[4];
      double2 w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        b[q] = bin(in);
        w[q] = __ldg(ph + d + q);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) add(b[q], w[q]);
    }
    for (; d < n_loc; ++d) add(bin(in), __ldg(ph + d));
  };
  auto from_sums = [&](bool store) {
    C = 0.0;
    for (int b = 0; b < nb; b += 2) {  // nb = 4^t
      const double2 v = acc[32 * b], u = acc[32 * (b + 1)];
      C = fma(v.x, v.x, fma(v.y, v.y, C));
      C = fma(u.x, u.x, fma(u.y, u.y, C));
      if (store)
        *reinterpret_cast<float4*>(anchors + a * ix.D + k * nb + b) = make_float4((float)v.x, (float)v.y, (float)u.x, (float)u.y);
    }
    peak = __double2hiint(C);
  };
  const int n_win = (int)min((int64_t)ix.A, ix.W - j0);
  // location d leaves for bin bo, location d + n_loc enters bin bi
  auto slide = [&](uint32_t bo, double2 wo, uint32_t bi, double2 wi) {
    double2 v = acc[32 * bo];
    const double p = fma(v.x, wo.x, v.y * wo.y);
    acc[32 * bo] = make_double2(v.x - wo.x, v.y - wo.y);
    v = acc[32 * bi];
    const double q = fma(v.x, wi.x, v.y * wi.y);
    acc[32 * bi] = make_double2(v.x + wi.x, v.y + wi.y);
    C = fma(2.0, q - p, C + 2.0);
    peak = max(peak, __double2hiint(C));
  };
  // C of window j over all bands; exact: formed from the sums where it has fallen
  auto total_of = [&](int j, bool exact) -> double {
    const bool low = __double2hiint(C) < peak - drop;
    if (exact) {
      if (low) from_sums(false);
    } else {
      fallen |= low && j < n_win;
    }
    double tot = C;
    if (m > 1) {
      tot = 0.0;
      for (int q = 0; q < m; ++q) tot += __shfl_sync(0xffffffffu, C, (group + q) & 31);
    }
    if (band_norm && live && j < n_win) band_norm[(j0 + j) * m + k] = (float)C;
    return tot;
  };
  auto walk = [&](auto exact_c) {
    constexpr bool exact = decltype(exact_c)::value;
    for (int jq = 0; jq < kAnchorPeriod; jq += 4) {
      double tot[4];
      if (kUnit && !exact) {
        uint32_t bo[4], bi[4];
        double2 wo[4], wi[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          bo[q] = bin(out);
          bi[q] = bin(in);
          // (the slide after the chunk's last window is not needed)
          const int d = min(jq + q, kAnchorPeriod - 2);
          wo[q] = __ldg(ph + d);
          wi[q] = __ldg(ph + d + n_loc);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          tot[q] = total_of(jq + q, exact);
          slide(bo[q], wo[q], bi[q], wi[q]);
        }
      } else {
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          const double v = total_of(jq + q, exact);
          tot[0] = q == 0 ? v : tot[0];
          tot[1] = q == 1 ? v : tot[1];
          tot[2] = q == 2 ? v : tot[2];
          tot[3] = q == 3 ? v : tot[3];
          if (jq + q == kAnchorPeriod - 1) break;
          const int d0 = (jq + q) * S;
          for (int u = 0; u < S; ++u) slide(bin(out), __ldg(ph + d0 + u), bin(in), __ldg(ph + d0 + u + n_loc));
        }
      }
      // the four roots are shared among the chunk's lanes (each knows all totals)
      for (int q = k; q < 4; q += m) {
        const double v = q < 2 ? (q == 0 ? tot[0] : tot[1]) : (q == 2 ? tot[2] : tot[3]);
        if (live && jq + q < n_win) inv_norm[j0 + jq + q] = v > (double)kZeroNorm2 ? inv_sqrt_f64(v) : 0.f;
      }
    }
  };
  first_window();
  from_sums(live);
  walk(std::false_type());
  if (__any_sync(0xffffffffu, fallen)) {
    first_window();
    from_sums(false);
    walk(std::true_type());
  }
}

cudaError_t launch_prepass(const DevIndex& ix, const PrepassTables& pt, float2* anchors, float* inv_norm,
                           float* band_norm, cudaStream_t st) {
  static_assert(kAnchorPeriod % 16 == 0, "chunks start at whole packed words; windows go four at a time");
  const int64_t n_chunks = (ix.W + ix.A - 1) / ix.A;
  const int cpw = 32 / ix.m;
  const int64_t warps = (n_chunks + cpw - 1) / cpw;
  // 512 nb bytes a warp: 4 warps a block (32 KB at nb = 16), one where the sums
  // are wide or the reference too short to give every SM a block of 4
  const int wpb = ix.nb > 16 || warps < 4 * 152 ? 1 : 4;
  const int64_t blocks = (warps + wpb - 1) / wpb;
  const size_t smem = (size_t)wpb * ix.nb * 32 * sizeof(double2);
  if (ix.stride == 1) {
    prepass_kernel<true><<<(unsigned)blocks, wpb * 32, smem, st>>>(ix, pt, anchors, inv_norm, band_norm);
  } else {
    prepass_kernel<false><<<(unsigned)blocks, wpb * 32, smem, st>>>(ix, pt, anchors, inv_norm, band_norm);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- a4: windows

// Each chain of D/4 lanes starts at one anchor and runs the FP32 recurrence
// through its chunk of A windows, storing the unnormalised c(j) of the
// requested windows. This is the generator the scans run, exposed for checks.
template <int D>
__global__ void window_embeddings_kernel(DevIndex ix, int64_t j_begin, int64_t count, float* __restrict__ out) {
  constexpr int LPC = Chain<D>::LPC;
  constexpr int CPW = 32 / LPC;
  const int lane = threadIdx.x & 31;
  const int lic = lane % LPC;
  const int64_t chain = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * CPW + lane / LPC;
  const int64_t a0 = j_begin / ix.A;
  const int64_t a = a0 + chain;
  const int64_t j_end = min(ix.W, j_begin + count);
  if (a * ix.A >= j_end) return;
  Chain<D> ch;
  ch.setup(ix, lic);
  ch.load(ix.anchors + a * ix.D, lic);
  const int S = ix.stride;
  const int64_t jlast = min(j_end, (a + 1) * ix.A);
  for (int64_t j = a * ix.A; j < jlast; ++j) {
    if (j >= j_begin) {
      float* o = out + (j - j_begin) * 2 * D;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        o[4 * lic + i] = ch.cr[i];
        o[D + 4 * lic + i] = ch.ci[i];
      }
    }
    const int64_t w = j * S;
    if (S == 1) {
      ch.step1(bin_at(ix.packed, w, ix.s, ix.map_lsb), bin_at(ix.packed, w + ix.N - ix.s + 1, ix.s, ix.map_lsb));
    } else {
      for (int u = 0; u < S; ++u) {
        ch.sub_at(bin_at(ix.packed, w + u, ix.s, ix.map_lsb), ix.eout[ch.band * S + u]);
        ch.add_at(bin_at(ix.packed, w + ix.N - ix.s + 1 + u, ix.s, ix.map_lsb), ix.ein[ch.band * S + u]);
      }
      ch.rotate();
    }
  }
}

cudaError_t launch_window_embeddings(const DevIndex& ix, int64_t j_begin, int64_t count, float* out,
                                     cudaStream_t st) {
  const int64_t j_end = min(ix.W, j_begin + count);
  if (j_end <= j_begin) return cudaSuccess;
  const int64_t n_chains = (j_end - 1) / ix.A - j_begin / ix.A + 1;
  const int LPC = ix.D / 4;
  const int cpb = 4 * (32 / LPC);  // 4 warps per block
  const unsigned blocks = (unsigned)((n_chains + cpb - 1) / cpb);
  switch (ix.D) {
    case 4: window_embeddings_kernel<4><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    case 8: window_embeddings_kernel<8><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    case 16: window_embeddings_kernel<16><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    case 32: window_embeddings_kernel<32><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    case 64: window_embeddings_kernel<64><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    case 128: window_embeddings_kernel<128><<<blocks, 128, 0, st>>>(ix, j_begin, count, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace rope
