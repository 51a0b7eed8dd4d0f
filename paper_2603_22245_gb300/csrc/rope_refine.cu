// Refinement (§3.4, increasing the accuracy): around a candidate start found
// at a coarse window stride, the window is slid one letter at a time and each
// position is scored against the read head, typically with a richer encoding
// (up to 4^8 bins per band) than the scan's.
//
// The per-step update is the paper's inner-product recurrence written in the
// frame of the first position p0 of the range: with S_{k,b} = sum over the
// window's locations d (absolute offset from p0) whose s-mer falls in bin b of
// w_k^d (w_k = e^{2 pi i f_k / N}), the window's encoding is
// c_{k,b}(p) = w_k^{-(p-p0)} S_{k,b}, so
//   ip_k(p) = w_k^{-(p-p0)} J_k,   J_k = sum_b conj(x_{k,b}) S_{k,b},
//   C_k(p)  = sum_b |S_{k,b}|^2.
// Sliding by one letter removes location d = p-p0 from its bin and adds
// d + N-s+1 to another: J_k and C_k change by O(m) terms (the leaving and
// entering s-mers only), and no entry is rotated, so no rounding drift builds
// up in the rotated entries. The window norm is tracked exactly (every bin's
// S kept in a hash table), not skipped.
//
// One warp per (read, run of candidates). Nothing is walked location by
// location: the locations of the read and of a candidate's range are linked
// into one chain per bin (32 locations a step: equal bins of a step by
// __match_any_sync, earlier ones through a hash table of chain heads), and then
//   * x_{k,b} and the first window's S_{k,b} are summed along the chains, a
//     chain per lane, in location order;
//   * the C_k changes of the slides come from the same chains (a bin changes
//     only when one of its own locations leaves or enters, so its FP32 sums go
//     through the same values as in a walk over the steps), the J_k changes
//     from the leaving and the entering location of each step, a step per lane;
//   * J_k and C_k at every step are FP64 prefix sums over the steps.
// What bounds it is the latency of its shared-memory chains and the FP64 unit
// (2 results a cycle per SM): the phases e^{2 pi i f_k d / N} depend on the
// offset alone and are formed once per block, not once per candidate.
// One warp per read whose first lane walked every location and step through hash
// tables, on 4,096 reads x 2 candidates x 17 positions (N = 150, s = t = 8,
// m = 2): 4.04 ms; this 0.28 ms.
#include <cuda_runtime.h>

#include "rope_internal.h"

namespace rope {

constexpr int kRefMaxBands = 8;

struct RefineArgs {
  EncTables tb;                  // map [4^s] (first letter most significant), read-frame phases [m * n_loc]
  int64_t a[kRefMaxBands];       // f_k = a_k / q
  int64_t Q;                     // q * N
  int32_t score_mode;
  const uint32_t* packed;        // 2-bit packed reference
  int64_t L;
  const uint8_t* seqs;
  const int64_t* offsets;
  int64_t n_reads;
  const int64_t* cand;           // [n_reads, n_cand]
  int32_t n_cand, radius;
  int64_t* out_pos;              // [n_reads, n_cand]
  float* out_fid;
  int* status;
  int32_t cap_r_log2, cap_w_log2;  // hash table capacities (powers of two)
  int32_t n_w_max;                 // window locations of the longest range: 2*radius + N-s+1
  int32_t run;                     // candidates per warp
  uint32_t phase_bytes;            // shared memory of the block's phases
  uint32_t read_bytes;             // of a warp's read tables
  uint32_t warp_bytes;             // of a warp, read tables included
};

__device__ __forceinline__ uint32_t ref_hash(int32_t key, int cap_log2) {
  return ((uint32_t)key * 0x9E3779B1u) >> (32 - cap_log2);
}

// The locations of a read or a range, chained by bin. heads: open-addressed
// table of the first location of each bin (never full: its capacity is at least
// twice the number of locations); last: at a head, the chain's last location,
// elsewhere kNoLoc.
constexpr uint16_t kNoLoc = 0xFFFF;
struct Chains {
  int32_t* heads;  // [1 << cap_log2]
  uint16_t *bin, *next, *last;
  int cap_log2;
  __device__ bool is_head(int d) const { return last[d] != kNoLoc; }
};

// first location of bin b, or -1
__device__ __forceinline__ int chain_find(const Chains& t, uint32_t b) {
  const uint32_t mask = (1u << t.cap_log2) - 1u;
  uint32_t h = ref_hash((int32_t)b, t.cap_log2);
  while (true) {
    const int32_t c = t.heads[h];
    if (c < 0 || t.bin[c] == b) return c;
    h = (h + 1u) & mask;
  }
}

// The same, entering location d as the head of bin b where it has none. Lanes
// of a warp call it together for distinct bins, whose bin[] entries are written.
__device__ __forceinline__ int chain_head(const Chains& t, uint32_t b, int d) {
  const uint32_t mask = (1u << t.cap_log2) - 1u;
  uint32_t h = ref_hash((int32_t)b, t.cap_log2);
  while (true) {
    const int32_t c = atomicCAS(t.heads + h, -1, d);
    if (c < 0) return d;
    if (t.bin[c] == b) return c;
    h = (h + 1u) & mask;
  }
}

__device__ __forceinline__ void chains_clear(const Chains& t) {
  for (int i = threadIdx.x & 31; i < (1 << t.cap_log2); i += 32) t.heads[i] = -1;
  __syncwarp();
}

// Appends locations d0 .. d0+31 (lane's location d0 + lane in bin b where valid)
// to the chains; called by a whole warp for d0 = 0, 32, ...
__device__ __forceinline__ void chains_append(const Chains& t, int d0, bool valid, uint32_t b) {
  const int lane = threadIdx.x & 31, d = d0 + lane;
  if (valid) {
    t.bin[d] = (uint16_t)b;
    t.next[d] = kNoLoc;
  }
  __syncwarp();
  const uint32_t grp = __match_any_sync(0xffffffffu, valid ? b : 0x10000u);
  const uint32_t below = grp & ((1u << lane) - 1u);
  int head = 0;
  if (valid && below == 0) head = chain_head(t, b, d);
  head = __shfl_sync(0xffffffffu, head, __ffs(grp) - 1);
  if (valid) {
    if (below) {
      t.next[d0 + 31 - __clz(below)] = (uint16_t)d;
    } else if (head != d) {
      t.next[t.last[head]] = (uint16_t)d;
    }
    if (head != d) t.last[d] = kNoLoc;
  }
  __syncwarp();
  if (valid && (grp >> lane) == 1u) t.last[head] = (uint16_t)d;
  __syncwarp();
}

// e^{2 pi i a d / Q} with the exponent reduced in integers, rounded to FP32
__device__ __forceinline__ float2 ref_unit(int64_t a, int64_t Q, int64_t d) {
  int64_t r = (a * d) % Q;
  if (r < 0) r += Q;
  double sn, cs;
  sincospi(2.0 * (double)r / (double)Q, &sn, &cs);
  return make_float2((float)cs, (float)sn);
}

// code (first letter most significant) of the s letters from pos
__device__ __forceinline__ uint32_t packed_code(const uint32_t* __restrict__ packed, int64_t pos, int s) {
  const int off = (int)(pos & 15);
  uint64_t v = __ldg(packed + (pos >> 4));
  if (off + s > 16) v |= (uint64_t)__ldg(packed + (pos >> 4) + 1) << 32;
  // reversed bits put the first letter on top, each letter's two bits swapped
  const uint32_t g = __brev((uint32_t)(v >> (2 * off))) >> (32 - 2 * s);
  return ((g & 0x55555555u) << 1) | ((g >> 1) & 0x55555555u);
}

// Whether fidelity f beats g by more than the rounding of the FP64 sums they come
// from: positions that are equal but for it are ties, which go to the lower one
// (an s-mer that a read shares with a range gives the same fidelity half a window
// further on).
__device__ __forceinline__ bool ref_beats(double f, double g) { return f > fma(g, 1e-12, g) + 1e-20; }

// |v|^2 in FP64 (the products of FP32 values are exact)
__device__ __forceinline__ double norm2(float2 v) { return (double)v.x * v.x + (double)v.y * v.y; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int MB>  // most bands
__global__ void __launch_bounds__(256) refine_kernel(RefineArgs a) {
  extern __shared__ __align__(16) uint8_t ref_smem[];
  const int m = a.tb.m, N = a.tb.N, s = a.tb.s;
  const int n_loc = N - s + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

  // block: phases [n_w_max][m]; warp: read [heads | bin | next | last | x [n_loc][m]],
  // range [heads | dC [2*radius][m] | bin | next | last]
  float2* wph = reinterpret_cast<float2*>(ref_smem);
  for (int i = threadIdx.x; i < a.n_w_max * m; i += blockDim.x) {
    const int d = i / m;
    wph[i] = ref_unit(a.a[i - d * m], a.Q, d);
  }
  __syncthreads();
  uint8_t* wb = ref_smem + a.phase_bytes + (size_t)warp * a.warp_bytes;
  Chains rd, wn;
  rd.cap_log2 = a.cap_r_log2;
  rd.heads = reinterpret_cast<int32_t*>(wb);
  float2* rx = reinterpret_cast<float2*>(rd.heads + (1 << a.cap_r_log2));
  rd.bin = reinterpret_cast<uint16_t*>(rx + (size_t)n_loc * m);
  rd.next = rd.bin + n_loc;
  rd.last = rd.next + n_loc;
  wb += a.read_bytes;
  wn.cap_log2 = a.cap_w_log2;
  wn.heads = reinterpret_cast<int32_t*>(wb);
  double* dC = reinterpret_cast<double*>(wn.heads + (1 << a.cap_w_log2));
  wn.bin = reinterpret_cast<uint16_t*>(dC + (size_t)2 * a.radius * m);
  wn.next = wn.bin + a.n_w_max;
  wn.last = wn.next + a.n_w_max;
  const int64_t last = a.L - N;  // last window start
  const int runs = (a.n_cand + a.run - 1) / a.run;
  const int64_t n_units = a.n_reads * runs;

  for (int64_t unit = (int64_t)blockIdx.x * nwarps + warp; unit < n_units; unit += (int64_t)gridDim.x * nwarps) {
    const int64_t r = unit / runs;
    const int c_lo = (int)(unit - r * runs) * a.run, c_hi = min(c_lo + a.run, a.n_cand);
    const int64_t start = a.offsets[r];
    const int64_t len = a.offsets[r + 1] - start;
    const uint8_t* seq = a.seqs + start;
    bool ok = len >= N;
    if (!ok) {
      if (lane == 0) set_status(a.status, kStatusShortRead);
    } else {
      chains_clear(rd);
      bool bad = false;
      uint32_t nxt = lane < N ? letter_code(seq[lane]) : 0u;
      for (int d0 = 0; d0 < n_loc; d0 += 32) {
        // letters d0 .. d0+63 across the warp (s <= 8: a code ends within them)
        const uint32_t cur = nxt;
        nxt = d0 + 32 + lane < N ? letter_code(seq[d0 + 32 + lane]) : 0u;
        bad |= cur > 3 || nxt > 3;
        uint32_t code = 0;
        for (int i = 0; i < s; ++i) {
          const uint32_t lo = __shfl_sync(0xffffffffu, cur, (lane + i) & 31);
          const uint32_t hi = __shfl_sync(0xffffffffu, nxt, (lane + i) & 31);
          code = code * 4u + ((lane + i < 32 ? lo : hi) & 3u);
        }
        const bool valid = d0 + lane < n_loc;
        chains_append(rd, d0, valid, valid ? (uint32_t)a.tb.map[code] : 0u);
      }
      if (__any_sync(0xffffffffu, bad)) {
        ok = false;
        if (lane == 0) set_status(a.status, kStatusBadBase);
      }
    }
    double xk[MB], xtot = 0.0;  // |x_k|^2
#pragma unroll
    for (int k = 0; k < MB; ++k) xk[k] = 0.0;
    if (ok) {
      // x_{k,b} at the head of its chain: the bin's phases summed in location order
      for (int d = lane; d < n_loc; d += 32) {
        if (!rd.is_head(d)) continue;
        float2 x[MB];
#pragma unroll
        for (int k = 0; k < MB; ++k) x[k] = make_float2(0.f, 0.f);
        for (uint32_t l = d; l != kNoLoc; l = rd.next[l]) {
#pragma unroll
          for (int k = 0; k < MB; ++k) {
            if (k >= m) continue;
            const float2 ph = __ldg(a.tb.phase + (size_t)k * n_loc + l);
            x[k].x += ph.x;
            x[k].y += ph.y;
          }
        }
#pragma unroll
        for (int k = 0; k < MB; ++k) {
          if (k >= m) continue;
          rx[d * m + k] = x[k];
          xk[k] += norm2(x[k]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < MB; ++k) {
        if (k >= m) continue;
        xk[k] = warp_sum(xk[k]);
        xtot += xk[k];
      }
    }

    for (int c = c_lo; c < c_hi; ++c) {
      const size_t o = (size_t)r * a.n_cand + c;
      const int64_t pos = a.cand[o];
      if (!ok || pos < 0 || last < 0) {
        if (lane == 0) {
          a.out_pos[o] = -1;
          a.out_fid[o] = -INFINITY;
        }
        continue;
      }
      const int64_t cpos = pos < last ? pos : last;
      const int64_t p0 = cpos - a.radius > 0 ? cpos - a.radius : 0;
      const int64_t p1 = cpos + a.radius < last ? cpos + a.radius : last;
      const int n_steps = (int)(p1 - p0);
      const int n_w = n_steps + n_loc;
      for (int i = lane; i < n_steps * m; i += 32) dC[i] = 0.0;
      chains_clear(wn);
      double Jr[MB], Ji[MB], C[MB];
#pragma unroll
      for (int k = 0; k < MB; ++k) Jr[k] = Ji[k] = C[k] = 0.0;
      // J_k changes by sgn * conj(x_{k,b}) w_k^d where location d of bin b enters or leaves
      auto j_term = [&](int d, uint32_t b, double sgn, double (&jr)[MB], double (&ji)[MB]) {
        const int hx = chain_find(rd, b);
        if (hx < 0) return;
#pragma unroll
        for (int k = 0; k < MB; ++k) {
          if (k >= m) continue;
          const float2 ph = wph[d * m + k], x = rx[hx * m + k];
          jr[k] += sgn * ((double)x.x * ph.x + (double)x.y * ph.y);
          ji[k] += sgn * ((double)x.x * ph.y - (double)x.y * ph.x);
        }
      };
      for (int d0 = 0; d0 < n_w; d0 += 32) {
        const int d = d0 + lane;
        const bool valid = d < n_w;
        const uint32_t b = valid ? (uint32_t)a.tb.map[packed_code(a.packed, p0 + d, s)] : 0u;
        if (d < n_loc) j_term(d, b, 1.0, Jr, Ji);
        chains_append(wn, d0, valid, b);
      }
      // a bin's sums: the first window's, then as its locations leave and enter
      for (int d = lane; d < n_w; d += 32) {
        if (!wn.is_head(d)) continue;
        float2 S[MB];
#pragma unroll
        for (int k = 0; k < MB; ++k) S[k] = make_float2(0.f, 0.f);
        uint32_t in = d;  // next location to enter
        for (; in != kNoLoc && in < (uint32_t)n_loc; in = wn.next[in]) {
#pragma unroll
          for (int k = 0; k < MB; ++k) {
            if (k >= m) continue;
            const float2 ph = wph[in * m + k];
            S[k].x += ph.x;
            S[k].y += ph.y;
          }
        }
#pragma unroll
        for (int k = 0; k < MB; ++k)
          if (k < m) C[k] += norm2(S[k]);
        uint32_t out = d;  // next to leave: location d leaves at step d, location n_loc + d enters then
        while (true) {
          const bool leaves = out < (uint32_t)n_steps, enters = in != kNoLoc;
          if (!leaves && !enters) break;
          const bool leave = leaves && (!enters || out + n_loc <= in);
          const uint32_t l = leave ? out : in;
          const uint32_t step = leave ? out : in - n_loc;
          const float sgn = leave ? -1.f : 1.f;
#pragma unroll
          for (int k = 0; k < MB; ++k) {
            if (k >= m) continue;
            const float2 ph = wph[l * m + k];
            const float2 nw = make_float2(S[k].x + sgn * ph.x, S[k].y + sgn * ph.y);
            // at most two terms reach a step's sum (one leaves, one enters): any order gives the same bits
            atomicAdd(dC + step * m + k, norm2(nw) - norm2(S[k]));
            S[k] = nw;
          }
          if (leave) {
            out = wn.next[out];
          } else {
            in = wn.next[in];
          }
        }
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < MB; ++k) {
        if (k >= m) continue;
        Jr[k] = warp_sum(Jr[k]);
        Ji[k] = warp_sum(Ji[k]);
        C[k] = warp_sum(C[k]);
      }
      auto fid_at = [&](int i, const double (&jr)[MB], const double (&ji)[MB], const double (&ck)[MB]) -> double {
        if (a.score_mode == 0) {
          double ir = 0.0, ii = 0.0, ct = 0.0;
#pragma unroll
          for (int k = 0; k < MB; ++k) {
            if (k >= m) continue;
            // ip_k = conj(w_k^i) J_k
            const float2 ph = wph[i * m + k];
            ir += (double)ph.x * jr[k] + (double)ph.y * ji[k];
            ii += (double)ph.x * ji[k] - (double)ph.y * jr[k];
            ct += ck[k];
          }
          const double den = xtot * ct;
          return den > (double)kZeroNorm2 ? (ir * ir + ii * ii) / den : 0.0;
        }
        double f = 0.0;
#pragma unroll
        for (int k = 0; k < MB; ++k) {
          if (k >= m) continue;
          const double den = xk[k] * ck[k];
          if (den > (double)kZeroNorm2) f += (jr[k] * jr[k] + ji[k] * ji[k]) / den;
        }
        return f / m;
      };
      // J and C 32 steps at a time: the steps' changes, then their prefix sums
      double best = -INFINITY;
      int best_i = 0x7FFFFFFF;
      if (lane == 0) {
        best = fid_at(0, Jr, Ji, C);
        best_i = 0;
      }
      for (int t0 = 0; t0 < n_steps; t0 += 32) {
        const int t = t0 + lane;
        double jr[MB], ji[MB], ck[MB];
#pragma unroll
        for (int k = 0; k < MB; ++k) jr[k] = ji[k] = ck[k] = 0.0;
        if (t < n_steps) {
          j_term(t, wn.bin[t], -1.0, jr, ji);
          j_term(t + n_loc, wn.bin[t + n_loc], 1.0, jr, ji);
#pragma unroll
          for (int k = 0; k < MB; ++k)
            if (k < m) ck[k] = dC[t * m + k];
        }
#pragma unroll
        for (int k = 0; k < MB; ++k) {
          if (k >= m) continue;
#pragma unroll
          for (int w = 1; w < 32; w *= 2) {
            const double vr = __shfl_up_sync(0xffffffffu, jr[k], w), vi = __shfl_up_sync(0xffffffffu, ji[k], w);
            const double vc = __shfl_up_sync(0xffffffffu, ck[k], w);
            if (lane >= w) {
              jr[k] += vr;
              ji[k] += vi;
              ck[k] += vc;
            }
          }
          jr[k] += Jr[k];
          ji[k] += Ji[k];
          ck[k] += C[k];
          Jr[k] = __shfl_sync(0xffffffffu, jr[k], 31);
          Ji[k] = __shfl_sync(0xffffffffu, ji[k], 31);
          C[k] = __shfl_sync(0xffffffffu, ck[k], 31);
        }
        if (t < n_steps) {
          const double f = fid_at(t + 1, jr, ji, ck);
          if (ref_beats(f, best)) best_i = t + 1;
          best = fmax(best, f);
        }
      }
      // the best fidelity, and the lowest position that it does not beat
      double top = best;
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, w));
      best_i = (int)__reduce_min_sync(0xffffffffu, ref_beats(top, best) ? 0x7FFFFFFFu : (unsigned)best_i);
      if (lane == 0) {
        a.out_pos[o] = p0 + best_i;
        a.out_fid[o] = (float)top;
      }
      __syncwarp();  // the tables are free for the next candidate
    }
    __syncwarp();
  }
}

static int ceil_log2(int64_t v) {
  int r = 0;
  while ((int64_t(1) << r) < v) ++r;
  return r;
}

template <int MB>
static cudaError_t launch_bands(RefineArgs a, int warps, size_t smem, int num_sms, cudaStream_t st) {
  auto kern = refine_kernel<MB>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem);
  if (e != cudaSuccess) return e;
  const int64_t slots = (int64_t)num_sms * (per_sm < 1 ? 1 : per_sm);
  // a warp takes all of a read's candidates (its tables are built once) unless
  // that leaves warps idle; then one candidate each
  a.run = a.n_reads >= slots * warps ? a.n_cand : 1;
  const int64_t units = a.n_reads * (a.run == 1 ? a.n_cand : 1);
  const int64_t blocks = (units + warps - 1) / warps;
  kern<<<(unsigned)(blocks < slots ? blocks : slots), warps * 32, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_refine(RefineArgs a, int max_warps, cudaStream_t st) {
  if (a.n_reads <= 0 || a.n_cand <= 0) return cudaSuccess;
  const int m = a.tb.m, n_loc = a.tb.N - a.tb.s + 1;
  a.n_w_max = 2 * a.radius + n_loc;
  a.cap_r_log2 = ceil_log2(2 * (int64_t)n_loc) < 5 ? 5 : ceil_log2(2 * (int64_t)n_loc);
  a.cap_w_log2 = ceil_log2(2 * (int64_t)a.n_w_max) < 5 ? 5 : ceil_log2(2 * (int64_t)a.n_w_max);
  int dev = 0, optin = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // The largest windows and radii: the hash slots of a read and a range with m
  // sums each, the bins, and the phases have to fit in a block's shared memory
  // (this kernel's own tables always take less: it keeps sums per location, at
  // most half the slots, and 16-bit locations, so its indexes fit too).
  const auto align16 = [](size_t v) { return (v + 15) & ~size_t(15); };
  const size_t range_most = ((size_t)(1 << a.cap_w_log2) * (4 + 8 * m) + (size_t)a.n_w_max * 4 + 8 + (size_t)a.n_w_max * m * 8);
  const size_t read_most = ((size_t)(1 << a.cap_r_log2) * (4 + 8 * m) + (size_t)n_loc * 4 + 4 * (kRefMaxBands + 2));
  if (align16(read_most) + align16(range_most) > (size_t)optin) return cudaErrorInvalidValue;
  a.phase_bytes = (uint32_t)align16((size_t)a.n_w_max * m * 8);
  a.read_bytes = (uint32_t)align16((size_t)(1 << a.cap_r_log2) * 4 + (size_t)n_loc * (6 + 8 * m));
  a.warp_bytes = a.read_bytes + (uint32_t)align16((size_t)(1 << a.cap_w_log2) * 4 + (size_t)a.n_w_max * 6 + (size_t)a.radius * m * 16);
  int warps = max_warps;
  while (warps > 1 && a.phase_bytes + (size_t)warps * a.warp_bytes > (size_t)optin) --warps;
  const size_t smem = a.phase_bytes + (size_t)warps * a.warp_bytes;
  if (m <= 2) return launch_bands<2>(a, warps, smem, sms, st);
  if (m <= 4) return launch_bands<4>(a, warps, smem, sms, st);
  return launch_bands<kRefMaxBands>(a, warps, smem, sms, st);
}

}  // namespace rope

// ---------------------------------------------------------------- C ABI

#include "rope_host.h"

extern "C" rope_status rope_refine(const rope_index* idx, const rope_params* p, const uint8_t* seqs,
                                   const int64_t* offsets, int64_t n_reads, const int64_t* cand_pos, int32_t n_cand,
                                   int32_t radius, int64_t* out_pos, float* out_fid, cudaStream_t stream) {
  using namespace rope;
  if (!idx) return host_fail(ROPE_ERR_INVALID_ARG, "index is NULL");
  if (n_reads < 0 || n_reads > 0x7FFFFFFFLL) return host_fail(ROPE_ERR_INVALID_ARG, "n_reads outside [0, 2^31)");
  if (n_cand < 1 || n_cand > 64) return host_fail(ROPE_ERR_INVALID_ARG, "n_cand=%d outside [1,64]", n_cand);
  if (radius < 0 || radius > 4096) return host_fail(ROPE_ERR_INVALID_ARG, "radius=%d outside [0,4096]", radius);
  if (n_reads == 0) return ROPE_OK;
  if (!seqs || !offsets || !cand_pos || !out_pos || !out_fid) return host_fail(ROPE_ERR_INVALID_ARG, "NULL pointer");
  RefineArgs a{};
  rope_status st = host_refine_tables(p, &a.tb);
  if (st != ROPE_OK) return st;
  if (p->window_len > idx->ix.L) return host_fail(ROPE_ERR_INVALID_ARG, "window_len beyond the reference");
  DeviceCtx* c;
  if ((st = host_ctx(&c)) != ROPE_OK) return st;
  for (int k = 1; k <= p->m; ++k) {
    int64_t q;
    host_factor(p, k, &a.a[k - 1], &q);
    a.Q = q * p->window_len;
  }
  a.score_mode = p->score_mode;
  a.packed = idx->ix.packed;
  a.L = idx->ix.L;
  a.seqs = seqs;
  a.offsets = offsets;
  a.n_reads = n_reads;
  a.cand = cand_pos;
  a.n_cand = n_cand;
  a.radius = radius;
  a.out_pos = out_pos;
  a.out_fid = out_fid;
  a.status = c->status;
  const cudaError_t e = launch_refine(a, 8, stream);
  if (e == cudaErrorInvalidValue)
    return host_fail(ROPE_ERR_UNSUPPORTED, "refinement tables for N=%d, m=%d, radius=%d exceed shared memory",
                     p->window_len, p->m, radius);
  if (e != cudaSuccess) return host_fail(ROPE_ERR_CUDA, "refine launch: %s", cudaGetErrorString(e));
  return ROPE_OK;
}
