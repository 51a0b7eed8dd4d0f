// Tensor-core scan (BF16 in, FP32 accumulate) on sm_103a with tcgen05.
//
// The fidelity of a read x against a window c is |<x|c>|^2 for normalised
// vectors (§2.4); with x = xr + i xi and c = cr + i ci, Re<x|c> = xr.cr + xi.ci
// and Im<x|c> = xr.ci - xi.cr (the real identity of §4). Per block (one per SM):
//   * A operand (shared memory, 128-byte swizzled K-major): NT tiles of 128
//     reads, row = the read's normalised [xr | xi] in BF16 (K = 2D), written
//     once per work item by the epilogue warps.
//   * B operand (shared memory, same layout): per stage T windows as 2T rows,
//     row n = [cr | ci] and row T+n = [ci | -cr] of window n. The generator
//     warps produce them: each chain of LPC lanes runs the §3.4 recurrence from
//     an exact anchor through 64 consecutive windows and emits one window per
//     stage, scaled by the stored 1/sqrt(C_j) and rounded to BF16.
//   * D (tensor memory): per stage and tile a 128 x 2T FP32 accumulator whose
//     columns are Re (0..T-1) and Im (T..2T-1).
//   * NM threads issue tcgen05.mma (M = 128, N = 2T = 128, K = 16 per
//     instruction; an MMA costs at least ~45 cycles whatever N is, so N = 128
//     keeps the tensor pipe saturated) and commit to mbarriers; a bin warp
//     streams the 2-bit packed reference of each super-tile into shared memory
//     with bulk copies (TMA) and turns its letters into bins a super-tile ahead
//     of the generators; epilogue warps (thread = read; EW warps split an
//     accumulator's windows) load the accumulators with tcgen05.ld in 16-column
//     chunks and keep the read's best windows in LH lists per read.
//
// What bounds it at d = 64 (256 reads x 64 windows a stage): the MMAs alone take
// ~580 cycles a stage (operands at 128 B a cycle, all that shared memory gives),
// the hand-overs with neither generators nor epilogue 77 ms on 32,768 reads x 20 M
// windows, with the generators 96 ms; the epilogue (issue slots and the latency
// of its tensor-memory loads) is what the rest waits for. Measured on that case
// and on 16,384 reads x 100 M windows, against one issuing thread, a bin fill by
// the generators, scores formed for every column and list updates before the
// hand-over (234 ms and 553 ms): 171 ms and 385 ms.
// Every wait is bounded; a wait that runs out sets the timeout status bit and
// the block drains its in-flight copies and MMAs, frees tensor memory and exits.
#include <cuda_bf16.h>

#include "rope_internal.h"
#include "rope_topk.cuh"

namespace rope {

// Scale of both operands in the E4M3 scan (a power of two, so exact): the
// normalised entries (|.| <= 1, typically 1/sqrt(2D)) land in [2^-6, 448],
// the normal range of E4M3, except for entries near 0.
constexpr float kFp8Scale = 32.f;

template <int D_, int NT_, int T_, int NB_, int LPC_, int EW_, int NM_, bool ISOLATE_MMA_, bool FP8_ = false>
struct TcShape {
  static constexpr int D = D_, NT = NT_, T = T_, NB = NB_;  // NB: most B ring slots
  static constexpr int A = kAnchorPeriod;
  static constexpr int LPC = LPC_;               // lanes per chain
  static constexpr int BPL = D / LPC;            // complex entries per generator lane
  static constexpr int CPW = 32 / LPC;           // chains per warp
  static constexpr int GEN_WARPS = T / CPW;
  static constexpr int EW = EW_;                 // epilogue warps sharing one accumulator's columns
  static constexpr int LH = EW;                  // candidate lists per read: one per warp's share of the columns
  static constexpr int WPH = T / EW;             // windows per epilogue warp per stage
  static constexpr int EPI_WARPS = 4 * NT * EW;
  // Roles after the epilogue warps: a bin warp, NM MMA-issuing warps and the
  // generators. With ISOLATE_MMA the issuers take the warp numbers that are
  // multiples of 4, so that these single threads share scheduler 0 with
  // epilogue warps only and get their instructions issued promptly.
  static constexpr int NM = NM_;  // MMA-issuing warps
  static constexpr bool ISOLATE_MMA = ISOLATE_MMA_;
  static constexpr int WARP_MMA = EPI_WARPS;      // the first issuer (EPI_WARPS is a multiple of 4)
  static constexpr int WARP_BIN = EPI_WARPS + 1;
  __host__ __device__ static constexpr int mma_index(int w) {
    const int r = w - EPI_WARPS;
    if (r < 0) return -1;
    if (ISOLATE_MMA) return r % 4 == 0 && r / 4 < NM ? r / 4 : -1;
    return r == 0 ? 0 : r >= 2 && r <= NM ? r - 1 : -1;
  }
  __host__ __device__ static constexpr int gen_index(int w) {
    const int r = w - EPI_WARPS;
    if (r < 2 || mma_index(w) >= 0) return -1;
    int g = r - 2;  // less the issuers between warp EPI_WARPS + 2 and w
    for (int v = EPI_WARPS + 2; v < w; ++v) g -= mma_index(v) >= 0 ? 1 : 0;
    return g < GEN_WARPS ? g : -1;
  }
  __host__ __device__ static constexpr int nwarps() {
    int n = EPI_WARPS + 1 + NM;
    for (int w = EPI_WARPS; w < 64; ++w)
      if ((gen_index(w) >= 0 || mma_index(w) >= 0) && w + 1 > n) n = w + 1;
    return n;
  }
  static constexpr int NWARPS = nwarps();
  static constexpr int NTHREADS = 32 * NWARPS;
  static constexpr int SUP = T * A;                   // windows per super-tile
  static constexpr int GROUP = NT * 128;              // reads per work item
  // operands: BF16, or E4M3 scaled by kFp8Scale (scores then carry kFp8Scale^4)
  static constexpr bool FP8 = FP8_;
  static constexpr int EB = FP8 ? 1 : 2;               // bytes per operand element
  static constexpr int ROW_BYTES = 2 * D * EB;         // one operand row, K = 2D
  static constexpr int KBLK = ROW_BYTES < 128 ? ROW_BYTES : 128;  // swizzle row: 64 or 128 bytes
  static constexpr int KSTEPS = ROW_BYTES / 32;        // 32 bytes of K per MMA (16 BF16 or 32 E4M3)
  static constexpr int STEPS_PER_KBLK = KBLK / 32;
  static constexpr int KBLOCKS = ROW_BYTES / KBLK;     // swizzled K blocks per row
  static constexpr int A_KBLK_BYTES = 128 * KBLK;      // one K block of an A tile
  static constexpr int A_TILE_BYTES = KBLOCKS * A_KBLK_BYTES;
  static constexpr int B_KBLK_BYTES = 2 * T * KBLK;    // one K block of a B tile
  static constexpr int B_SLOT_BYTES = KBLOCKS * B_KBLK_BYTES;
  static constexpr int TMEM_COLS = 512;
  static constexpr int NACC = TMEM_COLS / (2 * T);     // accumulators of one (stage, read tile) each
  static constexpr int STG = NACC / NT;                // accumulators per read tile, used in turn
  static constexpr int STEP = NM / NT;                 // MMA issuers a tile's stages alternate over
  static constexpr int BIN_PITCH = A + 4;              // stride 1: bytes of one chain's row of bins
  static constexpr uint32_t IDESC = FP8 ? idesc_e4m3_f32(128, 2 * T) : idesc_bf16_f32(128, 2 * T);
  static constexpr float SCORE_SCALE = FP8 ? 1.f / (kFp8Scale * kFp8Scale * kFp8Scale * kFp8Scale) : 1.f;
  static constexpr int PIECE = BPL * EB == 8 ? 8 : 16;  // bytes of one generator store
  static constexpr int NPC = BPL * EB / PIECE;           // generator stores per half-row
  static constexpr int WPC = PIECE / 4;                  // 32-bit words per store
  // byte offset of (row r, byte o) of a K block
  __host__ __device__ static uint32_t swz(uint32_t r, uint32_t o) {
    return KBLK == 128 ? sw128_offset(r, o) : sw64_offset(r, o);
  }
  __device__ static uint64_t desc(uint32_t saddr) { return KBLK == 128 ? smem_desc_sw128(saddr) : smem_desc_sw64(saddr); }
  static_assert(D == 32 || D == 64, "complex dimension");
  static_assert(GEN_WARPS * CPW == T, "T must be a multiple of chains per warp");
  static_assert((NM == 2 || NM == 4) && NM % NT == 0 && (NM == NT || NM == NT * STG) && STG >= 1 && STG * NT * 2 * T <= TMEM_COLS, "tensor memory budget");
  static_assert(A % STEP == 0, "every item starts at the first of a tile's issuers");
  static_assert(WPH % 16 == 0, "the epilogue loads 16-column chunks");
  static_assert(BPL * EB == 8 || (BPL * EB) % 16 == 0, "generator lanes write 8-byte or whole 16-byte pieces");
  static_assert(KBLK == 64 || KBLK == 128, "swizzle row");
  static_assert((2 * T) % 16 == 0 && 2 * T <= 256, "MMA N");
  static_assert(NTHREADS <= 1024, "block size");
};

constexpr int kMaxPhaseTab = 16 * 8;  // m * stride <= 16 * 8 (D <= 64 complex, t >= 1)

// two floats rounded to E4M3 (nearest, saturating), lo in the low byte
__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ uint32_t f32x4_to_e4m3(float a, float b, float c, float d) {
  return e4m3x2(a, b) | (e4m3x2(c, d) << 16);
}
// four BF16 (two packed pairs, first entry in the low half) times kFp8Scale, as E4M3
__device__ __forceinline__ uint32_t bf16x4_to_e4m3(uint32_t p, uint32_t q) {
  return f32x4_to_e4m3(__uint_as_float(p << 16) * kFp8Scale, __uint_as_float(p & 0xFFFF0000u) * kFp8Scale,
                       __uint_as_float(q << 16) * kFp8Scale, __uint_as_float(q & 0xFFFF0000u) * kFp8Scale);
}

struct TcLaunch {
  int32_t nb;              // B ring slots in use (1..NB, the most that fit in shared memory)
  int32_t words_per_slot;  // packed words staged per super-tile (multiple of 4)
  int32_t st_slot_bytes;   // bytes of one super-tile data slot
  int32_t bins_bytes;      // bytes of one buffer of bins (per chain at stride 1, per location otherwise)
  int32_t n_bin;           // buffers of bins (2, or 1 where shared memory is short)
  int32_t pend;            // candidates a read's queue holds (1..kPend)
  ThrOut thr;              // threshold mode's output (unused otherwise)
};

// bins of the four positions from p (relative to the first staged letter), one per byte
__device__ __forceinline__ uint32_t bins4_staged(const uint32_t* words, uint32_t rel, int s,
                                                 const uint16_t* __restrict__ map_lsb) {
  const uint32_t wi = rel >> 4;
  const uint64_t v = (((uint64_t)words[wi + 1] << 32) | words[wi]) >> ((rel & 15) * 2);
  const uint32_t mask = (1u << (2 * s)) - 1u;
  uint32_t b = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) b |= (uint32_t)__ldg(map_lsb + ((uint32_t)(v >> (2 * q)) & mask)) << (8 * q);
  return b;
}

// Largest Re^2 + Im^2 of 16 columns: a depth-3 tree of 3-input maxima.
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max_abs2(const uint32_t (&vr)[16], const uint32_t (&vi)[16]) {
  float sc[16];
#pragma unroll
  for (int n = 0; n < 16; n += 2) abs2_pair(vr[n], vr[n + 1], vi[n], vi[n + 1], sc[n], sc[n + 1]);
  const float m0 = fmax3(sc[0], sc[1], sc[2]), m1 = fmax3(sc[3], sc[4], sc[5]), m2 = fmax3(sc[6], sc[7], sc[8]);
  const float m3 = fmax3(sc[9], sc[10], sc[11]), m4 = fmax3(sc[12], sc[13], sc[14]);
  return fmaxf(fmax3(m0, m1, m2), fmax3(m3, m4, sc[15]));
}

// Candidates wait in a short queue per read (up to kPend entries in shared memory)
// and enter the read's lists in batches: a list update costs a warp the same
// for one lane as for all 32, and with a queue it is paid once per several
// arrivals, after the accumulator has been handed back. The queue only defers
// updates: a list's content is the best of all offered, whatever the order.
//
// Per epilogue lane, words at a stride of QS bytes (the block's epilogue lanes):
// a head (count in bits 0-7, the list's worst entry in bits 8-15), then the
// entries' (score, window) pairs.
constexpr int kPend = 4;  // most entries (fewer where shared memory is short)
constexpr int queue_words(int pend) { return 1 + 2 * pend; }

__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// What the out-of-line part of the epilogue needs besides its arguments.
struct ListRef {
  uint32_t queue;    // this lane's queue
  uint32_t list;     // this lane's list (scores)
  uint32_t win_off;  // from its scores to its windows, bytes
  int32_t depth, sep, stride, pend;
};

// The queued candidates into the list; head: the queue's head word, thr: the
// list's worst score. Leaves the queue empty.
template <class Sh>
__device__ __forceinline__ void flush_queue(const ListRef& q, uint32_t& head, float& thr) {
  constexpr uint32_t QS = 4u * Sh::GROUP * Sh::EW;
  const uint32_t cnt = head & 0xFFu;
  const uint32_t n = __reduce_max_sync(0xffffffffu, cnt);
  for (uint32_t e = 0; e < n; ++e) {
    if (e < cnt) {
      const float v = __uint_as_float(lds_u32(q.queue + (1 + 2 * e) * QS));
      const uint32_t j = lds_u32(q.queue + (2 + 2 * e) * QS);
      if (v >= thr) {
        ThreadList tl;
        tl.s = static_cast<float*>(__cvta_shared_to_generic(q.list));
        tl.w = static_cast<uint32_t*>(__cvta_shared_to_generic(q.list + q.win_off));
        tl.stride = Sh::GROUP * Sh::LH;
        tl.depth = q.depth;
        tl.worst = (int)((head >> 8) & 0xFFu);
        tl.thr = thr;
        tl.insert(v, j, q.sep, q.stride);
        head = (head & ~0xFF00u) | ((uint32_t)tl.worst << 8);
        thr = tl.thr;
      }
    }
    __syncwarp();
  }
  head &= ~0xFFu;
}

// Every queued candidate into its list (the end of a read group).
template <class Sh>
__device__ __noinline__ void flush_all(ListRef q, float thr) {
  uint32_t head = lds_u32(q.queue);
  flush_queue<Sh>(q, head, thr);
}

// An accumulator with something to offer (16-column chunks `todo` of this warp's
// share): the chunks are read again, every window at or above its list's
// threshold is queued, the accumulator handed back as soon as the last chunk is
// in registers, and full queues emptied.
// Out of line, and its state in shared memory, so that the hot loop holds few
// registers and spills none: a block's local memory exceeds the L1 that its
// shared memory leaves, so a reload in that loop would cost an L2 round trip.
// jc0: window of the share's first column. Returns the new threshold.
template <class Sh>
__device__ __noinline__ float offer_chunks(ListRef q, uint32_t tcol, uint32_t todo, uint32_t jc0, uint32_t jlo,
                                           uint32_t jhi, float thr, uint64_t* bar_empty) {
  constexpr uint32_t QS = 4u * Sh::GROUP * Sh::EW;
  constexpr int A = Sh::A;
  uint32_t head = lds_u32(q.queue);
  while (todo) {
    const int c0 = 16 * (__ffs(todo) - 1);
    uint32_t vr[16], vi[16];
    tmem_ld16(tcol + c0, vr);
    tmem_ld16(tcol + Sh::T + c0, vi);
    tc_wait_ld();
    reg_fence(vr);
    reg_fence(vi);
    todo &= todo - 1;
    if (!todo) {
      // the last chunk is in registers: hand the accumulator back first
      tc_fence_before();
      __syncwarp();
      if ((threadIdx.x & 31) == 0) mbar_arrive(bar_empty);
    }
    float sc[16];
#pragma unroll
    for (int n = 0; n < 16; n += 2) abs2_pair(vr[n], vr[n + 1], vi[n], vi[n + 1], sc[n], sc[n + 1]);
    uint32_t pass = 0;  // the windows at or above the threshold
#pragma unroll
    for (int n = 0; n < 16; ++n) pass |= sc[n] >= thr ? (1u << n) : 0u;
    while (__any_sync(0xffffffffu, pass != 0)) {
      while (pass != 0 && (head & 0xFFu) < (uint32_t)q.pend) {
        const int n = __ffs(pass) - 1;
        pass &= pass - 1;
        float v = sc[0];
#pragma unroll
        for (int k2 = 1; k2 < 16; ++k2) v = n == k2 ? sc[k2] : v;
        const uint32_t j = jc0 + (uint32_t)((c0 + n) * A);
        if (j >= jlo && j < jhi) {
          sts_u32(q.queue + (1 + 2 * (head & 0xFFu)) * QS, __float_as_uint(v));
          sts_u32(q.queue + (2 + 2 * (head & 0xFFu)) * QS, j);
          ++head;
        }
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, (head & 0xFFu) == (uint32_t)q.pend)) flush_queue<Sh>(q, head, thr);
    }
  }
  sts_u32(q.queue, head);
  return thr;
}

// kDense: every score written to a.dense. kThr: every score at or above its
// window's threshold L.thr.thr[j] appended to the L.thr pair arrays.
// Otherwise: per-read candidate lists (top-k).
template <class Sh, bool kDense, bool kThr = false>
__global__ void __launch_bounds__(Sh::NTHREADS, 1) scan_tc_kernel(DevIndex ix, ScanArgs a, TcLaunch L) {
  constexpr bool kLists = !kDense && !kThr;
  constexpr int D = Sh::D, NT = Sh::NT, T = Sh::T, NB = Sh::NB, A = Sh::A, BPL = Sh::BPL;
  constexpr int NACC = Sh::NACC, STG = Sh::STG;
  extern __shared__ __align__(1024) uint8_t tc_smem_raw[];
  __shared__ __align__(8) uint64_t bar_bfull[NB], bar_bempty[NB];
  __shared__ __align__(8) uint64_t bar_afull[NACC], bar_aempty[NACC];
  __shared__ __align__(8) uint64_t bar_stfull[2], bar_binfull[2], bar_binempty[2];
  __shared__ __align__(8) uint64_t bar_aready, bar_drain[4];
  __shared__ float2 e_tab[2][kMaxPhaseTab];     // leaving / entering phases [band * S + u]
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;

  // dynamic shared memory:
  //   [A tiles | B ring | 2 packed-word slots | n_bin buffers of bins | lists | queues]
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* a_tiles = smem;
  uint8_t* b_ring = a_tiles + NT * Sh::A_TILE_BYTES;
  uint8_t* st_slots = b_ring + L.nb * Sh::B_SLOT_BYTES;
  uint8_t* bins_t = st_slots + 2 * L.st_slot_bytes;
  float* list_s = reinterpret_cast<float*>(bins_t + L.n_bin * L.bins_bytes);
  uint32_t* list_w = reinterpret_cast<uint32_t*>(list_s + (size_t)a.cand_depth * Sh::GROUP * Sh::LH);
  uint32_t* queues = list_w + (size_t)a.cand_depth * Sh::GROUP * Sh::LH;
  const uint64_t wlim = a.wait_limit_ns;

  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be uniform over the warp
  const int lane = tid & 31;
  const int S = ix.stride;
  volatile int* abort_flag = &abort_s;

  if (tid == 0) {
    for (int i = 0; i < L.nb; ++i) {
      mbar_init(&bar_bfull[i], Sh::GEN_WARPS);
      mbar_init(&bar_bempty[i], NT);  // every read tile's MMAs
    }
    for (int i = 0; i < NACC; ++i) {
      mbar_init(&bar_afull[i], 1);
      mbar_init(&bar_aempty[i], 4 * Sh::EW);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar_stfull[i], 1);
      mbar_init(&bar_binfull[i], 1);
      mbar_init(&bar_binempty[i], Sh::GEN_WARPS);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&bar_drain[i], 1);
    mbar_init(&bar_aready, Sh::EPI_WARPS);
    abort_s = 0;
    fence_barrier_init();
  }
  for (int q = tid; q < ix.m * S; q += Sh::NTHREADS) {
    e_tab[0][q] = ix.eout[q];
    e_tab[1][q] = ix.ein[q];
  }
  if (warp == Sh::WARP_MMA) {
    tmem_alloc(&tmem_base_s, Sh::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tmem_base_s;
  // items (read group, window range) in group-major order; each block takes a
  // contiguous run, so consecutive items of one group reuse the A operand and
  // keep one candidate list per read across their ranges
  const int64_t n_items = (int64_t)a.n_groups * a.n_ranges;
  const int64_t it_lo = n_items * blockIdx.x / gridDim.x;
  const int64_t it_hi = n_items * (blockIdx.x + 1) / gridDim.x;
  // first window and super-tiles of an item's range
  auto range_of = [&](int64_t item, int64_t& st_begin) -> int64_t {
    st_begin = a.st0 + (item % a.n_ranges) * a.range_len;
    return (min(st_begin + a.range_len, a.je) - st_begin + Sh::SUP - 1) / Sh::SUP;
  };
  // read tiles of an item's group that hold reads (the others are skipped by
  // the MMA threads and their epilogue warps alike)
  auto live_tiles = [&](int64_t item) -> int {
    const int64_t left = a.n_reads - (item / a.n_ranges) * Sh::GROUP;
    return left >= Sh::GROUP ? NT : (int)((left + 127) / 128);
  };

  if (warp < Sh::EPI_WARPS) {
    // ================================================================ epilogue
    // warp = (share w, tile, lane quarter q); share w holds windows
    // [w*WPH, (w+1)*WPH) of each stage and a candidate list per read over them.
    const int q = warp & 3;
    const int tile = (warp >> 2) % NT;
    const int w = warp / (4 * NT);
    const int rs = tile * 128 + 32 * q + lane;  // read slot in the group
    const int arow = 32 * q + lane;             // its row in the A tile
    constexpr int lstride = Sh::GROUP * Sh::LH;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    uint32_t use = 0;      // accumulators of this tile consumed
    int prev_grp = -1;     // read group of the list being kept
    int seg_rng = 0;       // range whose slot receives that list
    // threshold: the list's worst kept score (+inf for a missing read, whose list takes nothing)
    float thr_list = INFINITY;
    const ListRef lref{smem_u32(queues + w * Sh::GROUP + rs), smem_u32(list_s + w * Sh::GROUP + rs),
                       4u * a.cand_depth * Sh::GROUP * Sh::LH, a.cand_depth, a.sep, S, L.pend};
    // writes the kept list of read r to the slot of range rng
    auto flush = [&](int64_t r, int rng) {
      const float* ls = list_s + w * Sh::GROUP + rs;
      const uint32_t* lw = list_w + w * Sh::GROUP + rs;
      Candidate* out = a.cand + (((size_t)r * a.n_ranges + rng) * Sh::LH + w) * a.cand_depth;
      for (int e = 0; e < a.cand_depth; ++e) out[e] = Candidate{ls[e * lstride] * Sh::SCORE_SCALE, lw[e * lstride]};
    };
    for (int64_t item = it_lo; item < it_hi; ++item) {
      const int grp = (int)(item / a.n_ranges);
      const int rng = (int)(item % a.n_ranges);
      const int64_t r = (int64_t)grp * Sh::GROUP + rs;
      const bool have_read = r < a.n_reads;
      int64_t st_begin;
      const int64_t n_st = range_of(item, st_begin);
      // window numbers fit in 32 bits with room for a super-tile past the last
      // window (the index refuses W > 2^32 - 2^16)
      const uint32_t jlo = (uint32_t)max(st_begin, a.jb);
      const uint32_t jhi = (uint32_t)min(st_begin + a.range_len, a.je);
      if (grp != prev_grp) {
        // a new read group: hand over the previous group's list, load the A
        // operand and start an empty list. The previous item's MMAs on this
        // tile have all completed: its warps consumed every accumulator.
        if (kLists && prev_grp >= 0) {
          const int64_t pr = (int64_t)prev_grp * Sh::GROUP + rs;
          flush_all<Sh>(lref, thr_list);
          if (pr < a.n_reads) flush(pr, seg_rng);
        }
        if (w == 0) {
          // this read's normalised BF16 row, 16-byte chunks into the swizzled
          // tile (E4M3: each chunk of 8 entries scaled, rounded and written as 8 bytes)
          const uint4* src = reinterpret_cast<const uint4*>(a.emb_bf16 + (have_read ? r : 0) * 2 * D);
          uint8_t* arow_base = a_tiles + tile * Sh::A_TILE_BYTES;
#pragma unroll
          for (int c = 0; c < 2 * D / 8; ++c) {
            const uint4 v = have_read ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
            const int byte = c * 8 * Sh::EB;  // first byte of the chunk in the operand row
            uint8_t* dst = arow_base + (byte / Sh::KBLK) * Sh::A_KBLK_BYTES +
                           Sh::swz((uint32_t)arow, (uint32_t)(byte % Sh::KBLK));
            if constexpr (Sh::FP8) {
              *reinterpret_cast<uint2*>(dst) = make_uint2(bf16x4_to_e4m3(v.x, v.y), bf16x4_to_e4m3(v.z, v.w));
            } else {
              *reinterpret_cast<uint4*>(dst) = v;
            }
          }
          fence_proxy_async_smem();
        }
        thr_list = have_read ? -INFINITY : INFINITY;
        if (kLists) {
          sts_u32(lref.queue, 0u);
          float* ls = list_s + w * Sh::GROUP + rs;
          uint32_t* lw = list_w + w * Sh::GROUP + rs;
          for (int e = 0; e < a.cand_depth; ++e) {
            ls[e * lstride] = -INFINITY;
            lw[e * lstride] = kEmptyWin;
          }
        }
        prev_grp = grp;
        seg_rng = rng;
      } else if (kLists && have_read) {
        // the list carries on: this range's own slot holds no list
        a.cand[(((size_t)r * a.n_ranges + rng) * Sh::LH + w) * a.cand_depth].win = kUnusedWin;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_aready);
      if (tile >= live_tiles(item)) {
        // no reads in this tile: keep in step with the others, one arrival per item
        if (!mbar_wait_warp(&bar_aready, (uint32_t)(item - it_lo) & 1u, abort_flag, a.status, wlim)) goto epi_done;
        continue;
      }
      // stages of the range, 32-bit: A per super-tile; column n holds window jbase + n*A
      uint32_t jbase = (uint32_t)st_begin;
      const uint32_t j_end = jbase + (uint32_t)(n_st * Sh::SUP);
      while (jbase != j_end) {
        {
          const uint32_t acc = (use % STG) * NT + tile;
          if (!mbar_wait_warp(&bar_afull[acc], (use / STG) & 1, abort_flag, a.status, wlim)) goto epi_done;
          tc_fence_after();
          const uint32_t tcol = tbase + lane_base + acc * 2 * T + w * Sh::WPH;
          if constexpr (kLists) {
            // Hot path. The tensor-memory load itself reduces each 16-column
            // chunk to max|Re| and max|Im| (tcgen05.ld.red): squares and sums
            // round monotonically, so no score of the chunk exceeds mr^2 + mi^2
            // rounded the same way, and a chunk whose bound stays below the
            // thresholds of all 32 reads costs two loads and three operations
            // instead of the 16 scores and their maximum. A bound that reaches a
            // threshold is looked at exactly (the columns are in registers).
            // Forming every score measured 450 ms, this 385 ms (16,384 reads x
            // 100 M windows); with lists of under ~10^6 windows, where half of
            // the bounds pass, the two are equal.
            constexpr int NCH = Sh::WPH / 16;
            uint32_t todo = 0;  // chunks with something to offer in this lane
#pragma unroll
            for (int u = 0; u < NCH; ++u) {
              uint32_t vr[16], vi[16];
              float mr, mi;
              tmem_ld16_absmax(tcol + 16 * u, vr, mr);
              tmem_ld16_absmax(tcol + T + 16 * u, vi, mi);
              tc_wait_ld();
              reg_fence(vr);
              reg_fence(vi);
              reg_fence(mr, mi);
              if (__any_sync(0xffffffffu, fmaf(mr, mr, mi * mi) >= thr_list)) todo |= max_abs2(vr, vi) >= thr_list ? 1u << u : 0u;
            }
            if (__any_sync(0xffffffffu, todo != 0)) {
              todo = __reduce_or_sync(0xffffffffu, todo);
              thr_list = offer_chunks<Sh>(lref, tcol, todo, jbase + (uint32_t)(w * Sh::WPH * A), jlo, jhi, thr_list,
                                      &bar_aempty[acc]);
            } else {
              // nothing to offer: hand the accumulator back
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&bar_aempty[acc]);
            }
          } else {
            // threshold mode: lane l holds the thresholds of this warp's
            // columns w*WPH + 32u + l (+inf outside the scanned range), and each
            // 16-column chunk's smallest threshold is known to all lanes
            constexpr int TPL = kThr ? Sh::WPH / 32 : 1;
            float thr_lane[TPL], thr_min[2 * TPL];
            if constexpr (kThr) {
              static_assert(Sh::WPH % 32 == 0, "threshold mode: whole columns per lane");
#pragma unroll
              for (int u = 0; u < TPL; ++u) {
                const uint32_t jl = jbase + (uint32_t)((w * Sh::WPH + 32 * u + lane) * A);
                thr_lane[u] = (jl >= jlo && jl < jhi) ? __ldg(L.thr.thr + jl) : INFINITY;
                float mn = thr_lane[u];
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                thr_min[2 * u] = __shfl_sync(0xffffffffu, mn, 0);
                thr_min[2 * u + 1] = __shfl_sync(0xffffffffu, mn, 16);
              }
            }
#pragma unroll
            for (int c0 = 0; c0 < Sh::WPH; c0 += 16) {
              uint32_t vr[16], vi[16];
              float mr, mi;
              tmem_ld16_absmax(tcol + c0, vr, mr);
              tmem_ld16_absmax(tcol + T + c0, vi, mi);
              tc_wait_ld();
              reg_fence(vr);
              reg_fence(vi);
              reg_fence(mr, mi);
              const uint32_t jc = jbase + (uint32_t)((w * Sh::WPH + c0) * A);
              float sc[16];
              if constexpr (kThr) {
                // the bound of the hot path above against the chunk's smallest threshold
                const bool any = have_read && fmaf(mr, mr, mi * mi) * Sh::SCORE_SCALE >= thr_min[c0 >> 4];
                if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                for (int n = 0; n < 16; n += 2) abs2_pair(vr[n], vr[n + 1], vi[n], vi[n + 1], sc[n], sc[n + 1]);
#pragma unroll
                for (int n = 0; n < 16; ++n) {
                  const float th = __shfl_sync(0xffffffffu, thr_lane[c0 >> 5], (c0 & 31) + n);
                  const float v = sc[n] * Sh::SCORE_SCALE;
                  if (have_read && v >= th) {
                    const unsigned long long slot = atomicAdd(L.thr.count, 1ull);
                    if (slot < (unsigned long long)L.thr.cap) {
                      L.thr.read[slot] = r;
                      L.thr.win[slot] = (int64_t)(jc + (uint32_t)(n * A));
                      L.thr.score[slot] = v;
                    }
                  }
                }
              } else if (have_read) {
#pragma unroll
                for (int n = 0; n < 16; n += 2) abs2_pair(vr[n], vr[n + 1], vi[n], vi[n + 1], sc[n], sc[n + 1]);
#pragma unroll
                for (int n = 0; n < 16; ++n) {
                  const uint32_t j = jc + (uint32_t)(n * A);
                  if (j >= jlo && j < jhi) a.dense[r * (a.je - a.jb) + ((int64_t)j - a.jb)] = sc[n] * Sh::SCORE_SCALE;
                }
              }
            }
          }
          if (!kLists) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_aempty[acc]);
          }
          ++use;
          ++jbase;
          if ((jbase & (A - 1)) == 0) jbase += Sh::SUP - A;
        }
      }
    }
    if (kLists && prev_grp >= 0) {
      const int64_t pr = (int64_t)prev_grp * Sh::GROUP + rs;
      flush_all<Sh>(lref, thr_list);
      if (pr < a.n_reads) flush(pr, seg_rng);
    }
  epi_done:;
  } else if (Sh::mma_index(warp) >= 0) {
    // ================================================================ MMA issue
    // NM issuing threads; thread x takes the (stage k, read tile t) units with
    // (k NT + t) mod NM = x. A single thread's path through a unit (two barrier
    // waits, the MMAs, two commits) is longer than the tensor pipe's time for
    // it; with several in turn the pipe does not wait for it.
    //
    // A wait names a fill of a slot by its parity alone, so a thread may wait for
    // a stage only once the slot's previous fill is complete. A thread that waits
    // for stage k has seen stage k - STEP filled, and with it (generators fill in
    // order) every earlier one: the slot's previous fill, stage k - nb, is among
    // them if nb >= STEP. The launch takes a shape with one issuer per tile where
    // shared memory leaves fewer slots.
    if (lane == 0) {
      constexpr int STEP = Sh::STEP;  // a thread's units lie in every STEP-th stage
      const int x = Sh::mma_index(warp);
      const int t = x % NT;
      uint32_t it = 0, use = 0;
      uint32_t slot = x / NT, phase = 0;  // window slot of its next unit
      while (slot >= (uint32_t)L.nb) {
        slot -= L.nb;
        phase ^= 1u;
      }
      bool ok = true;
      const uint64_t tile_desc = Sh::desc(smem_u32(a_tiles + t * Sh::A_TILE_BYTES));
      const uint64_t b_desc0 = Sh::desc(smem_u32(b_ring));
      for (int64_t item = it_lo; item < it_hi && ok; ++item, ++it) {
        int64_t st_begin;
        const uint32_t n_unit = (uint32_t)(range_of(item, st_begin) * A) / STEP;
        const bool live = t < live_tiles(item);
        if (!mbar_wait(&bar_aready, it & 1, abort_flag, a.status, wlim)) break;
        for (uint32_t k = 0; k < n_unit; ++k) {
          if (!mbar_wait(&bar_bfull[slot], phase, abort_flag, a.status, wlim)) { ok = false; break; }
          if (live) {
            const uint32_t acc = STEP == 1 ? (use % STG) * NT + t : x;
            const uint32_t turn = STEP == 1 ? use / STG : use;
            if (!mbar_wait(&bar_aempty[acc], (turn & 1) ^ 1, abort_flag, a.status, wlim)) { ok = false; break; }
            ++use;
            tc_fence_after();
            const uint32_t d_tmem = tbase + acc * 2 * T;
            // descriptors differ only in the start-address field (16-byte units)
            const uint64_t slot_desc = b_desc0 + (uint64_t)((slot * Sh::B_SLOT_BYTES) >> 4);
#pragma unroll
            for (int kk = 0; kk < Sh::KSTEPS; ++kk) {
              const uint32_t kb = kk / Sh::STEPS_PER_KBLK, ko = (kk % Sh::STEPS_PER_KBLK) * 32;
              const uint64_t ad = tile_desc + (uint64_t)((kb * Sh::A_KBLK_BYTES + ko) >> 4);
              const uint64_t bd = slot_desc + (uint64_t)((kb * Sh::B_KBLK_BYTES + ko) >> 4);
              if constexpr (Sh::FP8) {
                tc_mma_ss_f8(d_tmem, ad, bd, Sh::IDESC, kk > 0 ? 1u : 0u);
              } else {
                tc_mma_ss(d_tmem, ad, bd, Sh::IDESC, kk > 0 ? 1u : 0u);
              }
            }
            tc_commit(&bar_afull[acc]);
            tc_commit(&bar_bempty[slot]);
          } else {
            mbar_arrive(&bar_bempty[slot]);  // no reads in this tile: nothing reads the slot
          }
          slot += STEP;
          while (slot >= (uint32_t)L.nb) {
            slot -= L.nb;
            phase ^= 1u;
          }
        }
      }
      // drain: every MMA issued by this thread has completed (waited for even
      // after an abort, so that tensor memory is freed with no MMA in flight)
      tc_commit(&bar_drain[x]);
      mbar_drain_wait(&bar_drain[x], 0, a.status, wlim);
    }
  } else if (warp == Sh::WARP_BIN) {
    // ================================================================ bins
    // One warp stays a super-tile ahead of the generators: lane 0 streams the
    // packed reference of the next super-tile into shared memory by a bulk copy
    // (TMA) while all lanes turn the current one's letters into bins, so that
    // the generators' step loop waits for neither.
    int64_t p_item = it_lo, p_sti = 0, p_begin = 0, p_n = 0;  // the next super-tile to copy
    uint32_t issued = 0;
    if (p_item < it_hi) p_n = range_of(p_item, p_begin);
    auto copy_next = [&]() {
      if (p_item >= it_hi) return;
      if (lane == 0) {
        const int64_t word0 = (((p_begin + p_sti * Sh::SUP) * S) >> 4) & ~int64_t(3);
        const uint32_t wbytes = (uint32_t)L.words_per_slot * 4u;
        mbar_expect_tx(&bar_stfull[issued & 1], wbytes);
        bulk_g2s(st_slots + (issued & 1) * L.st_slot_bytes, ix.packed + word0, wbytes, &bar_stfull[issued & 1]);
      }
      ++issued;
      if (++p_sti == p_n) {
        p_sti = 0;
        if (++p_item < it_hi) p_n = range_of(p_item, p_begin);
      }
    };
    copy_next();
    uint32_t g = 0;
    const int in_off = ix.N - ix.s + 1;  // entering location relative to the leaving one
    bool ok = true;
    for (int64_t item = it_lo; item < it_hi && ok; ++item) {
      int64_t st_begin;
      const int64_t n_st = range_of(item, st_begin);
      for (int64_t sti = 0; sti < n_st; ++sti, ++g) {
        copy_next();  // into the slot whose letters (super-tile g-1) every lane has read
        const int64_t st = st_begin + sti * Sh::SUP;
        if (!mbar_wait_warp(&bar_stfull[g & 1], (g >> 1) & 1, abort_flag, a.status, wlim)) { ok = false; break; }
        const uint32_t buf = L.n_bin == 2 ? (g & 1) : 0u, turn = L.n_bin == 2 ? (g >> 1) : g;
        if (!mbar_wait_warp(&bar_binempty[buf], (turn & 1) ^ 1u, abort_flag, a.status, wlim)) { ok = false; break; }
        const uint32_t* words = reinterpret_cast<const uint32_t*>(st_slots + (g & 1) * L.st_slot_bytes);
        uint8_t* bt = bins_t + buf * L.bins_bytes;
        const uint32_t rel0 = (uint32_t)(st * S - ((((st * S) >> 4) & ~int64_t(3)) << 4));
        if (S == 1) {
          // rows of A leaving bins per chain, then rows of A entering bins; the
          // row pitch keeps the chains of a generator warp in distinct banks
#pragma unroll 2
          for (int t4 = lane; t4 < 2 * Sh::SUP / 4; t4 += 32) {
            const int t = (t4 % (Sh::SUP / 4)) * 4;
            const bool in = t4 >= Sh::SUP / 4;
            const uint32_t b = bins4_staged(words, rel0 + t + (in ? in_off : 0), ix.s, ix.map_lsb);
            *reinterpret_cast<uint32_t*>(bt + ((in ? T : 0) + t / A) * Sh::BIN_PITCH + t % A) = b;
          }
        } else {
          // one bin per location of the super-tile, shared by all chains
          const int n_pos = Sh::SUP * S + in_off;
#pragma unroll 2
          for (int t = 4 * lane; t < n_pos; t += 128)
            *reinterpret_cast<uint32_t*>(bt + t) = bins4_staged(words, rel0 + t, ix.s, ix.map_lsb);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_binfull[buf]);
      }
    }
    // wait for the copies still in flight into either slot (the latest phase
    // of each), also after an abort: the block's shared memory must not be
    // released with a copy still writing to it
    if (lane == 0)
      for (uint32_t c = (issued >= 2 ? issued - 2 : 0); c < issued; ++c)
        mbar_drain_wait(&bar_stfull[c & 1], (c >> 1) & 1, a.status, wlim);
  } else if (Sh::gen_index(warp) >= 0) {
    // ================================================================ window generators
    const int gw = Sh::gen_index(warp);
    const int chain = gw * Sh::CPW + lane / Sh::LPC;  // B row (Re) and column of its windows
    const int lic = lane % Sh::LPC;
    ChainB<BPL> ch;
    ch.setup(ix, lic);
    // byte offsets of this lane's pieces in a B slot: row chain = [cr | ci],
    // row T+chain = [ci | -cr]; BPL entries = BPL*EB bytes per half-row,
    // written as one 8-byte piece or 16-byte pieces
    constexpr int NPC = Sh::NPC;
    uint32_t off_re_cr[NPC], off_re_ci[NPC], off_im_ci[NPC], off_im_cr[NPC];
    {
      auto off = [&](int row, int e) -> uint32_t {
        const int byte = e * Sh::EB;
        return (uint32_t)((byte / Sh::KBLK) * Sh::B_KBLK_BYTES) + Sh::swz((uint32_t)row, (uint32_t)(byte % Sh::KBLK));
      };
#pragma unroll
      for (int pc = 0; pc < NPC; ++pc) {
        const int e_lo = BPL * lic + pc * Sh::PIECE / Sh::EB, e_hi = D + e_lo;
        off_re_cr[pc] = off(chain, e_lo);
        off_re_ci[pc] = off(chain, e_hi);
        off_im_ci[pc] = off(T + chain, e_lo);
        off_im_cr[pc] = off(T + chain, e_hi);
      }
    }
    uint32_t g = 0, bslot = 0, bphase = 0;
    const int in_off = ix.N - ix.s + 1;  // entering location relative to the leaving one
    // the current window, scaled by nv and rounded, into the next B slot
    auto emit = [&](float nv) -> bool {
      if (Sh::FP8) nv *= kFp8Scale;
      // packed operand words of cr, ci and -cr (sign bits flipped)
      constexpr int NW = BPL * Sh::EB / 4;
      uint32_t pr[NW], pi[NW], pn[NW];
#pragma unroll
      for (int hh = 0; hh < NW; ++hh) {
        if constexpr (Sh::FP8) {
          pr[hh] = f32x4_to_e4m3(ch.cr[4 * hh] * nv, ch.cr[4 * hh + 1] * nv, ch.cr[4 * hh + 2] * nv,
                                 ch.cr[4 * hh + 3] * nv);
          pi[hh] = f32x4_to_e4m3(ch.ci[4 * hh] * nv, ch.ci[4 * hh + 1] * nv, ch.ci[4 * hh + 2] * nv,
                                 ch.ci[4 * hh + 3] * nv);
          pn[hh] = pr[hh] ^ 0x80808080u;
        } else {
          const __nv_bfloat162 rr = __floats2bfloat162_rn(ch.cr[2 * hh] * nv, ch.cr[2 * hh + 1] * nv);
          const __nv_bfloat162 ii = __floats2bfloat162_rn(ch.ci[2 * hh] * nv, ch.ci[2 * hh + 1] * nv);
          pr[hh] = *reinterpret_cast<const uint32_t*>(&rr);
          pi[hh] = *reinterpret_cast<const uint32_t*>(&ii);
          pn[hh] = pr[hh] ^ 0x80008000u;
        }
      }
      if (!mbar_wait_warp(&bar_bempty[bslot], bphase ^ 1u, abort_flag, a.status, wlim)) return false;
      uint8_t* bt = b_ring + bslot * Sh::B_SLOT_BYTES;
      if constexpr (Sh::PIECE == 8) {
        *reinterpret_cast<uint2*>(bt + off_re_cr[0]) = make_uint2(pr[0], pr[1]);
        *reinterpret_cast<uint2*>(bt + off_re_ci[0]) = make_uint2(pi[0], pi[1]);
        *reinterpret_cast<uint2*>(bt + off_im_ci[0]) = make_uint2(pi[0], pi[1]);
        *reinterpret_cast<uint2*>(bt + off_im_cr[0]) = make_uint2(pn[0], pn[1]);
      } else {
#pragma unroll
        for (int pc = 0; pc < NPC; ++pc) {
          const int o = 4 * pc;
          *reinterpret_cast<uint4*>(bt + off_re_cr[pc]) = make_uint4(pr[o], pr[o + 1], pr[o + 2], pr[o + 3]);
          *reinterpret_cast<uint4*>(bt + off_re_ci[pc]) = make_uint4(pi[o], pi[o + 1], pi[o + 2], pi[o + 3]);
          *reinterpret_cast<uint4*>(bt + off_im_ci[pc]) = make_uint4(pi[o], pi[o + 1], pi[o + 2], pi[o + 3]);
          *reinterpret_cast<uint4*>(bt + off_im_cr[pc]) = make_uint4(pn[o], pn[o + 1], pn[o + 2], pn[o + 3]);
        }
      }
      return true;
    };
    // the written slot to the MMA threads
    auto publish = [&]() {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_bfull[bslot]);
      if (++bslot == (uint32_t)L.nb) {
        bslot = 0;
        bphase ^= 1u;
      }
    };
    for (int64_t item = it_lo; item < it_hi; ++item) {
      int64_t st_begin;
      const int64_t n_st = range_of(item, st_begin);
      for (int64_t sti = 0; sti < n_st; ++sti, ++g) {
        const int64_t st = st_begin + sti * Sh::SUP;
        // this chain's norms, and its anchor (both padded past the last window)
        const float* inv = ix.inv_norm + st + chain * A;
        ch.load(ix.anchors + (st / A + chain) * D, lic);
        const uint32_t buf = L.n_bin == 2 ? (g & 1) : 0u, turn = L.n_bin == 2 ? (g >> 1) : g;
        if (S == 1) {
          // four windows' norms and bins per load, one load ahead
          float4 nv = __ldg(reinterpret_cast<const float4*>(inv));
          if (!mbar_wait_warp(&bar_binfull[buf], turn & 1, abort_flag, a.status, wlim)) goto gen_done;
          const uint8_t* bo = bins_t + buf * L.bins_bytes + chain * Sh::BIN_PITCH;
          uint32_t o4 = *reinterpret_cast<const uint32_t*>(bo);
          uint32_t n4 = *reinterpret_cast<const uint32_t*>(bo + T * Sh::BIN_PITCH);
#pragma unroll 1
          for (int i = 0; i < A; i += 4) {
            const float nq[4] = {nv.x, nv.y, nv.z, nv.w};
            const uint32_t co = o4, cn = n4;
            if (i + 4 < A) {
              nv = __ldg(reinterpret_cast<const float4*>(inv + i + 4));
              o4 = *reinterpret_cast<const uint32_t*>(bo + i + 4);
              n4 = *reinterpret_cast<const uint32_t*>(bo + T * Sh::BIN_PITCH + i + 4);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (!emit(nq[u])) goto gen_done;
              // the step's arithmetic overlaps the stores that the fence waits for
              ch.step1((co >> (8 * u)) & 0xFFu, (cn >> (8 * u)) & 0xFFu);
              publish();
            }
          }
        } else {
          float nv = __ldg(inv);
          if (!mbar_wait_warp(&bar_binfull[buf], turn & 1, abort_flag, a.status, wlim)) goto gen_done;
          const uint8_t* bl = bins_t + buf * L.bins_bytes;
          const float2* eo = e_tab[0] + ch.band * S;
          const float2* ei = e_tab[1] + ch.band * S;
          for (int i = 0; i < A; ++i) {
            const float nx = i + 1 < A ? __ldg(inv + i + 1) : 0.f;
            if (!emit(nv)) goto gen_done;
            publish();
            nv = nx;
            const int base = (chain * A + i) * S;
            for (int u = 0; u < S; ++u) {
              ch.sub_at(bl[base + u], eo[u]);
              ch.add_at(bl[base + in_off + u], ei[u]);
            }
            ch.rotate();
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_binempty[buf]);
      }
    }
  gen_done:;
  }

  tc_fence_before();
  __syncthreads();
  if (warp == Sh::WARP_MMA) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tbase, Sh::TMEM_COLS);
  }
}

// ---------------------------------------------------------------- configurations

// d = 64:  256 reads x 64 windows per stage, MMA N = 128; 16 epilogue warps (two
//          per accumulator quarter, a list each), 8 generator warps (chains of 4
//          lanes x 8 entries), four issuers, up to 6 window slots between
//          generators and MMAs; 29 warps of 64 registers. With 8 epilogue warps
//          (the second variant) 416 instead of 385 ms on 16,384 reads x 100 M
//          windows; with two issuers (27 warps of 72 registers) 445 ms.
using TcShape32 = TcShape<32, 2, 64, 6, 4, 2, 4, false>;
// d = 64, second tile variant: one epilogue warp per accumulator quarter and
//          tile (8 warps, each reading all 64 windows of a stage; one candidate
//          list per read), more registers per thread. Faster at large strides.
using TcShape32b = TcShape<32, 2, 64, 4, 4, 1, 4, true>;
// d = 64, third tile variant: 512 reads (4 tiles) x 32 windows per stage, MMA
//          N = 64 (twice the MMA instructions per score), super-tiles of half
//          the windows: a finer split of short references.
using TcShape32c = TcShape<32, 4, 32, 4, 4, 1, 4, false>;
// d = 128: 256 reads x 64 windows per stage, MMA N = 128 (twice the tensor time
//          per stage); 8 epilogue warps, 16 generator warps (chains of 8 lanes x 8 entries)
using TcShape64 = TcShape<64, 2, 64, 2, 8, 1, 2, false>;
// the same tiles with E4M3 operands (kind::f8f6f4): half the operand bytes,
// half the MMA instructions per stage; 64-byte swizzled rows at d = 64
using TcShape32f8 = TcShape<32, 2, 64, 4, 4, 2, 4, false, true>;
using TcShape32bf8 = TcShape<32, 2, 64, 4, 4, 1, 4, true, true>;
using TcShape32cf8 = TcShape<32, 4, 32, 4, 4, 1, 4, false, true>;
using TcShape64f8 = TcShape<64, 2, 64, 2, 8, 1, 2, false, true>;

// Dynamic shared memory one block of this kernel may take: the device's
// opt-in maximum per block less the kernel's static shared memory (barriers,
// phase tables). 0 if the attributes cannot be read.
// Read once per device and kept (so that launches made while a stream is
// being captured into a graph query nothing).
constexpr int kMaxDevices = 64;

template <class Sh, bool kDense, bool kThr = false>
static size_t tc_dyn_limit() {
  static size_t cached[kMaxDevices] = {};  // value + 1, 0 = not read yet
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return 0;
  }
  if (cached[dev]) return cached[dev] - 1;
  cudaFuncAttributes fa{};
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, scan_tc_kernel<Sh, kDense, kThr>) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t v = optin > (int)fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
  cached[dev] = v + 1;
  return v;
}

int scan_tc_supported(int D) { return D == 32 || D == 64; }

int64_t scan_tc_super_tile(int D, int variant) {
  if (D == 32) return variant == 2 ? TcShape32c::SUP : TcShape32::SUP;
  return D == 64 ? TcShape64::SUP : 0;
}

int scan_tc_group(int D, int variant) {
  if (D == 32) return variant == 2 ? TcShape32c::GROUP : TcShape32::GROUP;
  return D == 64 ? TcShape64::GROUP : 0;
}

int scan_tc_max_stride() { return 8; }

int scan_tc_variants(int D) { return D == 32 ? 3 : D == 64 ? 1 : 0; }

int scan_tc_lists_per_range(int D, int variant) {
  if (D == 32) return variant == 1 ? TcShape32b::LH : variant == 2 ? TcShape32c::LH : TcShape32::LH;
  return D == 64 ? TcShape64::LH : 1;
}

// Dynamic shared memory with nb B slots, n_bin buffers of bins and queues of pend entries.
template <class Sh>
static size_t tc_smem_bytes(const DevIndex& ix, int cand_depth, bool lists, int nb, int n_bin, int pend, TcLaunch* Lout) {
  TcLaunch L;
  L.nb = nb;
  L.n_bin = n_bin;
  L.pend = pend;
  const int S = ix.stride;
  int64_t words = ((int64_t)Sh::SUP * S + ix.N + 64) / 16 + 8;
  words = (words + 3) & ~int64_t(3);
  L.words_per_slot = (int32_t)words;
  int64_t slot = words * 4;
  slot = (slot + 127) & ~int64_t(127);
  L.st_slot_bytes = (int32_t)slot;
  // stride 1: a row of leaving and a row of entering bins per chain; stride > 1:
  // one bin per location of the super-tile, shared by the chains
  L.bins_bytes = S == 1 ? 2 * Sh::T * Sh::BIN_PITCH : (int32_t)((Sh::SUP * S + ix.N - ix.s + 1 + 15) & ~15);
  const size_t list_bytes =
      lists ? (size_t)cand_depth * Sh::GROUP * Sh::LH * 8 + (size_t)queue_words(pend) * Sh::GROUP * Sh::EW * 4 : 0;
  if (Lout) *Lout = L;
  return 1024 + (size_t)Sh::NT * Sh::A_TILE_BYTES + (size_t)nb * Sh::B_SLOT_BYTES + 2 * (size_t)L.st_slot_bytes +
         (size_t)n_bin * L.bins_bytes + list_bytes;
}

// The same tiles with one MMA issuer per read tile, for a ring of one slot.
template <class Sh>
using TcOneSlot = TcShape<Sh::D, Sh::NT, Sh::T, 1, Sh::LPC, Sh::EW, Sh::NT, Sh::ISOLATE_MMA, Sh::FP8>;

// The most B slots, with two buffers of bins before one and whole queues before
// shorter ones, that fit in `limit` bytes; 0 if none do. Where a tile has two MMA
// issuers, two slots with a shorter queue come before one slot.
template <class Sh>
static size_t tc_plan_smem(const DevIndex& ix, int cand_depth, bool lists, size_t limit, TcLaunch* L) {
  for (int n_bin = 2; n_bin >= 1; --n_bin)
    for (int nb = Sh::NB; nb >= 2; --nb) {
      const size_t b = tc_smem_bytes<Sh>(ix, cand_depth, lists, nb, n_bin, kPend, L);
      if (b <= limit) return b;
    }
  for (int nb = Sh::STEP; nb >= 1; --nb)
    for (int pend = kPend; pend >= 1; --pend) {
      const size_t b = tc_smem_bytes<Sh>(ix, cand_depth, lists, nb, 1, pend, L);
      if (b <= limit) return b;
    }
  return 0;
}

// Whether the scan takes candidate lists of this depth: tiles, lists and one B
// slot beside a super-tile of window norms and one byte per chain and step of
// leaving and entering bins. The launch itself needs less (no norms in shared
// memory, and queues that can shrink to one entry), so every depth this takes
// has a plan; the rule is kept so that the depths it takes do not move.
template <class Sh>
static int tc_fits(const DevIndex& ix, int cand_depth) {
  constexpr size_t kBarriers = 64;  // static shared memory beyond what the rule was written for
  const size_t queue = (size_t)queue_words(1) * Sh::GROUP * Sh::EW * 4;
  const size_t bins = ix.stride == 1 ? (size_t)2 * Sh::T * (Sh::BIN_PITCH - Sh::A) : 0;
  static_assert(queue_words(1) * Sh::GROUP * Sh::EW * 4 + 2 * Sh::T * (Sh::BIN_PITCH - Sh::A) + 128 <= Sh::SUP * 4,
                "a plan exists wherever the rule holds");
  return tc_smem_bytes<Sh>(ix, cand_depth, true, 1, 1, 1, nullptr) - queue - bins + (size_t)Sh::SUP * 4 <=
         tc_dyn_limit<Sh, false>() + kBarriers;
}

int scan_tc_fits(const DevIndex& ix, int cand_depth, int variant, int fp8) {
  if (ix.D == 32 && variant == 1) return fp8 ? tc_fits<TcShape32bf8>(ix, cand_depth) : tc_fits<TcShape32b>(ix, cand_depth);
  if (ix.D == 32 && variant == 2) return fp8 ? tc_fits<TcShape32cf8>(ix, cand_depth) : tc_fits<TcShape32c>(ix, cand_depth);
  if (ix.D == 32) return fp8 ? tc_fits<TcShape32f8>(ix, cand_depth) : tc_fits<TcShape32>(ix, cand_depth);
  if (ix.D == 64) return fp8 ? tc_fits<TcShape64f8>(ix, cand_depth) : tc_fits<TcShape64>(ix, cand_depth);
  return 0;
}

template <class Sh, bool kDense, bool kThr = false>
static cudaError_t launch_tc(const DevIndex& ix, const ScanArgs& a, int num_sms, cudaStream_t st,
                             const ThrOut* thr = nullptr) {
  // the deepest B ring that fits (long windows at large strides and deep
  // candidate lists leave room for fewer slots)
  TcLaunch L;
  const size_t smem = tc_plan_smem<Sh>(ix, a.cand_depth, !(kDense || kThr), tc_dyn_limit<Sh, kDense, kThr>(), &L);
  if (smem == 0) return cudaErrorInvalidValue;
  if constexpr (Sh::STEP > 1) {
    if (L.nb < Sh::STEP) {
      // (without lists two slots always fit: 214 KB at the longest windows and the largest stride)
      if constexpr (kDense || kThr) return cudaErrorInvalidValue;
      else return launch_tc<TcOneSlot<Sh>, kDense, kThr>(ix, a, num_sms, st, thr);
    }
  }
  L.thr = thr ? *thr : ThrOut{};
  auto kern = scan_tc_kernel<Sh, kDense, kThr>;
  const cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const int64_t n_items = (int64_t)a.n_groups * a.n_ranges;
  const int grid = (int)(num_sms < n_items ? num_sms : n_items);
  if (grid < 1) return cudaSuccess;
  kern<<<grid, Sh::NTHREADS, smem, st>>>(ix, a, L);
  return cudaGetLastError();
}

template <class Sh>
static cudaError_t launch_tc_any(const DevIndex& ix, const ScanArgs& a, bool dense, int num_sms, cudaStream_t st) {
  return dense ? launch_tc<Sh, true>(ix, a, num_sms, st) : launch_tc<Sh, false>(ix, a, num_sms, st);
}

cudaError_t launch_scan_tc(const DevIndex& ix, const ScanArgs& a, bool dense, int num_sms, cudaStream_t st) {
  if (ix.stride > scan_tc_max_stride()) return cudaErrorInvalidValue;
  if (ix.D == 32 && a.tc_variant == 1)
    return a.fp8 ? launch_tc_any<TcShape32bf8>(ix, a, dense, num_sms, st)
                 : launch_tc_any<TcShape32b>(ix, a, dense, num_sms, st);
  if (ix.D == 32 && a.tc_variant == 2)
    return a.fp8 ? launch_tc_any<TcShape32cf8>(ix, a, dense, num_sms, st)
                 : launch_tc_any<TcShape32c>(ix, a, dense, num_sms, st);
  if (ix.D == 32)
    return a.fp8 ? launch_tc_any<TcShape32f8>(ix, a, dense, num_sms, st)
                 : launch_tc_any<TcShape32>(ix, a, dense, num_sms, st);
  if (ix.D == 64)
    return a.fp8 ? launch_tc_any<TcShape64f8>(ix, a, dense, num_sms, st)
                 : launch_tc_any<TcShape64>(ix, a, dense, num_sms, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_scan_tc_threshold(const DevIndex& ix, const ScanArgs& a, const ThrOut& out, int num_sms,
                                     cudaStream_t st) {
  if (ix.stride > scan_tc_max_stride() || a.fp8) return cudaErrorInvalidValue;
  if (ix.D == 32) return launch_tc<TcShape32, false, true>(ix, a, num_sms, st, &out);
  if (ix.D == 64) return launch_tc<TcShape64, false, true>(ix, a, num_sms, st, &out);
  return cudaErrorInvalidValue;
}

}  // namespace rope
