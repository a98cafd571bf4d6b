// W4A16 grouped GEMM (dense projection, MoE gate_up, MoE down) on 4-bit weights expanded next to the tensor core:
//
//   y[t, n] = sum_k x[t, k] * w^[n, k],   w^ = bf16( s * (W_q - z) )  or  bf16( s * value )   (Dequant of Sec. 2.2)
//
// The 128 expanded WEIGHT rows of a block are the M side of tcgen05.mma and live in TENSOR MEMORY; NT token rows are
// its N side:
//   D[n, t] = sum_k w^[n, k] x[t, k]      (kind::f16, M = 128, N = NT, K = 16, A from TMEM)
// The bf16 products are exact, and the whole K reduction accumulates in TMEM in ascending k whatever NT is, so a
// token's output row has the same bits for every tile size and batch (App. C; the tests compare the sizes).
//
// Why tensor memory: expanded weights that travel through shared memory cost a 128-byte-per-clock port 2 bytes of
// stores and 2 of operand reads per weight.  Measured per 64 KB (256 rows x 128 k) on one SM: 616 clocks of stores with
// their proxy fences against 69 clocks of tcgen05.st, and an MMA 128 x 32 x 16 takes 40 clocks with A in shared
// memory (bound by reading A) against 16 with A in TMEM (its multiply rate).  What is left is the expansion's own
// arithmetic (measured 740 clocks per 64 KB for integer codes, 920 for e2m1 with its general scale: bf16x2 instructions
// issue at half rate) and, at decode, the weight stream.  Layer of 96 / 1024 / 4096 tokens (128 experts, top-8): integer 177 /
// 223 / 562 -> 113 / 170 / 467 us, e2m1 209 / 238 / 585 -> 121 / 188 / 472.
//
// A tile = (expert e, pair of weight blocks j, chunk of <= NT rows of the expert's group):
//   gate_up: blocks j (gate rows) and j + I/128 (the matching up rows); down/linear: blocks 2j, 2j+1.
// CTA: 8 epilogue warps (thread = weight row: TMEM -> SwiGLU / weighting -> bf16, transposed
// through shared memory so that global stores are whole token rows), 16 dequantization warps in two groups that take A
// stages in turn (thread = one of the pair's 256 weight rows), a producer warp for the codes (bulk copies into a
// shared-memory ring, scales and zero points with them), one for the token rows (TMA), two MMA issuers (one per block).
// TMEM: the accumulators of 2 NT columns (two with NT = 32 and 64; with NT = 128 one: four A stages instead of two keep
// the tensor pipe fed, and the exposed epilogue costs less), the rest A stages.
// What the hand-offs cost decides the stage sizes: a step of one issuing thread (two waits, its MMAs, the
// commits) takes 300-450 clocks whatever the MMAs, so codes and token rows move in 128-element quantization groups, and
// with NT = 32 an A stage is a whole group too (NT = 128: half of one, its MMAs take 512 clocks).
// Every barrier wait is bounded; an expired wait aborts the CTA cleanly.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "sched.cuh"
#include "w4_dequant.cuh"

namespace qarl {
namespace {

using namespace ptx;

constexpr int BW = 128;            // weight rows per block (UMMA M)
constexpr int BK = 64;             // bf16 elements per K-step (128 bytes)
constexpr uint32_t kQStepBytes = BW * BK / 2;  // 4 KB: 128 rows x 32 bytes of codes (one K-step of one block)
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxExperts = 1024;
constexpr int kOutRowBytes = 2 * BW * 2 + 16;  // bf16 row of 256 outputs, padded
constexpr uint32_t kPrefetchChunk = 32768;     // bytes per L2 prefetch instruction
constexpr int kMaxStages = 8;
// one quantization group of a pair of blocks in the ring: codes, then scales [2][128] bf16, zero points [2][128]
constexpr uint32_t kCodeBytes = 2 * 2 * kQStepBytes;
constexpr uint32_t kGroupBytes = kCodeBytes + 2 * BW * 2 + 2 * BW;

// NT = 32 for groups of a few rows (decode), kMid and kWide for larger ones.
constexpr int kNarrow = 32;
constexpr int kMid = 64;
constexpr int kWide = 128;
constexpr int kMaxAccBufs = 2;
constexpr int kDqWarps = 16;       // two groups of eight
template <int NT>
struct Cfg {
  // epilogue warps 0 ..: TMEM quadrant = warp % 4, warp / 4 = which token columns of it, 16 at a time
  static constexpr int kEpiWarps = 8;
  static constexpr int kCodeWarp = kEpiWarps + kDqWarps;             // producer of the codes
  static constexpr int kTokenWarp = kCodeWarp + 1;                   // producer of the token rows
  static constexpr int kMmaWarp = kCodeWarp + 2;                     // and + 3: one issuer per weight block
  static constexpr int kThreads = (kCodeWarp + 4) * 32;
  static constexpr uint32_t kXBytes = 2 * NT * BK * 2;               // token rows of one group: two boxes of 64 elements
  static constexpr int kXStages = NT == kWide ? 3 : 4;
  static constexpr int kQStages = NT == kNarrow ? 8 : NT == kMid ? 6 : 3;
  static constexpr int kAK = NT == kNarrow ? 2 : 1;                  // K-steps of 64 per A stage
  static constexpr int kStageCols = 2 * 32 * kAK;                    // two blocks
  static constexpr int kAccBufs = NT == kWide ? 1 : 2;
  static constexpr int kAStages = (static_cast<int>(kTmemCols) - kAccBufs * 2 * NT) / kStageCols;
  static constexpr uint32_t kABase = kAccBufs * 2 * NT;
};
static_assert(Cfg<kNarrow>::kAStages == 3 && Cfg<kWide>::kAStages == 4, "TMEM budget");

struct W4Params {
  const uint8_t* b_packed;   // tile-major 4 KB chunks [E][N/128][K/64]
  const uint16_t* b_scales;  // bf16 bits [E][K/128][N]
  const uint8_t* b_zeros;    // [E][K/128][N]
  const int32_t* offsets;
  int rows_total;
  int ksteps;                // K / 64 (even)
  int N;
  int E;
  int n_pairs;
  int I;
  int early_prefetch;
  int sz_bulk;               // scales and zero points are 16-byte aligned
  uint16_t* out_bf16;        // linear: y; down: contributions; gate_up (debug): bf16 gate_up
  float* out_f32;
  uint16_t* h_bf16;
  const float* pair_weights;
  int* status;
  unsigned long long wait_limit_ns;
  int stop_after_stages;     // test harness only (< 0: off): the producers stop arming stages after this many
};

struct __align__(8) SmemTail {
  uint64_t x_full[kMaxStages];
  uint64_t x_empty[kMaxStages];
  uint64_t q_full[kMaxStages];
  uint64_t q_empty[kMaxStages];
  uint64_t a_full[kMaxStages];
  uint64_t a_empty[kMaxStages];
  uint64_t tmem_full[kMaxAccBufs];
  uint64_t tmem_empty[kMaxAccBufs];
  uint64_t teardown[2];
  uint32_t tmem_addr;
  int abort_flag;
  float weight[2][kWide];      // down: the tile's pair weights, by tile parity
  int32_t off[kMaxExperts + 1];
  int32_t prefix[kMaxExperts + 1];
};

template <int NT>
constexpr size_t kSmemBytes = 1024 + static_cast<size_t>(Cfg<NT>::kXStages) * Cfg<NT>::kXBytes + static_cast<size_t>(Cfg<NT>::kQStages) * kGroupBytes +
                              static_cast<size_t>(NT) * kOutRowBytes + sizeof(SmemTail);
static_assert(kSmemBytes<kNarrow> <= 227 * 1024 && kSmemBytes<kMid> <= 227 * 1024 && kSmemBytes<kWide> <= 227 * 1024, "shared memory budget");

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const W4Params& p) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 128; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*reinterpret_cast<volatile int*>(&s->abort_flag)) return false;
    if (globaltimer_ns() - t0 > p.wait_limit_ns) {
      set_status(p.status, QARL_ERR_DEVICE_TIMEOUT);
      *reinterpret_cast<volatile int*>(&s->abort_flag) = 1;
      return false;
    }
  }
}
// whole warp: every lane polls, then the lanes vote (no split warp after a wait)
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const W4Params& p) {
  return __all_sync(0xFFFFFFFFu, wait_or_abort(bar, parity, s, p) ? 1 : 0) != 0;
}

// Barrier among `n` threads that also tells every one of them whether `pred` held for all.
__device__ __forceinline__ bool named_bar_all(uint32_t id, uint32_t n, bool pred) {
  __syncwarp();  // (bar.red is an aligned instruction)
  uint32_t r;
  asm volatile(
      "{\n\t"
      ".reg .pred p, q;\n\t"
      "setp.ne.b32 q, %3, 0;\n\t"
      "bar.red.and.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "}"
      : "=r"(r)
      : "r"(id), "r"(n), "r"(static_cast<uint32_t>(pred))
      : "memory");
  return r != 0;
}

__device__ __forceinline__ float silu_mul(float g, float u) { return __fdividef(g, 1.0f + __expf(-g)) * u; }

// 128-row blocks (within the expert) of a tile's two halves
template <int MODE>
__device__ __forceinline__ void tile_blocks(const W4Params& p, int j, int& nb_lo, int& nb_hi) {
  const int NB = p.N / BW;
  if (MODE == kModeGateUp) {
    nb_lo = j;
    nb_hi = j + p.I / BW;
  } else {
    nb_lo = 2 * j;
    nb_hi = min(2 * j + 1, NB - 1);  // a half past N re-reads the last block; its columns are never stored
  }
}

template <int MODE, int FMT, int NT>
__global__ void __launch_bounds__(Cfg<NT>::kThreads, 1)
gemm_w4a16_kernel(const __grid_constant__ CUtensorMap tm_x, const W4Params p) {
  using C = Cfg<NT>;
  constexpr int kXStages = C::kXStages, kQStages = C::kQStages, kAStages = C::kAStages, kAK = C::kAK, kStageCols = C::kStageCols;
  constexpr int kAccBufs = C::kAccBufs, kEpiWarps = C::kEpiWarps, kCodeWarp = C::kCodeWarp, kTokenWarp = C::kTokenWarp, kMmaWarp = C::kMmaWarp;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* x_base = smem;  // [stage][K-step][NT rows x 128 bytes], swizzled
  uint8_t* q_base = x_base + static_cast<size_t>(kXStages) * C::kXBytes;
  uint8_t* out_tile = q_base + static_cast<size_t>(kQStages) * kGroupBytes;
  SmemTail* s = reinterpret_cast<SmemTail*>(out_tile + NT * kOutRowBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // ---- set-up: barriers, TMEM, tile list ------------------------------------------------
  if (threadIdx.x == 0) {
    for (int i = 0; i < kXStages; ++i) {
      mbar_init(&s->x_full[i], 1);
      mbar_init(&s->x_empty[i], 2);                                  // the commits of the two issuers
    }
    for (int i = 0; i < kQStages; ++i) {
      mbar_init(&s->q_full[i], 2);                                   // the bulk copies, the scales
      mbar_init(&s->q_empty[i], kAK == 2 ? kDqWarps / 2 : kDqWarps);  // the warps that read it
    }
    for (int i = 0; i < kAStages; ++i) {
      mbar_init(&s->a_full[i], kDqWarps / 2);
      mbar_init(&s->a_empty[i], 2);
    }
    for (int i = 0; i < kAccBufs; ++i) {
      mbar_init(&s->tmem_full[i], 2);
      mbar_init(&s->tmem_empty[i], kEpiWarps);
    }
    mbar_init(&s->teardown[0], 1);
    mbar_init(&s->teardown[1], 1);
    s->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kTokenWarp && lane == 0) prefetch_tensormap(&tm_x);
  if (warp == kMmaWarp) {
    tmem_alloc(&s->tmem_addr, kTmemCols);
    pdl_trigger();  // not before the allocation: see pdl_trigger
    tmem_relinquish();
  }
  const int KS = p.ksteps;
  const int KG = KS / 2;             // 128-element groups along K
  const int NB = p.N / BW;
  // codes of tile (expert e, block pair j): the two blocks' chunks, each KS x 4 KB contiguous
  auto tile_codes = [&](int e, int j, const uint8_t*& q_lo, const uint8_t*& q_hi) {
    int nb_lo, nb_hi;
    tile_blocks<MODE>(p, j, nb_lo, nb_hi);
    q_lo = p.b_packed + (static_cast<int64_t>(e) * NB + nb_lo) * KS * kQStepBytes;
    q_hi = p.b_packed + (static_cast<int64_t>(e) * NB + nb_hi) * KS * kQStepBytes;
  };
  if (warp == kCodeWarp && lane == 0 && p.early_prefetch) {
    // The weights do not depend on the kernels before this one in the stream: start pulling this CTA's
    // first tile (guessed as expert T / n_pairs, pair T % n_pairs: exact when every expert has one chunk).
    const int T = blockIdx.x;
    if (T < p.E * p.n_pairs) {
      const uint8_t *q_lo, *q_hi;
      tile_codes(T / p.n_pairs, T % p.n_pairs, q_lo, q_hi);
      const uint32_t bytes = static_cast<uint32_t>(KS) * kQStepBytes;
      for (uint32_t o = 0; o < bytes; o += kPrefetchChunk) {
        bulk_prefetch_l2(q_lo + o, min(kPrefetchChunk, bytes - o));
        bulk_prefetch_l2(q_hi + o, min(kPrefetchChunk, bytes - o));
      }
    }
  }
  pdl_wait();  // nothing above read the predecessor's results
  build_tile_list(s->off, s->prefix, p.offsets, p.rows_total, p.E, NT, p.n_pairs);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = s->tmem_addr;
  const int total_tiles = s->prefix[p.E];
  const int num_ctas = gridDim.x;
  const int first_tile = blockIdx.x;

  if (warp == kTokenWarp) {
    // =============================== producer of the token rows =======================
    if (elect_one()) {
      int xs = 0, cur_e = 0, left = p.stop_after_stages;
      uint32_t x_phase = 0, armed = 0, armed_parity = 0;
      bool ok = true;
      for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
        const TileCoord c = decode_tile(s->off, s->prefix, NT, T, cur_e);
        for (int g = 0; g < KG; ++g) {
          if (left-- == 0 || !wait_or_abort(&s->x_empty[xs], x_phase ^ 1, s, p)) { ok = false; break; }
          mbar_arrive_expect_tx(&s->x_full[xs], C::kXBytes);
          uint8_t* dst = x_base + static_cast<size_t>(xs) * C::kXBytes;
          tma_load_2d(dst, &tm_x, &s->x_full[xs], 2 * g * BK, c.m0);
          tma_load_2d(dst + C::kXBytes / 2, &tm_x, &s->x_full[xs], (2 * g + 1) * BK, c.m0);
          armed |= 1u << xs;
          armed_parity = (armed_parity & ~(1u << xs)) | (x_phase << xs);
          if (++xs == kXStages) { xs = 0; x_phase ^= 1; }
        }
      }
      if (!ok) {  // let copies in flight land before the CTA's shared memory is released
        for (int i = 0; i < kXStages; ++i)
          if (armed & (1u << i)) mbar_wait_bounded(&s->x_full[i], (armed_parity >> i) & 1u, 20000000ull);
      }
    }
  } else if (warp == kCodeWarp && p.sz_bulk) {
    // =============================== producer of the codes ============================
    // Per quantization group bulk copies of the two blocks' codes (8 KB each), scales and zero points.
    if (elect_one()) {
      int qs = 0, cur_e = 0, left = p.stop_after_stages;
      uint32_t q_phase = 0, armed = 0, armed_parity = 0;
      bool ok = true;
      for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
        const TileCoord c = decode_tile(s->off, s->prefix, NT, T, cur_e);
        const uint8_t *q_lo, *q_hi;
        tile_codes(c.e, c.n_tile, q_lo, q_hi);
        int nb_lo, nb_hi;
        tile_blocks<MODE>(p, c.n_tile, nb_lo, nb_hi);
        int64_t sz = static_cast<int64_t>(c.e) * KG * p.N;
        for (int g = 0; g < KG; ++g, sz += p.N) {
          if (left-- == 0 || !wait_or_abort(&s->q_empty[qs], q_phase ^ 1, s, p)) { ok = false; break; }
          uint8_t* dst = q_base + static_cast<size_t>(qs) * kGroupBytes;
          uint64_t* bar = &s->q_full[qs];
          mbar_arrive_expect_tx(bar, FMT == kFmtInt4 ? kGroupBytes : kCodeBytes + 4 * BW);
          bulk_load_1d(dst, q_lo + static_cast<int64_t>(g) * (2 * kQStepBytes), 2 * kQStepBytes, bar);
          bulk_load_1d(dst + kCodeBytes / 2, q_hi + static_cast<int64_t>(g) * (2 * kQStepBytes), 2 * kQStepBytes, bar);
          bulk_load_1d(dst + kCodeBytes, p.b_scales + sz + nb_lo * BW, 2 * BW, bar);
          bulk_load_1d(dst + kCodeBytes + 2 * BW, p.b_scales + sz + nb_hi * BW, 2 * BW, bar);
          if constexpr (FMT == kFmtInt4) {
            bulk_load_1d(dst + kCodeBytes + 4 * BW, p.b_zeros + sz + nb_lo * BW, BW, bar);
            bulk_load_1d(dst + kCodeBytes + 5 * BW, p.b_zeros + sz + nb_hi * BW, BW, bar);
          }
          mbar_arrive(bar);  // (the slower form below arrives twice)
          armed |= 1u << qs;
          armed_parity = (armed_parity & ~(1u << qs)) | (q_phase << qs);
          if (++qs == kQStages) { qs = 0; q_phase ^= 1; }
        }
      }
      if (!ok) {
        for (int i = 0; i < kQStages; ++i)
          if (armed & (1u << i)) mbar_wait_bounded(&s->q_full[i], (armed_parity >> i) & 1u, 20000000ull);
      }
    }
  } else if (warp == kCodeWarp) {
    // The same for scales and zero points that are not 16-byte aligned (the interface promises 2 and 1): plain loads,
    // lane l rows l, l + 32, ..., written to the stage by this warp; their latency is paid per group (gate_up of 96
    // tokens 94 us instead of 70).
    int qs = 0, cur_e = 0, left = p.stop_after_stages;
    uint32_t q_phase = 0, armed = 0, armed_parity = 0;
    bool ok = true;
    for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
      const TileCoord c = decode_tile(s->off, s->prefix, NT, T, cur_e);
      const uint8_t *q_lo, *q_hi;
      tile_codes(c.e, c.n_tile, q_lo, q_hi);
      int nb_lo, nb_hi;
      tile_blocks<MODE>(p, c.n_tile, nb_lo, nb_hi);
      int64_t sz = static_cast<int64_t>(c.e) * KG * p.N + lane;
      for (int g = 0; g < KG; ++g, sz += p.N) {
        uint16_t sc[8];
        uint8_t z[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int64_t at = sz + (r < 4 ? nb_lo : nb_hi) * BW + 32 * (r & 3);
          sc[r] = __ldg(p.b_scales + at);
          if constexpr (FMT == kFmtInt4) z[r] = __ldg(p.b_zeros + at);
        }
        if (left-- == 0 || !warp_wait_or_abort(&s->q_empty[qs], q_phase ^ 1, s, p)) { ok = false; break; }
        uint8_t* dst = q_base + static_cast<size_t>(qs) * kGroupBytes;
        if (lane == 0) {
          mbar_arrive_expect_tx(&s->q_full[qs], kCodeBytes);
          bulk_load_1d(dst, q_lo + static_cast<int64_t>(g) * (2 * kQStepBytes), 2 * kQStepBytes, &s->q_full[qs]);
          bulk_load_1d(dst + kCodeBytes / 2, q_hi + static_cast<int64_t>(g) * (2 * kQStepBytes), 2 * kQStepBytes, &s->q_full[qs]);
        }
        uint16_t* sdst = reinterpret_cast<uint16_t*>(dst + kCodeBytes);
        uint8_t* zdst = dst + kCodeBytes + 2 * BW * 2;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          sdst[32 * r + lane] = sc[r];
          if constexpr (FMT == kFmtInt4) zdst[32 * r + lane] = z[r];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->q_full[qs]);
        armed |= 1u << qs;
        armed_parity = (armed_parity & ~(1u << qs)) | (q_phase << qs);
        if (++qs == kQStages) { qs = 0; q_phase ^= 1; }
      }
    }
    if (!ok && lane == 0) {
      for (int i = 0; i < kQStages; ++i)
        if (armed & (1u << i)) mbar_wait_bounded(&s->q_full[i], (armed_parity >> i) & 1u, 20000000ull);
    }
  } else if (warp >= kMmaWarp) {
    // =============================== MMA issuers ======================================
    // One thread per weight block, each with its own NT accumulator columns and its half of an A stage.
    if (elect_one()) {
      const int h = warp - kMmaWarp;
      constexpr uint32_t idesc = umma_idesc_bf16_f32(BW, NT);
      int xs = 0, as = 0, acc = 0;
      uint32_t x_phase = 0, a_phase = 0, acc_phase = 0;
      bool ok = true;
      for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
        if (!wait_or_abort(&s->tmem_empty[acc], acc_phase ^ 1, s, p)) { ok = false; break; }
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc) * (2 * NT) + static_cast<uint32_t>(h) * NT;
        for (int g = 0; ok && g < KG; ++g) {
          if (!wait_or_abort(&s->x_full[xs], x_phase, s, p)) { ok = false; break; }
          const uint32_t x_addr = smem_u32(x_base + static_cast<size_t>(xs) * C::kXBytes);
#pragma unroll
          for (int u0 = 0; u0 < 2; u0 += kAK) {
            if (!wait_or_abort(&s->a_full[as], a_phase, s, p)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t a_tmem = tmem_base + C::kABase + static_cast<uint32_t>(as * kStageCols + h * (kStageCols / 2));
#pragma unroll
            for (int u = 0; u < kAK; ++u) {
              const uint64_t x_desc = umma_desc_k_sw128(x_addr + (u0 + u) * (C::kXBytes / 2));
#pragma unroll
              for (int k4 = 0; k4 < BK / 16; ++k4)  // +16 elements: 8 TMEM columns of A, 2 in the 16-byte address field of B
                umma_bf16_ts(d_tmem, a_tmem + 32 * u + 8 * k4, x_desc + 2 * k4, idesc, (g > 0 || u0 + u > 0 || k4 > 0) ? 1u : 0u);
            }
            umma_commit(&s->a_empty[as]);
            if (++as == kAStages) { as = 0; a_phase ^= 1; }
          }
          if (!ok) break;
          umma_commit(&s->x_empty[xs]);
          if (g == KG - 1) umma_commit(&s->tmem_full[acc]);
          if (++xs == kXStages) { xs = 0; x_phase ^= 1; }
        }
        if (++acc == kAccBufs) { acc = 0; acc_phase ^= 1; }
      }
      if (!ok) {  // after an abort MMAs may still be executing: wait (bounded) before TMEM goes away
        umma_commit(&s->teardown[h]);
        mbar_wait_bounded(&s->teardown[h], 0, 20000000ull);
      }
    }
  } else if (warp >= kEpiWarps) {
    // =============================== dequantization warps =============================
    // A stage of kAK K-steps is filled by one group of eight warps; the groups take stages in turn (a tile has an
    // even number of K-steps; with kAK = 2 the turn goes on across tiles).
    const int grp = (warp - kEpiWarps) >> 3;
    const int h = ((warp - kEpiWarps) >> 2) & 1;     // weight block of the pair
    const int nr = (warp & 3) * 32 + lane;           // weight row of the block = TMEM lane
    const uint32_t a_base = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + C::kABase + static_cast<uint32_t>(h) * (kStageCols / 2);
    const int groups = first_tile < total_tiles ? ((total_tiles - 1 - first_tile) / num_ctas + 1) * KG : 0;  // of this CTA
    // this thread's codes of a group: kAK K-steps, [block][K-step][word quad 0..1][row][16 bytes] in the ring
    struct Codes {
      uint4 w[2 * kAK];
      uint32_t s, z;
    };
    auto fetch = [&](int g, Codes& c) {  // the group's stage is full; hands the stage back
      const int qs = g % kQStages;
      const uint8_t* q = q_base + static_cast<size_t>(qs) * kGroupBytes;
      const uint8_t* src = q + h * (2 * kQStepBytes) + (kAK == 2 ? 0 : grp) * kQStepBytes + nr * 16;
#pragma unroll
      for (int i = 0; i < 2 * kAK; ++i) c.w[i] = *reinterpret_cast<const uint4*>(src + i * (kQStepBytes / 2));
      c.s = *reinterpret_cast<const uint16_t*>(q + kCodeBytes + 2 * (h * BW + nr));
      if constexpr (FMT == kFmtInt4) c.z = q[kCodeBytes + 4 * BW + h * BW + nr];
      __syncwarp();
      if (lane == 0) mbar_arrive(&s->q_empty[qs]);
    };
    auto q_parity = [&](int g) { return static_cast<uint32_t>(g / kQStages) & 1u; };
    // Expands group g from `cur`; the next one's codes are fetched into `nxt` first if they are there already, so
    // that their barrier and shared-memory latency hide behind this group's arithmetic.
    auto step = [&](int g, Codes& cur, Codes& nxt) -> bool {
      const int gn = g + kAK;
      bool have_next = gn >= groups;
      if (!have_next && __all_sync(0xFFFFFFFFu, mbar_try_wait(&s->q_full[gn % kQStages], q_parity(gn)))) {
        fetch(gn, nxt);
        have_next = true;
      }
      const uint32_t n = static_cast<uint32_t>(kAK == 2 ? g : 2 * g + grp);  // A stages of this CTA before this one
      const int as = static_cast<int>(n % kAStages);
      if (!warp_wait_or_abort(&s->a_empty[as], ((n / kAStages) & 1u) ^ 1u, s, p)) return false;
      tc_fence_after_sync();
      const uint32_t dst = a_base + static_cast<uint32_t>(as) * kStageCols;
      auto expand = [&](auto sc) {
#pragma unroll
        for (int i = 0; i < 2 * kAK; ++i) {
          const uint32_t words[4] = {cur.w[i].x, cur.w[i].y, cur.w[i].z, cur.w[i].w};
          uint32_t r[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint4 v = sc.expand(words[j]);
            r[4 * j] = v.x;
            r[4 * j + 1] = v.y;
            r[4 * j + 2] = v.z;
            r[4 * j + 3] = v.w;
          }
          tmem_st_x16(dst + 16 * i, r);
        }
      };
      if constexpr (FMT == kFmtInt4) {
        expand(W4Scale<0>(cur.s, cur.z));
      } else {
        if (__all_sync(0xFFFFFFFFu, ((cur.s >> 7) & 0xFFu) <= 127u)) expand(W4Scale<2>(cur.s, 0));
        else expand(W4Scale<1>(cur.s, 0));
      }
      tmem_st_wait();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s->a_full[as]);
      if (!have_next) {
        if (!warp_wait_or_abort(&s->q_full[gn % kQStages], q_parity(gn), s, p)) return false;
        fetch(gn, nxt);
      }
      return true;
    };
    const int g0 = kAK == 2 ? grp : 0;
    Codes ca{}, cb{};
    if (g0 < groups && warp_wait_or_abort(&s->q_full[g0], 0, s, p)) {
      fetch(g0, ca);
      for (int g = g0; g < groups; g += 2 * kAK) {
        if (!step(g, ca, cb)) break;
        if (g + kAK < groups && !step(g + kAK, cb, ca)) break;
      }
    }
  } else {
    // =============================== epilogue warps ===================================
    const int wr = (warp & 3) * 32 + lane;  // weight row within a block = TMEM lane
    constexpr int kTurn = 16 * (kEpiWarps / 4);  // the warps of a quadrant take 16 token columns in turn
    const int tc0 = (warp >> 2) * 16;
    constexpr uint32_t kEpiThreads = kEpiWarps * 32;
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    int acc = 0, cur_e = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    uint16_t* T16 = reinterpret_cast<uint16_t*>(out_tile);
    uint32_t par = 0;
    for (int T = first_tile; T < total_tiles; T += num_ctas, par ^= 1) {
      const TileCoord c = decode_tile(s->off, s->prefix, NT, T, cur_e);
      const int rows = min(NT, c.m_end - c.m0);  // live token rows of this tile (>= 1)
      const int j = c.n_tile;
      // The pair weights come in while the tile is still being multiplied: loaded where they are used, with the
      // accumulators waiting, they cost more than the MMAs of a short contraction (I = 256, 65536 pairs of 512 experts:
      // down 167 us against 145).  (The barrier below is between this and their use, and two tiles share no slot.)
      if (MODE == kModeDown && threadIdx.x < NT)
        s->weight[par][threadIdx.x] = __ldg(p.pair_weights + min(c.m0 + static_cast<int>(threadIdx.x), p.rows_total - 1));
      ok = warp_wait_or_abort(&s->tmem_full[acc], acc_phase, s, p);
      ok = named_bar_all(1, kEpiThreads, ok);  // one decision for the eight warps; the previous tile's row readers are done
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t t0 = tmem_base + lane_addr + static_cast<uint32_t>(acc) * (2 * NT);
      const int col_lo = 2 * j * BW + wr, col_hi = col_lo + BW;  // down / linear: this thread's two output columns
      const bool hi_ok = col_hi < p.N;
      auto hand_back = [&]() {  // this warp's share of the accumulator is in registers
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->tmem_empty[acc]);
      };
      if (tc0 >= rows) hand_back();
      // 16 token columns at a time (the register budget of the CTA), the live ones only
#pragma unroll 1
      for (int tc = tc0; tc < rows; tc += kTurn) {
        uint32_t vl[16], vh[16];
        tmem_ld_x16(t0 + tc, vl);
        tmem_ld_x16(t0 + NT + tc, vh);
        tmem_ld_wait();
        if (tc + kTurn >= rows) hand_back();
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int t = tc + u;
          if (MODE == kModeGateUp) {
            // h = bf16( silu(bf16 gate) * bf16 up ), this thread's column of the tile's 128 h columns
            const uint32_t gb = f32_to_bf16_bits(__uint_as_float(vl[u])), ub = f32_to_bf16_bits(__uint_as_float(vh[u]));
            const uint32_t hb = f32_to_bf16_bits(silu_mul(bf16_bits_to_f32(gb), bf16_bits_to_f32(ub)));
            T16[t * (kOutRowBytes / 2) + wr] = static_cast<uint16_t>(hb);
            if (p.out_bf16 && t < rows) {  // debug dump of the bf16 gate_up row
              uint16_t* gd = p.out_bf16 + static_cast<int64_t>(c.m0 + t) * p.N + j * BW + wr;
              gd[0] = static_cast<uint16_t>(gb);
              gd[p.I] = static_cast<uint16_t>(ub);
            }
          } else {
            float lo = __uint_as_float(vl[u]), hi = __uint_as_float(vh[u]);
            if (p.out_f32 && t < rows) {  // fp32 accumulator dump (down: in sorted order)
              float* d = p.out_f32 + static_cast<int64_t>(c.m0 + t) * p.N;
              d[col_lo] = lo;
              if (hi_ok) d[col_hi] = hi;
            }
            if (MODE == kModeDown) {  // contribution = bf16( fl(w * y) )
              const float w = s->weight[par][t];
              lo = __fmul_rn(w, lo);
              hi = __fmul_rn(w, hi);
            }
            T16[t * (kOutRowBytes / 2) + wr] = static_cast<uint16_t>(f32_to_bf16_bits(lo));
            T16[t * (kOutRowBytes / 2) + BW + wr] = static_cast<uint16_t>(f32_to_bf16_bits(hi));
          }
        }
      }
      if (++acc == kAccBufs) { acc = 0; acc_phase ^= 1; }

      if (MODE == kModeGateUp) {
        named_bar_sync(2, kEpiThreads);
        for (int t = warp; t < rows; t += kEpiWarps) {  // a warp per token row: 256 bytes, 8 per lane
          const uint2 hv = *reinterpret_cast<const uint2*>(out_tile + t * kOutRowBytes + lane * 8);
          *reinterpret_cast<uint2*>(p.h_bf16 + static_cast<int64_t>(c.m0 + t) * p.I + j * BW + lane * 4) = hv;
        }
      } else {
        named_bar_sync(2, kEpiThreads);
        if (p.out_bf16) {
          for (int t = warp; t < rows; t += kEpiWarps) {  // a warp per output row: 512 bytes, 16 per lane
            const int row = c.m0 + t;
            const uint4 v = *reinterpret_cast<const uint4*>(out_tile + t * kOutRowBytes + lane * 16);
            const int col = 2 * j * BW + 8 * lane;
            if (col < p.N) *reinterpret_cast<uint4*>(p.out_bf16 + static_cast<int64_t>(row) * p.N + col) = v;
          }
        }
      }
    }
  }

  // ---- teardown ---------------------------------------------------------------------------
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

CUresult make_tmap_x(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t K, uint32_t box_rows) {
  // bf16 tensor [rows, K] row-major; box = 64 elements (128 bytes) x box_rows rows, 128-byte swizzle.
  const cuuint64_t dims[2] = {K, rows};
  const cuuint64_t strides[1] = {K * 2};
  const cuuint32_t box[2] = {BK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int MODE, int FMT, int NT>
cudaError_t launch_size(const Launch& L, const CUtensorMap& tx, const W4Params& p) {
  static std::atomic<bool> attr_set_dev[64];  // sticky per function and device; set idempotently
  std::atomic<bool>& attr_set = attr_set_dev[L.device & 63];
  if (!attr_set.load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_w4a16_kernel<MODE, FMT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kSmemBytes<NT>));
    if (e != cudaSuccess) return e;
    attr_set.store(true, std::memory_order_release);
  }
  // upper bound on the tile count (group sizes live on the device): each expert adds at most one partial chunk
  const int64_t chunks_max = p.rows_total / NT + p.E;
  const int grid = static_cast<int>(std::min<int64_t>(L.sm_count, chunks_max * p.n_pairs));
  ++*L.launches;
  return launch_pdl(gemm_w4a16_kernel<MODE, FMT, NT>, static_cast<unsigned>(grid), Cfg<NT>::kThreads, kSmemBytes<NT>, L.stream, tx, p);
}

template <int MODE>
cudaError_t launch_mode(const Launch& L, const CUtensorMap& tx, const W4Params& p, int fmt, int nt) {
  if (fmt == kFmtE2m1)
    return nt == kNarrow ? launch_size<MODE, kFmtE2m1, kNarrow>(L, tx, p)
         : nt == kMid    ? launch_size<MODE, kFmtE2m1, kMid>(L, tx, p)
                         : launch_size<MODE, kFmtE2m1, kWide>(L, tx, p);
  return nt == kNarrow ? launch_size<MODE, kFmtInt4, kNarrow>(L, tx, p)
       : nt == kMid    ? launch_size<MODE, kFmtInt4, kMid>(L, tx, p)
                       : launch_size<MODE, kFmtInt4, kWide>(L, tx, p);
}

}  // namespace

cudaError_t launch_gemm_w4a16(const Launch& L, EncodeTiledFn encode, const GemmW4Args& a, CUresult* cu_err) {
  *cu_err = CUDA_SUCCESS;
  if (a.rows_total == 0) return cudaSuccess;
  // Rows per tile by the average group: 32 up to 24 rows (a wider tile would multiply padding; groups scatter around
  // the average, and at 32 rows half of them already need a second 32-row tile: 512 tokens, top-8 of 128, 165 us against
  // 149 with 64-row tiles), 64 up to 56 rows (1024 tokens: equal), 128 beyond (2048 tokens: 279 us against 299: an
  // expansion serves more rows).
  const int nt = L.gemm_path == 1 ? kWide : L.gemm_path == 2 || a.rows_total <= 24 * a.E ? kNarrow : a.rows_total <= 56 * a.E ? kMid : kWide;
  CUtensorMap tx;
  const CUresult r = make_tmap_x(encode, &tx, a.a_bf16, static_cast<uint64_t>(a.rows_total), static_cast<uint64_t>(a.K),
                                 static_cast<uint32_t>(nt));
  if (r != CUDA_SUCCESS) {
    *cu_err = r;
    return cudaErrorUnknown;
  }
  W4Params p{};
  p.b_packed = a.b_packed;
  p.b_scales = a.b_scales;
  p.b_zeros = a.b_zeros;
  p.offsets = a.offsets;
  p.rows_total = static_cast<int>(a.rows_total);
  p.ksteps = static_cast<int>(a.K / BK);
  p.N = static_cast<int>(a.N);
  p.E = static_cast<int>(a.E);
  p.I = static_cast<int>(a.N / 2);
  p.n_pairs = a.mode == kModeGateUp ? static_cast<int>(a.N / 2 / BW) : static_cast<int>((a.N + 2 * BW - 1) / (2 * BW));
  p.early_prefetch = 2 * a.rows_total >= a.E;  // below, most experts have no rows and the guess is wrong
  p.sz_bulk = ((reinterpret_cast<uintptr_t>(a.b_scales) | reinterpret_cast<uintptr_t>(a.b_zeros)) & 15u) == 0;
  p.out_bf16 = a.out_bf16;
  p.out_f32 = a.out_f32;
  p.h_bf16 = a.h_bf16;
  p.pair_weights = a.pair_weights;
  p.status = L.d_status;
  p.wait_limit_ns = L.wait_limit_ns ? L.wait_limit_ns : 2000000000ull;
  p.stop_after_stages = L.stop_after_stages;
  switch (a.mode) {
    case kModeLinear: return launch_mode<kModeLinear>(L, tx, p, a.fmt, nt);
    case kModeGateUp: return launch_mode<kModeGateUp>(L, tx, p, a.fmt, nt);
    case kModeDown: return launch_mode<kModeDown>(L, tx, p, a.fmt, nt);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qarl
