// Persistent block-scaled FP8 GEMM for sm_100a (dense projection, MoE gate_up, MoE down).
//
// Computes, for every output row m (an activation row) and column n (a weight row),
//   acc[m,n] = sum over kb ascending, from 0.0f, of  fmaf( fl(s_x[m,kb] * s_w[n/128,kb]), p_kb[m,n], acc )
// where p_kb is the tensor-core dot product of the 128 e4m3 codes of K-block kb (Sec. 2.2:
// Y ~= (s_x s_w)(X_q W_q), applied per block with fp32 accumulation).  The order is the same
// for every M, group size, tile width and schedule (App. C): 128-row MMAs of K = 32 (a column's sum does not
// depend on how many columns the MMA has), four per K-block in ascending k, no split-K, no atomics.  A row's
// result depends only on that row's codes and scales and on the weight tile.
//
// A tile is 128 rows x (128 + 128) columns: two half tiles, rows [n_lo, n_lo+128) and
// [n_hi, n_hi+128) of the weight -- adjacent for linear/down, gate rows and the matching up
// rows for gate_up so that SwiGLU and the 1x128 re-quantization of h need no second pass.  Dense calls too
// small for that take tiles of 128 or 64 columns (COLS, see the host).
//
// Structure of a CTA (384 threads = 3 warpgroups, one CTA per SM, persistent, static tile list):
//   warp 8      TMA producer: per K-block one stage = A box 128x128 B + two B boxes 128x128 B
//               (SWIZZLE_128B) into a ring of 48 KB stages;
//   warp 9      MMA issuer: 4 x tcgen05.mma kind::f8f6f4 per K-block into one of two
//               256-column TMEM accumulators (overwrite on the first), then tcgen05.commit to
//               free the smem stage and to publish the accumulator;
//   warps 10-11 scales: fl(s_x s_w) of every row and half for the K-block in each accumulator;
//   warps 0-7   promotion (216 registers each via setmaxnreg): warp w reads TMEM lanes
//               32*(w%4).. (its hardware quadrant) and the 64-column slice (w/4) of each half,
//               releases the accumulator, and adds scale * partial into fp32 registers; the
//               MMA of block kb+1 overlaps the promotion of kb.  At the end of a tile it finishes
//               its 128 values itself: gate_up = SwiGLU, 1x128 amax / scale / e4m3 codes from registers;
//               linear, down = bf16 rows through a swizzled staging box and a TMA store.
//
// What bounds it: the promotion next to the MMA, and close to it the 48 KB per K-block that come into the SM (MMAs and loads
// alone ~800 clocks).  Per K-block the promotion reads 128 KB of TMEM and does 32768 FMAs (256 clocks of the FP32 pipes; alone it
// measures 573) against 512 clocks of MMAs, so what it must not do is wait or spill.  With scale loads, waits and separate
// epilogue warps inline a K-block took ~1210 clocks; as below 870 to 890, 935 with the tile ends of K = 2048 (dense M = 8192,
// N = 5120, K = 2048: 92 us in short runs).  What did it: scales from two warps of their own through shared memory, one stream
// of TMEM reads across K-blocks (the first chunk of the next accumulator is on its way before the last chunk
// of this one is accumulated), two FMAs per instruction, the loop body without spills (32-column chunks
// spill and lose), and no epilogue warps (their registers and polling cost more than they hid).
//
// Every wait on an mbarrier is bounded; on expiry the thread records
// QARL_ERR_DEVICE_TIMEOUT, raises a CTA-wide abort flag that all other waits poll, and the
// CTA drains and frees its TMEM, so a broken pipeline returns an error instead of hanging.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "quant_device.cuh"

namespace qarl {
namespace {

using namespace ptx;

constexpr int BM = 128;           // rows per tile (UMMA M)
constexpr int BNH = 128;          // columns per half tile
constexpr int BN = 2 * BNH;       // UMMA N
constexpr int BK = 128;           // one K-block = one 128-byte swizzle span of e4m3
constexpr int kMaxAccBufs = 4;
constexpr int kMaxStages = 16;
constexpr int kPromoWarps = 8;    // warps 0-7
constexpr int kTmaWarp = 8;
constexpr int kMmaWarp = 9;
constexpr int kScaleWarp = 10;    // and 11
constexpr int kThreads = 12 * 32;
// register re-allocation: 256 x 216 + 128 x 72 = 64512 = 384 x 168 (the launch allocation)
constexpr int kPromoRegs = 216;
constexpr int kAuxRegs = 72;
constexpr uint32_t kABytes = BM * BK;
constexpr uint32_t kBHalfBytes = BNH * BK;
constexpr uint32_t kTmemCols = 512;
// a promotion warp's bf16 rows on their way out: a box of 32 rows x 128 bytes (128-byte swizzle) per half
constexpr uint32_t kOutBoxBytes = 32 * 128;
constexpr int kMaxExperts = 1024;

struct GemmParams {
  const float* a_scales;
  const float* b_scales;
  const int32_t* offsets;  // [E+1] or nullptr (dense: one group of rows_total rows)
  int rows_total;
  int kblocks;             // K / 128
  int N;                   // weight rows per expert
  int E;
  int n_tiles;             // column tiles per expert
  int I;                   // gate_up: intermediate size (N = 2I)
  int a_rows, stages;      // COLS = 64: rows of the token box, stages of a_rows x 128 + 8192 bytes
  int weights_once;        // few row tiles per expert: weights are loaded with the evict-first policy
  const uint16_t* x;       // FUSED: the bf16 rows
  int early_prefetch;      // decode-sized calls: weight tiles to pull into L2 before the predecessor finishes
  uint16_t* out_bf16;
  float* out_f32;
  uint8_t* h_codes;
  float* h_scales;
  uint16_t* h_bf16;
  int h_vec32;             // h_bf16 is 32-byte aligned
  const float* pair_weights;  // down: combine weight of each sorted position
  int* status;
  unsigned long long wait_limit_ns;
  int stop_after_stages;   // test harness only (< 0: off): the TMA producer stops arming stages after this many
};

// SAVE (gate_up only): the call also wants the bf16 gate_up and / or h rows (a training forward, tests)
// COLS: columns of a tile, 256 (two halves); 128 and 64 are for dense calls that do not fill the SMs with 256
template <int MODE, bool SAVE, int COLS>
struct Cfg {
  static constexpr bool kStaged = MODE != kModeGateUp || SAVE;  // rows leave through the staging boxes
  static constexpr int kHalves = COLS == 256 ? 2 : 1;
  static constexpr int kSlice = COLS / kHalves / 2;             // columns of each half owned by one promotion warp
  // ring: fixed 48 or 32 KB stages; with 64 columns as many as fit (a decode call's token box is a few rows, see the host)
  static constexpr int kStages = COLS == 64 ? 0 : COLS == 128 ? 5 : kStaged ? 3 : 4;
  static constexpr uint32_t kStageBytes = kABytes + COLS * BK;
  static constexpr uint32_t kStaging = kStaged && COLS > 64 ? kPromoWarps * kHalves * kOutBoxBytes : 0;
  static constexpr int kAccBufs = COLS == 256 ? 2 : 4;
};

struct __align__(16) SmemTail {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t tmem_full[kMaxAccBufs];
  uint64_t tmem_empty[kMaxAccBufs];
  uint64_t amax_full[4];       // gate_up: the two warps of a TMEM quadrant have exchanged their row maxima
  uint64_t teardown;
  uint64_t x_ready;            // FUSED: the rows are quantized
  float2 scale[kMaxAccBufs][BM];  // products of the K-block in each accumulator: row scale x (lo, hi) weight scale
  uint32_t amax[2][2][BM];     // gate_up: [tile parity][column slice][row] |h| maxima (bf16 bits)
  // Grouped forms: what the promotion warps need to know about a tile, published by the scale warps with its first K-block
  // (they may be kMaxAccBufs tiles of one K-block ahead, hence twice as many slots).
  int4 tile[2 * kMaxAccBufs];  // first row, end of the group's rows, column tile
  float pair_w[4][BM];         // down (two accumulators): combine weight of every row
  uint32_t tmem_addr;
  int abort_flag;
  int32_t off[kMaxExperts + 1];
  int32_t prefix[kMaxExperts + 1];
};

template <int MODE, bool SAVE, int COLS>
constexpr size_t kSmemBytes = 1024 + static_cast<size_t>(Cfg<MODE, SAVE, COLS>::kStages) * Cfg<MODE, SAVE, COLS>::kStageBytes +
                              Cfg<MODE, SAVE, COLS>::kStaging + sizeof(SmemTail);
constexpr size_t kSmemLimit = 227 * 1024;
static_assert(kSmemBytes<kModeGateUp, false, 256> <= kSmemLimit && kSmemBytes<kModeGateUp, true, 256> <= kSmemLimit &&
                  kSmemBytes<kModeLinear, false, 128> <= kSmemLimit,
              "shared memory budget");

struct TileCoord {
  int e, n_tile, m0, m_end;
};

// Tile T -> (expert, column tile, first row, end of the expert's rows).  Within an expert the
// row tiles vary fastest, so CTAs running at the same time share one weight tile through L2.
__device__ __forceinline__ TileCoord decode_tile(const SmemTail* s, int T, int& cur_e) {
  while (T >= s->prefix[cur_e + 1]) ++cur_e;
  const int local = T - s->prefix[cur_e];
  const int rows = s->off[cur_e + 1] - s->off[cur_e];
  const int m_tiles = (rows + BM - 1) / BM;
  TileCoord c;
  c.e = cur_e;
  c.n_tile = local / m_tiles;
  c.m0 = s->off[cur_e] + (local % m_tiles) * BM;
  c.m_end = s->off[cur_e + 1];
  return c;
}

// Bounded wait of one thread.  False: the limit ran out here (the error is recorded and the
// CTA-wide abort flag raised) or another thread raised the flag; the caller leaves its loop.
__device__ __forceinline__ bool wait_or_abort_at(uint32_t bar, uint32_t parity, SmemTail* s, const GemmParams& p) {
  if (mbar_try_wait_at(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 128; ++i)
      if (mbar_try_wait_at(bar, parity)) return true;
    if (*reinterpret_cast<volatile int*>(&s->abort_flag)) return false;
    if (globaltimer_ns() - t0 > p.wait_limit_ns) {
      set_status(p.status, QARL_ERR_DEVICE_TIMEOUT);
      *reinterpret_cast<volatile int*>(&s->abort_flag) = 1;
      return false;
    }
  }
}
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const GemmParams& p) {
  return wait_or_abort_at(smem_u32(bar), parity, s, p);
}

// The same for a whole warp: every lane polls (one polling lane with 31 parked at a shuffle
// measured 2x slower on the short-K down projection), then the lanes vote, so all 32 take the
// same branch and the warp-wide shuffles and barriers that follow never see a split warp
// (lanes polling on their own could disagree when a barrier completes right at the limit).
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const GemmParams& p) {
  return __all_sync(0xFFFFFFFFu, wait_or_abort(bar, parity, s, p) ? 1 : 0) != 0;
}

// silu(g) * u in fp32 with the fast exp and reciprocal (relative error ~1e-6, far below the
// half-ulp of the bf16 the result is rounded to).
__device__ __forceinline__ float silu_mul(float g, float u) {
  return __fdividef(g, 1.0f + __expf(-g)) * u;
}

// acc[j] = fmaf(sc, v[j], acc[j]) for 16 values (8 float2 accumulators), two per instruction.
__device__ __forceinline__ void promote16(float2* acc, const uint32_t (&v)[16], float sc) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    acc[j] = __ffma2_rn(make_float2(sc, sc), make_float2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), acc[j]);
}

__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);  // .x = lo (low 16 bits), .y = hi
  return *reinterpret_cast<const uint32_t*>(&b);
}

// 32 bytes to global memory, 32-byte aligned
__device__ __forceinline__ void st_global_v8(void* dst, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// the same for a pointer that is only 16-byte aligned (caller-owned dumps)
__device__ __forceinline__ void st_global_2x16(void* dst, const uint32_t (&v)[8]) {
  uint4* d = static_cast<uint4*>(dst);
  d[0] = make_uint4(v[0], v[1], v[2], v[3]);
  d[1] = make_uint4(v[4], v[5], v[6], v[7]);
}

// The promotion warps (see the header).  What they need is read again here instead of being carried over from
// the kernel's set-up: with 160 registers of sums and partial sums every long-lived value counts.
template <int MODE, bool SAVE, int COLS>
__device__ __forceinline__ void promotion_role(const CUtensorMap& tm_o, const GemmParams& p, uint8_t* smem, SmemTail* s,
                                               const int first_tile, const int num_ctas, const int total_tiles) {
  using C = Cfg<MODE, SAVE, COLS>;
  constexpr int kAccBufs = C::kAccBufs, HALVES = C::kHalves, kSliceCols = C::kSlice;
  constexpr int kPerHalf = kSliceCols / 16, kChunks = kPerHalf * HALVES;  // 16-column chunks of this warp's slices
  uint32_t tid;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  const int warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3;          // TMEM lane quadrant this warp may read
  const int hs = warp >> 2;        // which 64-column slice of each half tile
  const int r = q * 32 + lane;     // row within the tile
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&s->tmem_addr) + (static_cast<uint32_t>(q * 32) << 16) +
                        static_cast<uint32_t>(hs * kSliceCols);
  const uint32_t full_bar = smem_u32(&s->tmem_full[0]), empty_bar = smem_u32(&s->tmem_empty[0]);
  const uint32_t scale_at = smem_u32(&s->scale[0][r]);
  const int KB = p.kblocks;
  int ks = 0;
  uint32_t acc_phase = 0;
  int cur_e = 0;
  uint32_t tile_iter = 0;

  auto full_wait = [&]() -> bool { return __all_sync(0xFFFFFFFFu, wait_or_abort_at(full_bar + 8 * ks, acc_phase, s, p)) != 0; };
  auto release = [&]() {  // this warp's reads of accumulator ks are done: hand it back to the MMA warp
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive_at(empty_bar + 8 * ks);
    if (++ks == kAccBufs) { ks = 0; acc_phase ^= 1; }
  };

  // bf16 rows leave through this warp's two boxes: 64 columns each, 16-byte chunk j of a row at j ^ (row % 8)
  uint8_t* boxes = smem + static_cast<size_t>(C::kStages) * C::kStageBytes + static_cast<size_t>(warp) * HALVES * kOutBoxBytes;
  auto box_chunk = [&](int box, int j) { return reinterpret_cast<uint4*>(boxes + box * kOutBoxBytes + lane * 128 + ((j ^ (lane & 7)) << 4)); };
  auto boxes_free = [&]() {  // the previous tile's boxes have been read
    if (lane == 0) bulk_wait_group_read_all();
    __syncwarp();
  };
  auto send_boxes = [&](int row0, int m_end, int col0, int col1) {
    if (MODE == kModeLinear || row0 + 32 <= m_end) {  // (a dense tile's rows past M are clipped by the tensor map)
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d(&tm_o, boxes, col0, row0);
        if (HALVES == 2 && col1 < p.N) tma_store_2d(&tm_o, boxes + kOutBoxBytes, col1, row0);
        bulk_commit_group();
      }
    } else {  // the rows past the group's end are the next expert's: 8 lanes per row and box, 2 rows at a time
      __syncwarp();
      const int box = (lane >> 3) & 1, chunk = lane & 7;
      const int col = (box ? col1 : col0) + 8 * chunk;
      for (int rr = lane >> 4; row0 + rr < m_end; rr += 2) {
        const uint4 v = *reinterpret_cast<const uint4*>(boxes + box * kOutBoxBytes + rr * 128 + ((chunk ^ (rr & 7)) << 4));
        if (col < p.N) *reinterpret_cast<uint4*>(p.out_bf16 + static_cast<int64_t>(row0 + rr) * p.N + col) = v;
      }
      __syncwarp();
    }
  };

  for (int T = first_tile; T < total_tiles; T += num_ctas, ++tile_iter) {
    // Grouped: looking the tile up and loading the combine weights here would keep the accumulators waiting at every tile's
    // start and end (1501 tokens, 128 experts: gate_up 88 -> 84 us, down 57 -> 51); a dense call's single group is
    // looked up faster than the scale warps publish it (M = 777, N = 2048, K = 4096: 17.0 against 17.5).
    TileCoord c;
    if constexpr (MODE == kModeLinear) {
      c = decode_tile(s, T, cur_e);
      if (!full_wait()) return;
    } else {
      if (!full_wait()) return;
      const int4 at = s->tile[tile_iter & (2 * kMaxAccBufs - 1)];
      c = TileCoord{0, at.z, at.x, at.y};
    }
    // a warp whose 32 rows all lie past the group's end (ragged tails, decode-sized groups)
    // keeps the barrier protocol going but reads and accumulates nothing
    const bool warp_live = c.m0 + q * 32 < c.m_end;
    float2 acc[8 * kChunks];  // columns of the low half, then of the high half
#pragma unroll
    for (int j = 0; j < 8 * kChunks; ++j) acc[j] = make_float2(0.0f, 0.0f);
    float2* const acc_lo = acc;
    float2* const acc_hi = acc + (HALVES == 2 ? 32 : 0);

    if (!warp_live) {
      for (int kb = 0;;) {
        release();
        if (++kb == KB) break;
        if (!full_wait()) return;
      }
    } else {
      // The 16-column chunks of the accumulators are one stream across the K-blocks of the tile: while a
      // chunk is accumulated the next one is on its way from TMEM, and behind the last chunk of a K-block
      // that is the first one of the next (whose barrier was polled a chunk earlier).
      uint32_t va[16], vb[16];
      float2 scale;
      auto read_scale = [&]() {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(scale.x), "=f"(scale.y)
                     : "r"(scale_at + static_cast<uint32_t>(ks) * static_cast<uint32_t>(sizeof(s->scale[0]))) : "memory");
      };
      auto chunk_at = [&](uint32_t t0, int c) { return t0 + (c / kPerHalf) * BNH + 16 * (c % kPerHalf); };
      auto add = [&](int c, const uint32_t (&v)[16]) { promote16(acc + 8 * c, v, c < kPerHalf ? scale.x : scale.y); };
      auto all_but_last = [&]() {  // every chunk of accumulator ks but the last two sums; on return the last is in flight
        const uint32_t t0 = tmem + static_cast<uint32_t>(ks * COLS);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < kChunks - 2; c += 2) {
          tmem_ld_x16(chunk_at(t0, c + 1), vb);
          add(c, va);
          tmem_ld_wait();
          tmem_ld_x16(chunk_at(t0, c + 2), va);
          add(c + 1, vb);
          tmem_ld_wait();
        }
        tmem_ld_x16(chunk_at(t0, kChunks - 1), vb);
      };
      tc_fence_after_sync();
      tmem_ld_x16(tmem + static_cast<uint32_t>(ks * COLS), va);
      read_scale();
#pragma unroll 1
      for (int kb = 1; kb < KB; ++kb) {
        all_but_last();
        // the next accumulator's barrier: the answer is needed one chunk later
        const int kn = ks + 1 == kAccBufs ? 0 : ks + 1;
        const bool next_ready = mbar_try_wait_at(full_bar + 8 * kn, kn == 0 ? acc_phase ^ 1u : acc_phase);
        add(kChunks - 2, va);
        tmem_ld_wait();
        const float last_scale = HALVES == 2 ? scale.y : scale.x;
        release();
        if (!__all_sync(0xFFFFFFFFu, next_ready) && !full_wait()) return;
        tc_fence_after_sync();
        tmem_ld_x16(tmem + static_cast<uint32_t>(ks * COLS), va);
        promote16(acc + 8 * (kChunks - 1), vb, last_scale);
        read_scale();
      }
      all_but_last();
      add(kChunks - 2, va);
      tmem_ld_wait();
      release();
      add(kChunks - 1, vb);
    }

    // ---- the tile is complete: finish it ------------------------------------------------
    const int row = c.m0 + r;
    const bool valid = row < c.m_end;
    if ((MODE == kModeLinear || MODE == kModeDown) && p.out_f32 && valid) {  // debug fp32 dump
      const int col_lo = c.n_tile * COLS + hs * kSliceCols;
      const int col_hi = col_lo + BNH;
      float2* d_lo = reinterpret_cast<float2*>(p.out_f32 + static_cast<int64_t>(row) * p.N + col_lo);
      float2* d_hi = reinterpret_cast<float2*>(p.out_f32 + static_cast<int64_t>(row) * p.N + col_hi);
#pragma unroll
      for (int j = 0; j < kSliceCols / 2; ++j) {
        d_lo[j] = acc_lo[j];
        if (HALVES == 2 && col_hi < p.N) d_hi[j] = acc_hi[j];
      }
    }
    if (MODE == kModeDown) {  // contribution = bf16( fl(w * y) )
      const float w = s->pair_w[tile_iter & 3][r];
      const float2 w2 = make_float2(w, w);
#pragma unroll
      for (int j = 0; j < kSliceCols / 2; ++j) {
        acc_lo[j] = __fmul2_rn(w2, acc_lo[j]);
        if (HALVES == 2) acc_hi[j] = __fmul2_rn(w2, acc_hi[j]);
      }
    }
    if constexpr (MODE == kModeGateUp) {
      // This thread holds gate columns [64 hs, 64 hs + 64) of its row in acc_lo and the up columns of the
      // same h columns in acc_hi.  h = bf16(silu(bf16 gate) * bf16 up); the other warp of the quadrant
      // (w ^ 4) holds the rest of the row's 128-wide quantization group: only the maxima are exchanged.
      uint32_t hb[32];
      uint32_t m = 0;
      const int64_t col = c.n_tile * BNH + hs * kSliceCols;
      if (warp_live) {
        if (SAVE && p.out_bf16) boxes_free();
#pragma unroll
        for (int j8 = 0; j8 < 4; ++j8) {  // 16 columns at a time
          uint32_t gw[8], uw[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            gw[j] = bf16x2_bits(acc_lo[8 * j8 + j].x, acc_lo[8 * j8 + j].y);
            uw[j] = bf16x2_bits(acc_hi[8 * j8 + j].x, acc_hi[8 * j8 + j].y);
            const float h0 = silu_mul(bf16_bits_to_f32(gw[j] & 0xFFFFu), bf16_bits_to_f32(uw[j] & 0xFFFFu));
            const float h1 = silu_mul(__uint_as_float(gw[j] & 0xFFFF0000u), __uint_as_float(uw[j] & 0xFFFF0000u));
            hb[8 * j8 + j] = bf16x2_bits(h0, h1);
            m = __vmaxu2(m, hb[8 * j8 + j] & 0x7FFF7FFFu);  // |bf16| bit patterns: exact, order-free max
          }
          if (SAVE && p.out_bf16) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              *box_chunk(0, 2 * j8 + k) = make_uint4(gw[4 * k], gw[4 * k + 1], gw[4 * k + 2], gw[4 * k + 3]);
              *box_chunk(1, 2 * j8 + k) = make_uint4(uw[4 * k], uw[4 * k + 1], uw[4 * k + 2], uw[4 * k + 3]);
            }
          }
        }
        if (SAVE && p.out_bf16) send_boxes(c.m0 + q * 32, c.m_end, static_cast<int>(col), static_cast<int>(col) + p.I);
      }
      m = max(m & 0xFFFFu, m >> 16);
      const uint32_t par = tile_iter & 1u;
      s->amax[par][hs][r] = m;
      __syncwarp();
      if (lane == 0) mbar_arrive(&s->amax_full[q]);
      if (!warp_wait_or_abort(&s->amax_full[q], par, s, p)) return;
      m = max(m, s->amax[par][hs ^ 1][r]);
      float inv;
      const float sc = block_scale(bf16_bits_to_f32(m), &inv);
      if (valid) {
        uint8_t* hc = p.h_codes + static_cast<int64_t>(row) * p.I + col;
#pragma unroll
        for (int j8 = 0; j8 < 2; ++j8) {
          uint32_t cw[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t x0 = hb[16 * j8 + 2 * j], x1 = hb[16 * j8 + 2 * j + 1];
            cw[j] = cvt_e4m3x4(__fmul_rn(bf16_bits_to_f32(x0 & 0xFFFFu), inv), __fmul_rn(__uint_as_float(x0 & 0xFFFF0000u), inv),
                               __fmul_rn(bf16_bits_to_f32(x1 & 0xFFFFu), inv), __fmul_rn(__uint_as_float(x1 & 0xFFFF0000u), inv));
          }
          st_global_v8(hc + 32 * j8, cw);
        }
        if (hs == 0) p.h_scales[static_cast<int64_t>(row) * (p.I / BNH) + c.n_tile] = sc;
        if (SAVE && p.h_bf16) {
          uint16_t* hd = p.h_bf16 + static_cast<int64_t>(row) * p.I + col;
#pragma unroll
          for (int j8 = 0; j8 < 4; ++j8) {
            uint32_t w8[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) w8[j] = hb[8 * j8 + j];
            if (p.h_vec32) st_global_v8(hd + 16 * j8, w8);
            else st_global_2x16(hd + 16 * j8, w8);
          }
        }
      }
    } else if constexpr (COLS == 64) {  // a few rows: 64 bytes of each straight from the registers
      if (valid) {
        uint4* d = reinterpret_cast<uint4*>(p.out_bf16 + static_cast<int64_t>(row) * p.N + c.n_tile * COLS + hs * kSliceCols);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          d[j] = make_uint4(bf16x2_bits(acc_lo[4 * j].x, acc_lo[4 * j].y), bf16x2_bits(acc_lo[4 * j + 1].x, acc_lo[4 * j + 1].y),
                            bf16x2_bits(acc_lo[4 * j + 2].x, acc_lo[4 * j + 2].y), bf16x2_bits(acc_lo[4 * j + 3].x, acc_lo[4 * j + 3].y));
      }
    } else if (warp_live) {
      boxes_free();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        *box_chunk(0, j) =
            make_uint4(bf16x2_bits(acc_lo[4 * j].x, acc_lo[4 * j].y), bf16x2_bits(acc_lo[4 * j + 1].x, acc_lo[4 * j + 1].y),
                       bf16x2_bits(acc_lo[4 * j + 2].x, acc_lo[4 * j + 2].y), bf16x2_bits(acc_lo[4 * j + 3].x, acc_lo[4 * j + 3].y));
        if (HALVES == 2)
          *box_chunk(1, j) =
              make_uint4(bf16x2_bits(acc_hi[4 * j].x, acc_hi[4 * j].y), bf16x2_bits(acc_hi[4 * j + 1].x, acc_hi[4 * j + 1].y),
                         bf16x2_bits(acc_hi[4 * j + 2].x, acc_hi[4 * j + 2].y), bf16x2_bits(acc_hi[4 * j + 3].x, acc_hi[4 * j + 3].y));
      }
      const int col_lo = c.n_tile * COLS + hs * kSliceCols;
      send_boxes(c.m0 + q * 32, c.m_end, col_lo, col_lo + BNH);
    }
  }
  if (C::kStaging > 0 && lane == 0) bulk_wait_group_all();  // this warp's rows are written
}

// FUSED (COLS = 64): the 128-element groups of the call's few bf16 rows are quantized by the promotion warps, 8 threads
// per group, into the operand layout (row r of K-block kb at kb * 1024 + r * 128, 128-byte swizzle) and their
// scales next to it, while the first weight stages are in flight.
constexpr int kFusedRows = 8;
__device__ __forceinline__ void quantize_rows(const GemmParams& p, uint8_t* smem, float* x_scale, SmemTail* s) {
  const int KB = p.kblocks, groups = p.rows_total * KB, sub = threadIdx.x & 7;
  constexpr int kStep = kPromoWarps * 4;  // groups per pass
  auto load = [&](int g, uint4& v0, uint4& v1) {
    if (g < groups) {
      const uint4* src = reinterpret_cast<const uint4*>(p.x + static_cast<int64_t>(g) * BK + sub * 16);
      v0 = __ldg(src);
      v1 = __ldg(src + 1);
    }
  };
  uint4 v0 = make_uint4(0, 0, 0, 0), v1 = v0;
  load(static_cast<int>(threadIdx.x) >> 3, v0, v1);
  for (int base = 0; base < groups; base += kStep) {  // (whole warps: the shuffles below)
    const int g = base + (static_cast<int>(threadIdx.x) >> 3);
    const uint4 c0 = v0, c1 = v1;
    load(g + kStep, v0, v1);
    uint32_t m = fold_halves(absmax_u4(absmax_u4(0, c0), c1));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    float inv;
    const float sc = block_scale(bf16_bits_to_f32(m), &inv);
    uint4 out;
    encode8(c0, inv, out.x, out.y);
    encode8(c1, inv, out.z, out.w);
    if (g < groups) {
      const int row = g / KB, kb = g % KB;
      *reinterpret_cast<uint4*>(smem + kb * 1024 + row * 128 + ((sub ^ row) << 4)) = out;
      if (sub == 0) x_scale[g] = sc;
    }
  }
  fence_proxy_async_smem();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&s->x_ready);
}

template <int MODE, bool SAVE, int COLS, bool FUSED>
__global__ void __launch_bounds__(kThreads, 1)
gemm_blockscaled_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                        const __grid_constant__ CUtensorMap tm_o, const GemmParams p) {
  using C = Cfg<MODE, SAVE, COLS>;
  constexpr int kAccBufs = C::kAccBufs, HALVES = C::kHalves;
  const int kStages = COLS == 64 ? p.stages : C::kStages;
  const uint32_t a_bytes = FUSED ? 0u : COLS == 64 ? static_cast<uint32_t>(p.a_rows) * BK : kABytes;
  const uint32_t kStageBytes = a_bytes + COLS * BK;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // (COLS = 64: the MMA reads 128 token rows from a stage whatever its box holds; what lies behind the box must be shared
  // memory too, and an output row depends on its own row only)
  uint8_t* ring = smem + (FUSED ? p.kblocks * 1024 : 0);
  uint8_t* out_tile = ring + static_cast<size_t>(kStages) * kStageBytes + (COLS == 64 ? kABytes : 0);
  SmemTail* s = reinterpret_cast<SmemTail*>(out_tile + C::kStaging);
  float* x_scale = reinterpret_cast<float*>(s + 1);  // FUSED: [rows][K-blocks]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // ---- set-up: barriers, TMEM, tile list ------------------------------------------------
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s->full[i], 1);
      mbar_init(&s->empty[i], 1);
    }
    for (int i = 0; i < kAccBufs; ++i) {
      mbar_init(&s->tmem_full[i], FUSED ? 2 : 3);  // the MMA commit and the two scale warps
      mbar_init(&s->tmem_empty[i], FUSED ? 2 : kPromoWarps);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&s->amax_full[i], 2);
    mbar_init(&s->teardown, 1);
    mbar_init(&s->x_ready, kPromoWarps);
    s->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kTmaWarp && lane == 0) {
    prefetch_tensormap(&tm_a);
    prefetch_tensormap(&tm_b);
    if (C::kStaging > 0) prefetch_tensormap(&tm_o);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&s->tmem_addr, kTmemCols);
    pdl_trigger();  // not before the allocation: see pdl_trigger
    tmem_relinquish();
  }
  if (warp == kTmaWarp && lane == 0 && p.early_prefetch > 0) {
    // Decode-sized calls are bound by streaming the weights from HBM, and the kernels before
    // this one in the stream (permute, activation quantization) leave the memory system idle.
    // The weights do not depend on them, so pull this CTA's first weight tiles into L2 now.
    // Tile T is guessed as (expert T / n_tiles, column tile T % n_tiles), exact when every
    // expert has one row tile; a wrong guess only costs an unused L2 fill.
    for (int t = 0; t < p.early_prefetch; ++t) {
      const int T = blockIdx.x + t * gridDim.x;
      if (T >= p.E * p.n_tiles) break;
      const int e = T / p.n_tiles, n_tile = T % p.n_tiles;
      int row_lo, row_hi;
      if (MODE == kModeGateUp) {
        row_lo = e * p.N + n_tile * BNH;
        row_hi = row_lo + p.I;
      } else {
        row_lo = e * p.N + n_tile * COLS;
        row_hi = row_lo + BNH;
      }
      const uint64_t stream_once = l2_policy_evict_first();
      for (int kb = 0; kb < p.kblocks; ++kb) {
        tma_prefetch_2d_hint(&tm_b, kb * BK, row_lo, stream_once);
        if (HALVES == 2) tma_prefetch_2d_hint(&tm_b, kb * BK, row_hi, stream_once);
      }
    }
  }
  pdl_wait();  // everything above read no data of the predecessor; from here on its results are needed
  // Group boundaries, forced into [0, rows_total]: whatever the caller's array holds, no tile
  // and no store mask derived from it can reach outside the tensors.
  for (int e = threadIdx.x; e <= p.E; e += kThreads) {
    const int raw = p.offsets ? p.offsets[e] : (e == 0 ? 0 : p.rows_total);
    const int v = min(max(raw, 0), p.rows_total);
    if (v != raw) set_status(p.status, QARL_ERR_INVALID_ARG);
    s->off[e] = v;
  }
  __syncthreads();
  if (warp == 0) {
    // exclusive scan of tiles per expert
    int carry = 0;
    for (int base = 0; base < p.E; base += 32) {
      const int e = base + lane;
      int v = 0;
      if (e < p.E) {
        // a group that ends before it starts (offsets out of order) is reported and gets no tile;
        // with every boundary inside [0, rows_total] the other groups stay inside the tensors
        const int rows = s->off[e + 1] - s->off[e];
        if (rows < 0) set_status(p.status, QARL_ERR_INVALID_ARG);
        v = ((max(rows, 0) + BM - 1) / BM) * p.n_tiles;
      }
      int inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += u;
      }
      if (e < p.E) s->prefix[e] = carry + inc - v;
      carry += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    if (lane == 0) s->prefix[p.E] = carry;
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = s->tmem_addr;
  const int total_tiles = s->prefix[p.E];
  // Balance the static schedule: with W = ceil(tiles / CTAs) rounds, ceil(tiles / W) CTAs already
  // finish in W rounds; using exactly that many keeps every round full (768 decode tiles: 128 CTAs
  // x 6 instead of 148 CTAs of which 120 idle through the sixth round) and leaves the streaming
  // bandwidth to the CTAs that still have work.  The CTAs beyond that count retire at once.
  int num_ctas = gridDim.x;
  if (total_tiles > 0) {
    const int rounds = (total_tiles + num_ctas - 1) / num_ctas;
    num_ctas = (total_tiles + rounds - 1) / rounds;
  }
  const int first_tile = static_cast<int>(blockIdx.x) < num_ctas ? static_cast<int>(blockIdx.x) : total_tiles;
  const int KB = p.kblocks;
  const int NB = p.N / BNH;  // weight scale block-rows per expert

  if (warp >= kPromoWarps) {
    setmaxnreg_dec<kAuxRegs>();
    if (warp == kTmaWarp) {
      // =============================== TMA producer =====================================
      if (elect_one()) {
        int stage = 0;
        uint32_t phase = 0;
        uint32_t armed = 0, armed_parity = 0;  // per-stage: has a load in flight / its parity
        int armed_total = 0;
        const uint64_t stream_once = l2_policy_evict_first();
        int cur_e = 0;
        bool ok = true;
        // weight rows of a tile's two halves
        auto b_rows = [&](const TileCoord& c, int& row_lo, int& row_hi) {
          if (MODE == kModeGateUp) {
            row_lo = c.e * p.N + c.n_tile * BNH;
            row_hi = row_lo + p.I;
          } else {
            row_lo = c.e * p.N + c.n_tile * COLS;
            row_hi = row_lo + BNH;
          }
        };
        for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
          const TileCoord c = decode_tile(s, T, cur_e);
          int row_lo, row_hi;
          b_rows(c, row_lo, row_hi);
          for (int kb = 0; kb < KB; ++kb) {
            if (p.stop_after_stages >= 0 && armed_total >= p.stop_after_stages) { ok = false; break; }
            ++armed_total;
            if (!wait_or_abort(&s->empty[stage], phase ^ 1, s, p)) { ok = false; break; }
            uint8_t* a_dst = ring + static_cast<size_t>(stage) * kStageBytes;
            uint8_t* b_dst = a_dst + a_bytes;
            mbar_arrive_expect_tx(&s->full[stage], kStageBytes);
            if (!FUSED) tma_load_2d(a_dst, &tm_a, &s->full[stage], kb * BK, c.m0);
            if (p.weights_once) {
              tma_load_2d_hint(b_dst, &tm_b, &s->full[stage], kb * BK, row_lo, stream_once);
              if (HALVES == 2) tma_load_2d_hint(b_dst + kBHalfBytes, &tm_b, &s->full[stage], kb * BK, row_hi, stream_once);
            } else {
              tma_load_2d(b_dst, &tm_b, &s->full[stage], kb * BK, row_lo);
              if (HALVES == 2) tma_load_2d(b_dst + kBHalfBytes, &tm_b, &s->full[stage], kb * BK, row_hi);
            }
            armed |= 1u << stage;
            armed_parity = (armed_parity & ~(1u << stage)) | (phase << stage);
            if (++stage == kStages) { stage = 0; phase ^= 1; }
          }
        }
        if (!ok) {  // let copies in flight land before the CTA's shared memory is released
          for (int i = 0; i < kStages; ++i)
            if (armed & (1u << i)) mbar_wait_bounded(&s->full[i], (armed_parity >> i) & 1u, 20000000ull);
        }
      }
    } else if (warp == kMmaWarp) {
      // =============================== MMA issuer =======================================
      if (elect_one()) {
        constexpr uint32_t idesc = umma_idesc_e4m3_f32(BM, COLS);
        int stage = 0, ks = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = !FUSED || wait_or_abort(&s->x_ready, 0, s, p);
        for (int T = first_tile; ok && T < total_tiles; T += num_ctas) {
          for (int kb = 0; kb < KB; ++kb) {
            if (!wait_or_abort(&s->tmem_empty[ks], acc_phase ^ 1, s, p)) { ok = false; break; }
            if (!wait_or_abort(&s->full[stage], phase, s, p)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t stage_addr = smem_u32(ring + static_cast<size_t>(stage) * kStageBytes);
            const uint32_t a_addr = FUSED ? smem_u32(smem) + kb * 1024 : stage_addr;
            const uint64_t a_desc = umma_desc_k_sw128(a_addr);
            const uint64_t b_desc = umma_desc_k_sw128(stage_addr + a_bytes);
            const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(ks * COLS);
#pragma unroll
            for (int k4 = 0; k4 < BK / 32; ++k4)  // +32 bytes of K = +2 in the 16-byte address field
              umma_f8(d_tmem, a_desc + 2 * k4, b_desc + 2 * k4, idesc, k4 > 0 ? 1u : 0u);
            umma_commit(&s->empty[stage]);
            umma_commit(&s->tmem_full[ks]);
            if (++stage == kStages) { stage = 0; phase ^= 1; }
            if (++ks == kAccBufs) { ks = 0; acc_phase ^= 1; }
          }
        }
        // Nothing of this CTA's tensor work may be in flight when its TMEM and shared memory
        // go away: after a normal run every MMA has been consumed already; after an abort
        // some may still be executing, so wait (bounded) for all of them.
        if (!ok) {
          umma_commit(&s->teardown);
          mbar_wait_bounded(&s->teardown, 0, 20000000ull);
        }
      }
    } else if (!FUSED || warp == kScaleWarp) {
      // =============================== scale warps ======================================
      // Two warps, 64 rows each, form the products fl(s_x s_w) of every K-block next to its accumulator: the
      // slot is free when the accumulator is and published with it (tmem_full counts the MMA and these
      // warps), so the promotion warps wait for nothing more than before and keep their registers for sums.
      const int r0 = (warp - kScaleWarp) * 64 + lane;
      int ks = 0, cur_e = 0;
      uint32_t acc_phase = 0;
      uint32_t tile_iter = 0;
      int4 tile_info = make_int4(0, 0, 0, 0);
      float pw0 = 0.f, pw1 = 0.f;
      const float *x0 = nullptr, *x1 = nullptr, *wl = nullptr, *wh = nullptr;
      float n0 = 0.f, n1 = 0.f, nl = 0.f, nh = 0.f;  // of the next K-block: its loads fly during this one
      auto open_tile = [&](int T) {
        const TileCoord c = decode_tile(s, T, cur_e);
        int nb_lo, nb_hi;
        if (MODE == kModeGateUp) {
          nb_lo = c.n_tile;
          nb_hi = c.n_tile + p.I / BNH;
        } else {
          nb_lo = COLS == 64 ? c.n_tile / 2 : HALVES * c.n_tile;
          nb_hi = min(nb_lo + HALVES - 1, NB - 1);
        }
        if (MODE != kModeLinear) tile_info = make_int4(c.m0, c.m_end, c.n_tile, 0);
        if (MODE == kModeDown) {
          pw0 = __ldg(p.pair_weights + min(c.m0 + r0, p.rows_total - 1));
          pw1 = __ldg(p.pair_weights + min(c.m0 + r0 + 32, p.rows_total - 1));
        }
        x0 = p.a_scales + static_cast<int64_t>(min(c.m0 + r0, p.rows_total - 1)) * KB;
        x1 = p.a_scales + static_cast<int64_t>(min(c.m0 + r0 + 32, p.rows_total - 1)) * KB;
        wl = p.b_scales + (static_cast<int64_t>(c.e) * NB + nb_lo) * KB;
        wh = p.b_scales + (static_cast<int64_t>(c.e) * NB + nb_hi) * KB;
        n0 = FUSED ? x_scale[min(r0, p.rows_total - 1) * KB] : __ldg(x0);
        n1 = FUSED ? n0 : __ldg(x1);  // (FUSED: rows from 8 on are never used)
        nl = __ldg(wl);
        nh = __ldg(wh);
      };
      bool ok = !FUSED || warp_wait_or_abort(&s->x_ready, 0, s, p);
      if (ok && first_tile < total_tiles) open_tile(first_tile);
      for (int T = first_tile; ok && T < total_tiles; T += num_ctas, ++tile_iter) {
        for (int kb = 0; kb < KB; ++kb) {
          const int4 info = tile_info;
          const float w0 = pw0, w1 = pw1;
          const float2 v0 = make_float2(__fmul_rn(n0, nl), __fmul_rn(n0, nh)), v1 = make_float2(__fmul_rn(n1, nl), __fmul_rn(n1, nh));
          if (kb + 1 < KB) {
            n0 = FUSED ? x_scale[min(r0, p.rows_total - 1) * KB + kb + 1] : __ldg(x0 + kb + 1);
            n1 = FUSED ? n0 : __ldg(x1 + kb + 1);
            nl = __ldg(wl + kb + 1);
            nh = __ldg(wh + kb + 1);
          } else if (T + num_ctas < total_tiles) {
            open_tile(T + num_ctas);
          }
          if (!warp_wait_or_abort(&s->tmem_empty[ks], acc_phase ^ 1, s, p)) { ok = false; break; }
          if (MODE != kModeLinear && kb == 0) {
            if (warp == kScaleWarp && lane == 0) s->tile[tile_iter & (2 * kMaxAccBufs - 1)] = info;
            if (MODE == kModeDown) {
              s->pair_w[tile_iter & 3][r0] = w0;
              s->pair_w[tile_iter & 3][r0 + 32] = w1;
            }
          }
          s->scale[ks][r0] = v0;
          s->scale[ks][r0 + 32] = v1;
          __syncwarp();
          if (lane == 0) mbar_arrive(&s->tmem_full[ks]);
          if (++ks == kAccBufs) { ks = 0; acc_phase ^= 1; }
        }
      }
    }
  } else {
    // =============================== promotion warps ==================================
    setmaxnreg_inc<kPromoRegs>();
    if constexpr (FUSED) quantize_rows(p, smem, x_scale, s);
    // (FUSED: all rows are in TMEM quadrant 0; warps that only keep the barriers going cost those that work: one token,
    // N = 5120, K = 2048 7.0 -> 6.8 us)
    if (!FUSED || (warp & 3) == 0) promotion_role<MODE, SAVE, COLS>(tm_o, p, smem, s, first_tile, num_ctas, total_tiles);
  }

  // ---- teardown ---------------------------------------------------------------------------
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace


namespace {

// Output bf16 [rows, cols]: box of 64 columns x 32 rows, 128-byte swizzle.
CUresult make_out_tmap(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {64, 32};
  const cuuint32_t estr[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

CUresult make_tmap(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  // u8 tensor [rows, cols] row-major; box = 128 bytes x box_rows rows, 128-byte swizzle, zero fill.
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols};
  const cuuint32_t box[2] = {BK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int MODE, bool SAVE, int COLS, bool FUSED = false>
cudaError_t launch_mode(const Launch& L, const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& to,
                        const GemmParams& p, int grid) {
  // sticky per function and device; atomic: contexts on several host threads may launch at once (both
  // would set the same value)
  static std::atomic<bool> attr_set_dev[64];
  std::atomic<bool>& attr_set = attr_set_dev[L.device & 63];
  if (!attr_set.load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_blockscaled_kernel<MODE, SAVE, COLS, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(COLS == 64 ? kSmemLimit : kSmemBytes<MODE, SAVE, COLS>));
    if (e != cudaSuccess) return e;
    attr_set.store(true, std::memory_order_release);
  }
  size_t smem = kSmemBytes<MODE, SAVE, COLS>;
  if (COLS == 64)
    smem += kABytes + static_cast<size_t>(p.stages) * (p.a_rows + COLS) * BK + (FUSED ? static_cast<size_t>(p.kblocks) * (1024 + kFusedRows * 4) : 0);
  ++*L.launches;
  return launch_pdl(gemm_blockscaled_kernel<MODE, SAVE, COLS, FUSED>, static_cast<unsigned>(grid), kThreads, smem, L.stream, ta, tb, to, p);
}

}  // namespace

bool linear_fused_applies(const Launch& L, int64_t M, int64_t N, int64_t K) {
  // One launch instead of two: every CTA quantizes all rows itself, two passes over its 8 warps at most (64 groups), and has
  // one tile (one token, by graph replay: N = 5120, K = 2048 7.8 -> 6.9 us, N = 2048, K = 768 5.5 -> 4.6; 256 groups
  // would cost 12.3 against 11.1).
  return L.gemm_path == 0 && L.dense_columns == 0 && M <= kFusedRows && M * (K / BK) <= 64 && N / 64 <= L.sm_count;
}

cudaError_t launch_gemm(const Launch& L, EncodeTiledFn encode, const GemmArgs& a, CUresult* cu_err) {
  *cu_err = CUDA_SUCCESS;
  if (a.rows_total == 0) return cudaSuccess;
  // decode-sized calls: the swapped-operand kernel (bitwise the same rows, bound by the weight stream).  A dense call
  // whose 64-column tiles fit on the SMs in one round stays here: each CTA streams one tile and nobody waits for the
  // drawing of tiles (N = 2048, K = 4096, one token, by graph replay: 14.4 us there, 10.2 here; N = 16384, K = 2048:
  // 10.9 there, 13.6 here).
  const bool one_round = a.offsets == nullptr && a.N / 64 <= L.sm_count;
  const bool forced = L.dense_columns != 0 && a.mode == kModeLinear && a.offsets == nullptr;
  if (L.gemm_path == 2 ? ((a.offsets != nullptr || a.E == 1) && a.K / BK <= 64)
                       : (L.gemm_path == 0 && !forced && !one_round && gemm_decode_applies(a)))
    return launch_gemm_decode(L, encode, a, cu_err);
  // Columns per tile of a dense call: the width whose full rounds over the SMs cost least.  Per round 128 columns take
  // ~0.6 of what 256 take, 64 ~0.45 (M = 777, N = 2048, K = 4096: 56 tiles of 256 on 148 SMs 23.6 us, 112 of 128
  // columns 16.5; M = 65: 12.9 us with 128 columns, 11.6 with 64).
  int cols = BN;
  if (a.mode == kModeLinear && a.offsets == nullptr) {
    auto cost = [&](int c, double unit) {
      const int64_t tiles = ((a.rows_total + BM - 1) / BM) * ((a.N + c - 1) / c);
      return static_cast<double>((tiles + L.sm_count - 1) / L.sm_count) * unit;
    };
    double best = cost(BN, 1.0);
    if (const double c = cost(128, 0.6); c < best) { best = c; cols = 128; }
    if (const double c = cost(64, 0.45); c < best) { best = c; cols = 64; }
    if (forced) cols = L.dense_columns;
  }
  GemmParams p{};
  if (a.x != nullptr) {
    cols = 64;
    const size_t room = kSmemLimit - kSmemBytes<kModeLinear, false, 64> - kABytes - static_cast<size_t>(a.K / BK) * (1024 + kFusedRows * 4);
    p.stages = static_cast<int>(std::min<size_t>({kMaxStages, room / (64 * BK), static_cast<size_t>(a.K / BK)}));
  } else if (cols == 64) {
    p.a_rows = static_cast<int>(std::min<int64_t>(BM, (a.rows_total + 7) / 8 * 8));
    const size_t room = kSmemLimit - kSmemBytes<kModeLinear, false, 64> - kABytes;
    p.stages = static_cast<int>(std::min<size_t>({kMaxStages, room / (static_cast<size_t>(p.a_rows + 64) * BK), static_cast<size_t>(a.K / BK)}));
  }
  CUtensorMap ta, tb, to{};
  CUresult r = a.x != nullptr ? CUDA_SUCCESS : make_tmap(encode, &ta, a.a_codes, static_cast<uint64_t>(a.rows_total), static_cast<uint64_t>(a.K),
                         cols == 64 ? static_cast<uint32_t>(p.a_rows) : BM);
  if (r == CUDA_SUCCESS)
    r = make_tmap(encode, &tb, a.b_codes, static_cast<uint64_t>(a.E * a.N), static_cast<uint64_t>(a.K), cols == 64 ? 64 : BNH);
  if (r == CUDA_SUCCESS && a.out_bf16 != nullptr)
    r = make_out_tmap(encode, &to, a.out_bf16, static_cast<uint64_t>(a.rows_total), static_cast<uint64_t>(a.N));
  if (r != CUDA_SUCCESS) {
    *cu_err = r;
    return cudaErrorUnknown;
  }
  p.x = a.x;
  p.a_scales = a.a_scales;
  p.b_scales = a.b_scales;
  p.offsets = a.offsets;
  p.rows_total = static_cast<int>(a.rows_total);
  p.kblocks = static_cast<int>(a.K / BK);
  p.N = static_cast<int>(a.N);
  p.E = static_cast<int>(a.E);
  p.I = static_cast<int>(a.N / 2);
  p.n_tiles = a.mode == kModeGateUp ? static_cast<int>(a.N / 2 / BNH) : static_cast<int>((a.N + cols - 1) / cols);
  p.out_bf16 = a.out_bf16;
  p.out_f32 = a.out_f32;
  p.h_codes = a.h_codes;
  p.h_scales = a.h_scales;
  p.h_bf16 = a.h_bf16;
  p.h_vec32 = (reinterpret_cast<uintptr_t>(a.h_bf16) & 31u) == 0;
  p.pair_weights = a.pair_weights;
  p.status = L.d_status;
  p.wait_limit_ns = L.wait_limit_ns ? L.wait_limit_ns : 2000000000ull;
  p.stop_after_stages = L.stop_after_stages;
  // About one row tile per expert: a weight is read once, and read with the evict-first policy it does not push the
  // small tensors that pass between the kernels out of L2 (1501 tokens, 128 experts: gate_up 97 -> 91 us, down 60 -> 57,
  // combine 16 -> 13).
  p.weights_once = a.offsets != nullptr && a.rows_total <= a.E * BM;
  // decode-sized call (at most one row tile per expert): see the early prefetch in the kernel
  if (a.rows_total <= a.E * BM) {
    const int64_t tile_bytes = static_cast<int64_t>(p.kblocks) * 2 * kBHalfBytes;
    const int64_t budget = 80ll << 20;  // stay well inside the 126 MB L2
    p.early_prefetch = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(3, budget / (tile_bytes * L.sm_count))));
  }
  // upper bound on the tile count (group sizes live on the device): each expert adds at most
  // one partial row tile
  const int64_t m_tiles_max = a.rows_total / BM + a.E;
  const int grid = static_cast<int>(std::min<int64_t>(L.sm_count, m_tiles_max * p.n_tiles));
  switch (a.mode) {
    case kModeLinear:
      return a.x != nullptr ? launch_mode<kModeLinear, false, 64, true>(L, tb, tb, to, p, grid)
             : cols == 64  ? launch_mode<kModeLinear, false, 64>(L, ta, tb, to, p, grid)
             : cols == 128 ? launch_mode<kModeLinear, false, 128>(L, ta, tb, to, p, grid)
                           : launch_mode<kModeLinear, false, 256>(L, ta, tb, to, p, grid);
    case kModeGateUp:
      return a.out_bf16 || a.h_bf16 ? launch_mode<kModeGateUp, true, 256>(L, ta, tb, to, p, grid)
                                    : launch_mode<kModeGateUp, false, 256>(L, ta, tb, to, p, grid);
    case kModeDown: return launch_mode<kModeDown, false, 256>(L, ta, tb, to, p, grid);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qarl
