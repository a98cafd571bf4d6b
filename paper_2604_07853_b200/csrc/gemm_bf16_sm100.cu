// Dense bf16 GEMM for sm_100a: the full-precision backward of the quantized linear layer
// (Sec. 3.1 item 2: low-bit forward, backward in full precision on the bf16 master weights,
// gradients passed through the quantizer by the straight-through estimator).
//
//   C[i, j] = sum over c ascending of A(i, c) * B(j, c),   fp32 accumulation in TMEM.
//
// Each operand is given as a row-major bf16 matrix in one of two orientations:
//   K-major   memory [rows = i or j][cols = c]   (the contraction index is contiguous)
//   MN-major  memory [rows = c][cols = i or j]   (the output index is contiguous)
// so that no transposed copy of dY, X or W is ever made:
//   dX[m, k] = sum_n dY[m, n] W[n, k]:  A = dY (K-major),  B = W  (MN-major, [c = n][j = k])
//   dW[n, k] = sum_m dY[m, n] X[m, k]:  A = dY (MN-major, [c = m][i = n]),  B = X (MN-major)
// (The two-launch router's logits, sum_h x[m, h] w[e, h], take A and B K-major.)
//
// Two grouped forms serve the expert GEMMs of the MoE layer, both on the forward's expert-sorted
// row layout (expert e owns rows offsets[e] .. offsets[e+1]-1), with no padding and no copies:
//   grouped rows         C[p, :] = A[p, :] . B_e  for the expert e that owns row p  (dX of an
//                        expert projection: A = dY sorted, K-major; B = W [E, N, K], MN-major)
//   grouped contraction  C_e = sum over the expert's rows p of A[p, :]^T B[p, :]  (dW of an
//                        expert projection: both operands MN-major, the contraction runs over a
//                        ragged row range).  The last 64-row step of an expert also holds rows of
//                        the next expert: a warp overwrites those rows of both staged tiles with zeros
//                        (generic stores + proxy fence) before the step is issued, so
//                        they contribute nothing whatever they hold.
//
// Tile 128 x 256 x 64 (or 256 x 256, 128 x 192: see the host).  TMA stages both operands with the 128-byte swizzle (a K-major tile is
// one box of R rows x 128 bytes; an MN-major tile is one box of 64 c-rows x 128 bytes per 64
// output indices); one thread issues 4 x tcgen05.mma kind::f16 (128 x 256 x 16) per stage with
// the matching operand-major bits; two 256-column TMEM accumulators let the epilogue of a tile
// overlap the main loop of the next.  The epilogue writes through shared-memory boxes of 32 rows x 128 bytes and
// TMA stores: rows stored straight from registers (16 bytes of 32 different rows per instruction, half
// sectors) took four times as long as the MMAs of a short contraction -- expert dW of 8192 tokens (128 experts,
// 1536 x 2048, 1.6 GB out) 1010 us of which the stores need 250.  Static persistent schedule, row tiles fastest
// (grouped contraction: long and short tiles in turn, see the producer).  One fixed
// order of accumulation: a result does not depend on the grid or on the other rows.
// Every wait on an mbarrier is bounded (status word + CTA-wide abort flag), as in the other GEMMs.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "sched.cuh"

namespace qarl {
namespace {

using namespace ptx;

constexpr int BM = 128, BK = 64;
constexpr int kMaxStages = 4, kMaxAccBufs = 2;
constexpr uint32_t kAHalfBytes = BM * BK * 2;   // 16 KB: 128 output rows x 64 contraction elements
// an epilogue warp's rows on their way out: boxes of 32 rows x 128 bytes (128-byte swizzle)
constexpr uint32_t kOutBoxBytes = 32 * 128;
// A tile holds MT x 128 output rows.  The kernel is bound by the bytes it can keep in flight from
// L2/HBM (shared-memory capacity over load latency: throughput grew linearly with the ring depth),
// so dense calls may take MT = 2 (the host picks by rounds): both 128-row halves share one B tile, a
// third fewer bytes per flop, but one set of accumulators is left, i.e. an epilogue that is not overlapped.
enum { kDense = 0, kGroupedRows = 1, kGroupedContraction = 2 };
template <int GROUP, int MT, int BN>
struct Cfg {
  static constexpr int kRows = MT * BM;
  static constexpr uint32_t kABytes = MT * kAHalfBytes;
  static constexpr uint32_t kBBytes = BN * BK * 2;
  static constexpr uint32_t kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = MT == 2 ? 3 : 4;
  static constexpr int kAccBufs = MT == 1 ? 2 : 1;
  // Warps 0 .. kEpiWarps - 1: TMEM quadrant = warp % 4; with eight, two share a quadrant and take the 128-byte
  // column chunks in turn (each has one box; grouped rows need the shared memory for the tile list).
  static constexpr int kEpiWarps = GROUP == kGroupedRows ? 4 : 8;
  static constexpr int kTmaWarp = kEpiWarps;
  static constexpr int kMmaWarp = kEpiWarps + 1;
  static constexpr int kFixWarp = kEpiWarps + 2;
  static constexpr int kThreads = (kEpiWarps + 3) * 32;
  static constexpr uint32_t kOutBytes = kEpiWarps * kOutBoxBytes;
};
constexpr uint32_t kBlockBytes = 64 * BK * 2;  // one MN-major block: 64 output indices x 64 c-rows
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxExperts = 1024;
constexpr int kTurn = 8;  // grouped contraction: steps of the long tile between two short ones:
// about the time a tile takes to be written (4 .. 20 measure alike)
struct Bf16Params {
  int Mo, No, Kc;           // grouped rows: Mo = total rows P;  grouped contraction: Kc unused (from offsets)
  const int32_t* offsets;   // [E + 1] (grouped forms)
  int E;
  int rows_total;           // grouped contraction: P
  int a3d, b3d;             // MN-major operand staged by one 3-D TMA box (64 columns x 64 rows x blocks)
  int col_fastest;          // dense: consecutive tiles walk the column tiles of a row tile (else the row tiles of a column tile)
  uint16_t* c_bf16;   // [Mo, No] or nullptr
  float* c_f32;       // [Mo, No] or nullptr
  int* status;
  unsigned long long wait_limit_ns;
  int stop_after_stages;  // test harness only (< 0: off): the TMA producer stops arming stages after this many
};

struct __align__(8) SmemTail {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t fixed[kMaxStages];  // grouped contraction: the overhang rows of a ragged step are zero
  uint64_t tmem_full[kMaxAccBufs];
  uint64_t tmem_empty[kMaxAccBufs];
  uint64_t teardown;
  uint32_t tmem_addr;
  int abort_flag;
};
// Grouped contraction: experts by falling row count.  (uint16 and at most kMaxSorted of them: what the ring and the
// boxes leave of shared memory; more experts are taken in index order.)
constexpr int kMaxSorted = 512;
struct SmemOrder {
  uint32_t step[kMaxStages];    // what a staged step is: accumulator | first << 1 | last << 2 | valid rows << 3
  int32_t tile_at[2][8];        // list index of the tiles opened in each accumulator, the last eight
  uint16_t order[kMaxSorted];
};
struct SmemLists {  // grouped rows: the tile list
  int32_t off[kMaxExperts + 1];
  int32_t prefix[kMaxExperts + 1];
};
template <int GROUP, int MT, int BN>
constexpr size_t smem_bytes() {
  using C = Cfg<GROUP, MT, BN>;
  return 1024 + static_cast<size_t>(C::kStages) * C::kStageBytes + C::kOutBytes + sizeof(SmemTail) +
         (GROUP == kGroupedRows ? sizeof(SmemLists) : GROUP == kGroupedContraction ? sizeof(SmemOrder) : 0);
}
static_assert(smem_bytes<kDense, 1, 256>() <= 227 * 1024 && smem_bytes<kDense, 1, 192>() <= 227 * 1024 &&
                  smem_bytes<kDense, 2, 256>() <= 227 * 1024 && smem_bytes<kGroupedRows, 1, 256>() <= 227 * 1024 &&
                  smem_bytes<kGroupedContraction, 1, 256>() <= 227 * 1024,
              "shared memory budget");

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const Bf16Params& p) {
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

// The same for a whole warp: every lane polls, then the lanes vote, so all 32 take the same
// branch and the warp-wide operations that follow never see a split warp (lanes polling on
// their own could disagree when a barrier completes right at the limit).
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t* bar, uint32_t parity, SmemTail* s, const Bf16Params& p) {
  return __all_sync(0xFFFFFFFFu, wait_or_abort(bar, parity, s, p) ? 1 : 0) != 0;
}

// Which accumulator's tile is complete (the whole warp takes the same answer); -1 after an abort.
__device__ __forceinline__ int either_full(SmemTail* s, const Bf16Params& p, uint32_t parity0, uint32_t parity1) {
  unsigned long long t0 = 0;
  for (int spins = 0;; ++spins) {
    const bool r0 = mbar_test_wait(&s->tmem_full[0], parity0), r1 = mbar_test_wait(&s->tmem_full[1], parity1);
    if (__all_sync(0xFFFFFFFFu, r0)) return 0;
    if (__all_sync(0xFFFFFFFFu, r1)) return 1;
    if ((spins & 255) == 255) {
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      bool stop = *reinterpret_cast<volatile int*>(&s->abort_flag) != 0;
      if (now - t0 > p.wait_limit_ns) {
        set_status(p.status, QARL_ERR_DEVICE_TIMEOUT);
        *reinterpret_cast<volatile int*>(&s->abort_flag) = 1;
        stop = true;
      }
      if (__any_sync(0xFFFFFFFFu, stop)) return -1;
    }
  }
}

__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&b);
}

template <bool A_MN, bool B_MN, int GROUP, int MT, int BN>
__global__ void __launch_bounds__(Cfg<GROUP, MT, BN>::kThreads, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                 const __grid_constant__ CUtensorMap tm_f32, const __grid_constant__ CUtensorMap tm_bf16,
                 const Bf16Params p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  using C = Cfg<GROUP, MT, BN>;
  constexpr int kStages = C::kStages, kAccBufs = C::kAccBufs, TM = C::kRows;
  constexpr uint32_t kABytes = C::kABytes, kStageBytes = C::kStageBytes;
  constexpr int kEpiWarps = C::kEpiWarps, kTmaWarp = C::kTmaWarp, kMmaWarp = C::kMmaWarp;
  uint8_t* out_boxes = smem + static_cast<size_t>(kStages) * kStageBytes;
  SmemTail* s = reinterpret_cast<SmemTail*>(out_boxes + C::kOutBytes);
  SmemLists* lists = reinterpret_cast<SmemLists*>(s + 1);
  SmemOrder* list = reinterpret_cast<SmemOrder*>(s + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s->full[i], 1);
      mbar_init(&s->empty[i], GROUP == kGroupedContraction ? 2 : 1);  // the MMAs (and the warp that follows ragged steps)
      mbar_init(&s->fixed[i], 1);
    }
    for (int i = 0; i < kAccBufs; ++i) {
      mbar_init(&s->tmem_full[i], 1);
      mbar_init(&s->tmem_empty[i], kEpiWarps);
    }
    mbar_init(&s->teardown, 1);
    s->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kTmaWarp && lane == 0) {
    prefetch_tensormap(&tm_a);
    prefetch_tensormap(&tm_b);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&s->tmem_addr, kTmemCols);
    pdl_trigger();  // not before the allocation: see pdl_trigger
    tmem_relinquish();
  }
  pdl_wait();
  const int n_tiles = (p.No + BN - 1) / BN;
  const int m_tiles = GROUP == kGroupedRows ? 1 : (p.Mo + TM - 1) / TM;  // grouped rows: tiles come from the offsets
  if (GROUP == kGroupedRows) {
    build_tile_list(lists->off, lists->prefix, p.offsets, p.Mo, p.E, TM, n_tiles);
  }
  auto expert_rows = [&](int e, int& first) {  // grouped contraction; whatever the array holds stays inside the tensors
    first = min(max(__ldg(p.offsets + e), 0), p.rows_total);
    return max(min(max(__ldg(p.offsets + e + 1), 0), p.rows_total) - first, 0);
  };
  if (GROUP == kGroupedContraction && p.E <= kMaxSorted) {
    int* rows = reinterpret_cast<int*>(out_boxes);  // (free until the first tile is written out)
    for (int e = threadIdx.x; e < p.E; e += C::kThreads) {
      int first;
      rows[e] = expert_rows(e, first);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < p.E; e += C::kThreads) {
      const int mine = rows[e];
      int rank = 0;
      for (int f = 0; f < p.E; ++f) rank += rows[f] > mine || (rows[f] == mine && f < e);
      list->order[rank] = static_cast<uint16_t>(e);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = s->tmem_addr;
  const int total_tiles = GROUP == kGroupedRows ? lists->prefix[p.E]
                        : GROUP == kGroupedContraction ? p.E * m_tiles * n_tiles : m_tiles * n_tiles;
  const int grid = gridDim.x;

  // Everything a role needs to know about tile T.  i0 / j0: first output row / column; a_c0 / b_c0:
  // first contraction coordinate of A / B; KS: 64-element contraction steps; last_valid: contraction
  // elements of the last step that belong to this tile (64 = all); row_end: end of the rows that
  // may be stored.
  struct Tile {
    int i0, j0, a_c0, b_c0, KS, last_valid, row_end;
    int e;       // grouped contraction: whose output matrix
    int b_row0;  // K-major B: first row of the expert's block
  };
  auto tile_of = [&](int T, int& cur_e) {  // cur_e: where the caller's walk over the groups stands
    Tile t{};
    t.last_valid = BK;
    if (GROUP == kDense) {
      // CTAs that run at the same time take consecutive T.  Walking the column tiles of one row tile
      // together (col_fastest) lets a wave of CTAs read each block of A once and share it through L2;
      // walking the row tiles of one column tile together does the same for B.  The host picks the
      // order that re-reads the smaller operand.
      if (p.col_fastest) {
        t.i0 = (T / n_tiles) * TM;
        t.j0 = (T % n_tiles) * BN;
      } else {
        t.i0 = (T % m_tiles) * TM;
        t.j0 = (T / m_tiles) * BN;
      }
      t.KS = (p.Kc + BK - 1) / BK;  // a ragged last step reads zeros (TMA out-of-range fill)
      t.row_end = p.Mo;
    } else if (GROUP == kGroupedRows) {
      const TileCoord c = decode_tile(lists->off, lists->prefix, TM, T, cur_e);
      t.i0 = c.m0;
      t.j0 = c.n_tile * BN;
      t.KS = p.Kc / BK;             // Kc is a multiple of 64 here: a step never runs into the next expert's weights
      t.a_c0 = 0;
      t.b_c0 = c.e * p.Kc;          // MN-major B: the expert's [Kc, No] block starts at row e Kc
      t.b_row0 = c.e * p.No;        // K-major B: the expert's [No, Kc] block starts at row e No
      t.row_end = c.m_end;
    }
    return t;
  };
  // Grouped contraction: this CTA's list holds every grid-th tile of the experts by falling row count, the direction
  // turning round with each lap (so that the CTAs' sums of rows stay close).
  const int list_len = total_tiles / grid + ((total_tiles / grid & 1 ? grid - 1 - static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x)) < total_tiles % grid);
  auto list_tile = [&](int i) {
    const int T = i * grid + (i & 1 ? grid - 1 - static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x));
    const int per_e = m_tiles * n_tiles, r = T % per_e;
    Tile t{};
    t.e = p.E <= kMaxSorted ? list->order[T / per_e] : T / per_e;
    t.i0 = (r % m_tiles) * TM;
    t.j0 = (r / m_tiles) * BN;
    int first;
    const int rows = expert_rows(t.e, first);
    t.KS = (rows + BK - 1) / BK;
    t.last_valid = rows - (t.KS - 1) * BK;
    t.a_c0 = t.b_c0 = first;
    t.row_end = p.Mo;
    return t;
  };
  int live_tiles = 0;  // of the list: with rows
  if (GROUP == kGroupedContraction) {
    for (int base = 0; base < list_len; base += 32)
      live_tiles += __popc(__ballot_sync(0xFFFFFFFFu, base + lane < list_len && list_tile(base + lane).KS > 0));
  }
  if (warp == kTmaWarp) {
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t armed = 0, armed_parity = 0;
      int armed_total = 0;
      bool ok = true;
      // steps [from, to) of tile t into the ring
      auto feed = [&](const Tile& t, int from, int to, int acc) {
        const int i0 = t.i0, j0 = t.j0;
        for (int ks = from; ks < to; ++ks) {
          if (p.stop_after_stages >= 0 && armed_total >= p.stop_after_stages) { ok = false; return; }
          ++armed_total;
          if (!wait_or_abort(&s->empty[stage], phase ^ 1, s, p)) { ok = false; return; }
          uint8_t* a_dst = smem + static_cast<size_t>(stage) * kStageBytes;
          uint8_t* b_dst = a_dst + kABytes;
          if (GROUP == kGroupedContraction) {
            const bool last = ks == t.KS - 1;
            *reinterpret_cast<volatile uint32_t*>(&list->step[stage]) =
                acc | (ks == 0 ? 2u : 0u) | (last ? 4u : 0u) | static_cast<uint32_t>(last ? t.last_valid : BK) << 3;
          }
          mbar_arrive_expect_tx(&s->full[stage], kStageBytes);
          if (A_MN && p.a3d) {
            tma_load_3d(a_dst, &tm_a, &s->full[stage], 0, t.a_c0 + ks * BK, i0 / 64);
          } else if (A_MN) {
#pragma unroll
            for (int b = 0; b < TM / 64; ++b)
              tma_load_2d(a_dst + b * kBlockBytes, &tm_a, &s->full[stage], i0 + 64 * b, t.a_c0 + ks * BK);
          } else {  // one box of TM rows x 128 bytes
            tma_load_2d(a_dst, &tm_a, &s->full[stage], t.a_c0 + ks * BK, i0);
          }
          if (B_MN && p.b3d) {
            tma_load_3d(b_dst, &tm_b, &s->full[stage], 0, t.b_c0 + ks * BK, j0 / 64);
          } else if (B_MN) {
#pragma unroll
            for (int b = 0; b < BN / 64; ++b)
              tma_load_2d(b_dst + b * kBlockBytes, &tm_b, &s->full[stage], j0 + 64 * b, t.b_c0 + ks * BK);
          } else {
            tma_load_2d(b_dst, &tm_b, &s->full[stage], ks * BK, t.b_row0 + j0);
          }
          armed |= 1u << stage;
          armed_parity = (armed_parity & ~(1u << stage)) | (phase << stage);
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      };
      if constexpr (GROUP == kGroupedContraction) {
        // Two tiles at a time, one per accumulator: long ones from the head of the list in the first, short ones
        // from its tail in the second, a short one whole after every kTurn steps of the long one.  Every tile writes
        // 128 KB however few rows its expert has, so a run of short tiles is bound by the stores and a long tile by
        // its MMAs; taken in turn they overlap (8192 tokens, 128 experts with Zipf popularity 1.1: the two dW GEMMs
        // 1027 us tile after tile by expert, 844 so).
        int head = 0, tail = list_len - 1;
        uint32_t opened[2] = {0, 0};
        auto open = [&](int i, int acc) {
          const Tile t = list_tile(i);
          if (t.KS > 0) *reinterpret_cast<volatile int32_t*>(&list->tile_at[acc][opened[acc]++ & 7]) = i;
          return t;
        };
        while (ok && head <= tail) {
          const Tile t = open(head++, 0);
          for (int ks = 0; ok && ks < t.KS;) {
            const int to = head <= tail ? min(ks + kTurn, t.KS) : t.KS;
            feed(t, ks, to, 0);
            ks = to;
            if (ok && head <= tail) {
              const Tile u = open(tail--, 1);
              feed(u, 0, u.KS, 1);
            }
          }
        }
      } else {
        int cur_e = 0;
        for (int T = blockIdx.x; ok && T < total_tiles; T += grid) {
          const Tile t = tile_of(T, cur_e);
          feed(t, 0, t.KS, 0);
        }
      }
      if (!ok) {
        for (int i = 0; i < kStages; ++i)
          if (armed & (1u << i)) mbar_wait_bounded(&s->full[i], (armed_parity >> i) & 1u, 20000000ull);
      }
    }
  } else if (warp == kMmaWarp) {
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc_bf16_f32_major(BM, BN, A_MN, B_MN);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // the first `slices` 16-element slices of the staged step; 16 contraction elements further on: 32 bytes
      // inside a K-major row, 16 rows of 128 bytes in an MN-major block (start-address field counts 16-byte units)
      auto issue = [&](uint32_t d_tmem, bool first, int slices) {
        tc_fence_after_sync();
        const uint32_t a_addr = smem_u32(smem + static_cast<size_t>(stage) * kStageBytes);
        const uint32_t b_addr = a_addr + kABytes;
        const uint64_t a_desc = A_MN ? umma_desc_mn_sw128(a_addr, kBlockBytes) : umma_desc_k_sw128(a_addr);
        const uint64_t b_desc = B_MN ? umma_desc_mn_sw128(b_addr, kBlockBytes) : umma_desc_k_sw128(b_addr);
        constexpr uint32_t a_step = A_MN ? (16 * 128) >> 4 : 32 >> 4;
        constexpr uint32_t b_step = B_MN ? (16 * 128) >> 4 : 32 >> 4;
        if (slices == BK / 16) {
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)  // the 128-row halves of A share the B tile
#pragma unroll
            for (int k4 = 0; k4 < BK / 16; ++k4)
              umma_bf16(d_tmem + mt * BN, a_desc + mt * (kAHalfBytes >> 4) + a_step * k4, b_desc + b_step * k4, idesc,
                        (!first || k4 > 0) ? 1u : 0u);
        } else {  // (MT is 1 in the form that has these)
          for (int k4 = 0; k4 < slices; ++k4)
            umma_bf16(d_tmem, a_desc + a_step * k4, b_desc + b_step * k4, idesc, (!first || k4 > 0) ? 1u : 0u);
        }
        umma_commit(&s->empty[stage]);
      };
      auto next_stage = [&]() {
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      };
      if constexpr (GROUP == kGroupedContraction) {
        uint32_t acc_phase = 0, fix_phase = 0;  // a bit per accumulator; per stage, flipping only when it held a ragged step
        for (int done = 0; done < live_tiles;) {
          if (!wait_or_abort(&s->full[stage], phase, s, p)) { ok = false; break; }
          const uint32_t step = *reinterpret_cast<volatile uint32_t*>(&list->step[stage]);
          const uint32_t acc = step & 1u;
          const int valid = static_cast<int>(step >> 3);
          if ((step & 2u) && !wait_or_abort(&s->tmem_empty[acc], ((acc_phase >> acc) & 1u) ^ 1u, s, p)) { ok = false; break; }
          if (valid < BK) {
            if (!wait_or_abort(&s->fixed[stage], (fix_phase >> stage) & 1u, s, p)) { ok = false; break; }
            fix_phase ^= 1u << stage;
          }
          issue(tmem_base + acc * BN, (step & 2u) != 0, (valid + 15) / 16);
          if (step & 4u) {
            umma_commit(&s->tmem_full[acc]);
            acc_phase ^= 1u << acc;
            ++done;
          }
          next_stage();
        }
      } else {
        int acc = 0, cur_e = 0;
        uint32_t acc_phase = 0;
        for (int T = blockIdx.x; ok && T < total_tiles; T += grid) {
          const Tile t = tile_of(T, cur_e);
          if (t.KS == 0) continue;  // an empty contraction: the epilogue writes zeros, no accumulator is used
          if (!wait_or_abort(&s->tmem_empty[acc], acc_phase ^ 1, s, p)) { ok = false; break; }
          for (int ks = 0; ks < t.KS; ++ks) {
            if (!wait_or_abort(&s->full[stage], phase, s, p)) { ok = false; break; }
            issue(tmem_base + static_cast<uint32_t>(acc * MT) * BN, ks == 0, BK / 16);
            if (ks == t.KS - 1) umma_commit(&s->tmem_full[acc]);
            next_stage();
          }
          if (++acc == kAccBufs) { acc = 0; acc_phase ^= 1; }
        }
      }
      // Nothing of this CTA's tensor work may be in flight when its TMEM and shared memory go
      // away: after an abort some MMAs may still be executing, so wait (bounded) for them.
      if (!ok) {
        umma_commit(&s->teardown);
        mbar_wait_bounded(&s->teardown, 0, 20000000ull);
      }
    }
  } else if (GROUP == kGroupedContraction && warp == C::kFixWarp) {
    // =============================== ragged steps =====================================
    // The last 64-row step of an expert also holds rows of the next one.  This warp zeroes what the last 16-row
    // slice holds of them in both staged tiles (in one alone 0 x inf and 0 x NaN would still be NaN) as soon as the
    // step has landed, ahead of the MMA thread (which did this itself once: ~2000 clocks of a tile's ~12000).
    int stage = 0;
    uint32_t phase = 0;
    // every step is followed (and counted in `empty`): a parity wait tells neighbouring fills apart, no more
    for (int done = 0; done < live_tiles;) {
      if (!warp_wait_or_abort(&s->full[stage], phase, s, p)) break;
      const uint32_t step = *reinterpret_cast<volatile uint32_t*>(&list->step[stage]);
      const int valid = static_cast<int>(step >> 3);
      if (valid < BK) {
        uint8_t* tiles = smem + static_cast<size_t>(stage) * kStageBytes;  // A's blocks of 64 columns, then B's
        const int chunks = (-valid & 15) * 8;
#pragma unroll
        for (int blk = 0; blk < (TM + BN) / 64; ++blk)
          for (int i = lane; i < chunks; i += 32)  // (rows are 128 bytes: chunk i of the overhang is at valid * 128 + 16 i)
            *reinterpret_cast<uint4*>(tiles + blk * kBlockBytes + valid * 128 + i * 16) = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->fixed[stage]);
      }
      if (step & 4u) ++done;
      __syncwarp();  // every lane has read the step's word
      if (lane == 0) mbar_arrive(&s->empty[stage]);
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
  } else if (warp < kEpiWarps) {
    // =============================== epilogue warps: TMEM -> box -> TMA store ==========
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    uint8_t* my_box = out_boxes + static_cast<size_t>(warp) * kOutBoxBytes;
    constexpr int kTurns = kEpiWarps / 4;  // warps that share a quadrant's columns
    // this warp's share of tile t out of accumulator `acc` (have_acc false: an expert without rows gets zeros)
    auto write_out = [&](const Tile& t, const bool have_acc, const int acc) {
#pragma unroll 1
      for (int mt = 0; mt < MT; ++mt) {
        const int row0 = t.i0 + mt * BM + (warp & 3) * 32;
        if (row0 >= t.row_end) continue;
        const uint32_t t0 = tmem_base + lane_addr + static_cast<uint32_t>((acc * MT + mt) * BN);
        // rows past a group's end are the next expert's: then the box is copied row by row
        const bool whole = GROUP != kGroupedRows || row0 + 32 <= t.row_end;
        auto start = [&](int col, uint32_t (&v)[32]) {
          if (have_acc) {
            tmem_ld_x32(t0 + col, v);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0u;
          }
        };
        auto box_free = [&]() {  // TMA has read what the box held
          if (lane == 0) bulk_wait_group_read_all();
          __syncwarp();
        };
        auto put = [&](int j, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
          *reinterpret_cast<uint4*>(my_box + lane * 128 + ((j ^ (lane & 7)) << 4)) = make_uint4(w0, w1, w2, w3);
        };
        // box of 32 rows x 128 bytes at output column `col` (element size `es`)
        auto send = [&](const CUtensorMap* m, void* base, int col, int es) {
          if (whole) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
              tma_store_3d(m, my_box, col, row0, GROUP == kGroupedContraction ? t.e : 0);
              bulk_commit_group();
            }
            __syncwarp();  // (an aligned tcgen05 instruction may follow)
          } else {
            __syncwarp();
            const int chunk = lane & 7, c = col + chunk * (16 / es);
            for (int rr = lane >> 3; row0 + rr < t.row_end; rr += 4) {
              const uint4 v = *reinterpret_cast<const uint4*>(my_box + rr * 128 + ((chunk ^ (rr & 7)) << 4));
              if (c < p.No)
                *reinterpret_cast<uint4*>(static_cast<uint8_t*>(base) + (static_cast<int64_t>(row0 + rr) * p.No + c) * es) = v;
            }
            __syncwarp();
          }
        };
        const int cols = min(BN, p.No - t.j0);
        if (p.c_f32) {
          // the next chunk is on its way from TMEM while this one is written out
          constexpr int kStep = 32 * kTurns;
          uint32_t v[2][32];
          const int first = (warp >> 2) * 32;
          if (first < cols) start(first, v[0]);
#pragma unroll 2
          for (int i = 0; first + i * kStep < cols; ++i) {
            const int c = first + i * kStep;
            tmem_ld_wait();
            if (c + kStep < cols) start(c + kStep, v[(i + 1) & 1]);
            box_free();
            const uint32_t(&u)[32] = v[i & 1];
#pragma unroll
            for (int j = 0; j < 8; ++j) put(j, u[4 * j], u[4 * j + 1], u[4 * j + 2], u[4 * j + 3]);
            send(&tm_f32, p.c_f32, t.j0 + c, 4);
          }
          tmem_ld_wait();
        }
        if (p.c_bf16) {
          for (int c = (warp >> 2) * 64; c < cols; c += 64 * kTurns) {
            uint32_t v[2][32];
            start(c, v[0]);
            start(c + 32, v[1]);
            tmem_ld_wait();
            box_free();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t* u = &v[j >> 2][8 * (j & 3)];
              put(j, bf16x2_bits(__uint_as_float(u[0]), __uint_as_float(u[1])), bf16x2_bits(__uint_as_float(u[2]), __uint_as_float(u[3])),
                  bf16x2_bits(__uint_as_float(u[4]), __uint_as_float(u[5])), bf16x2_bits(__uint_as_float(u[6]), __uint_as_float(u[7])));
            }
            send(&tm_bf16, p.c_bf16, t.j0 + c, 2);
          }
        }
      }
      if (have_acc) {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&s->tmem_empty[acc]);
      }
    };
    if constexpr (GROUP == kGroupedContraction) {
      if (live_tiles < list_len) {
        for (int i = 0; i < list_len; ++i) {
          const Tile t = list_tile(i);
          if (t.KS == 0) write_out(t, false, 0);
        }
      }
      uint32_t seen[2] = {0, 0};
      for (int done = 0; done < live_tiles; ++done) {  // whichever accumulator is complete
        const int acc = either_full(s, p, seen[0] & 1u, seen[1] & 1u);
        if (acc < 0) break;
        tc_fence_after_sync();
        const int i = *reinterpret_cast<volatile int32_t*>(&list->tile_at[acc][(acc ? seen[1] : seen[0]) & 7]);
        if (acc) ++seen[1];
        else ++seen[0];
        write_out(list_tile(i), true, acc);
      }
    } else {
      int acc = 0, cur_e = 0;
      uint32_t acc_phase = 0;
      for (int T = blockIdx.x; T < total_tiles; T += grid) {
        const Tile t = tile_of(T, cur_e);
        if (t.KS == 0) {
          write_out(t, false, 0);
          continue;
        }
        if (!warp_wait_or_abort(&s->tmem_full[acc], acc_phase, s, p)) break;
        tc_fence_after_sync();
        write_out(t, true, acc);
        if (++acc == kAccBufs) { acc = 0; acc_phase ^= 1; }
      }
    }
    if (lane == 0) bulk_wait_group_all();  // this warp's rows are written
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Tensor map of a row-major bf16 matrix [rows, cols] with a box of box_cols x box_rows elements.
CUresult make_tmap(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols,
                   uint32_t box_cols, uint32_t box_rows) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// An MN-major matrix [rows, cols] (cols % 64 == 0) seen as 64-column blocks: dims {64, rows, cols / 64};
// one box of 64 x 64 x nblocks lands as nblocks consecutive 8 KB blocks, the layout the descriptor expects.
// The issuing thread pays per TMA instruction, so one box per operand instead of one per block matters.
CUresult make_tmap_mn3d(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols,
                        uint32_t nblocks) {
  const cuuint64_t dims[3] = {64, rows, cols / 64};
  const cuuint64_t strides[2] = {cols * 2, 128};
  const cuuint32_t box[3] = {64, BK, nblocks};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// Output matrices [count][rows, cols] of elements of `es` bytes: box of 128 bytes x 32 rows, 128-byte swizzle.
CUresult make_out_tmap(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t count, uint64_t rows, uint64_t cols, uint32_t es) {
  const cuuint64_t dims[3] = {cols, rows, count};
  const cuuint64_t strides[2] = {cols * es, rows * cols * es};
  const cuuint32_t box[3] = {128 / es, 32, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return encode(m, es == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
                strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

struct Maps {
  CUtensorMap a, b, f32, bf16;
};

template <bool A_MN, bool B_MN, int GROUP, int MT, int BN>
cudaError_t launch_variant(const Launch& L, const Maps& tm, const Bf16Params& p, int64_t tiles) {
  // sticky per function and device; atomic: contexts on several host threads may launch at once (both
  // would set the same value)
  static std::atomic<bool> attr_set_dev[64];
  std::atomic<bool>& attr_set = attr_set_dev[L.device & 63];
  if (!attr_set.load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(gemm_bf16_kernel<A_MN, B_MN, GROUP, MT, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem_bytes<GROUP, MT, BN>()));
    if (e != cudaSuccess) return e;
    attr_set.store(true, std::memory_order_release);
  }
  // full rounds only: with W = ceil(tiles / SMs) rounds, ceil(tiles / W) CTAs finish in W rounds
  // (for grouped rows `tiles` is an upper bound: the surplus CTAs find no tile and retire)
  const int64_t rounds = std::max<int64_t>(1, (tiles + L.sm_count - 1) / L.sm_count);
  const int grid = static_cast<int>(std::max<int64_t>(1, (tiles + rounds - 1) / rounds));
  ++*L.launches;
  return launch_pdl(gemm_bf16_kernel<A_MN, B_MN, GROUP, MT, BN>, static_cast<unsigned>(grid), Cfg<GROUP, MT, BN>::kThreads, smem_bytes<GROUP, MT, BN>(), L.stream,
                    tm.a, tm.b, tm.f32, tm.bf16, p);
}

template <int GROUP, int MT, int BN>
cudaError_t launch_majors(const Launch& L, const Maps& tm, const Bf16Params& p, int64_t tiles, bool a_mn, bool b_mn) {
  if constexpr (GROUP == kGroupedContraction) return launch_variant<true, true, GROUP, MT, BN>(L, tm, p, tiles);
  if constexpr (GROUP != kGroupedRows)  // (grouped rows: A is K-major)
    if (a_mn)
      return b_mn ? launch_variant<true, true, GROUP, MT, BN>(L, tm, p, tiles) : launch_variant<true, false, GROUP, MT, BN>(L, tm, p, tiles);
  return b_mn ? launch_variant<false, true, GROUP, MT, BN>(L, tm, p, tiles) : launch_variant<false, false, GROUP, MT, BN>(L, tm, p, tiles);
}

}  // namespace

cudaError_t launch_gemm_bf16(const Launch& L, EncodeTiledFn encode, const GemmBf16Args& a, CUresult* cu_err) {
  *cu_err = CUDA_SUCCESS;
  if (a.Mo == 0 || a.No == 0) return cudaSuccess;
  const bool grouped_rows = a.group == 1, grouped_k = a.group == 2;
  // Tile of the dense form: the one whose full rounds over the SMs cost least.  A round of 128 x 256 tiles is the
  // unit; 256 x 256 tiles move a third fewer operand bytes (measured: 13 % less time per unit of work), 128 x 192
  // tiles cost in proportion.  The grouped forms keep 128 x 256 (ragged groups waste more of a 256-row tile
  // and its single accumulator set exposes the epilogue of short contractions).
  int MT = 1, BN = 256;
  if (a.group == 0) {
    auto cost = [&](int rows, int cols, double unit) {
      const int64_t tiles = ((a.Mo + rows - 1) / rows) * ((a.No + cols - 1) / cols);
      return static_cast<double>((tiles + L.sm_count - 1) / L.sm_count) * unit;
    };
    double best = cost(BM, 256, 1.0);
    if (const double c = cost(2 * BM, 256, 2.0 * 0.87); c < best) { best = c; MT = 2; }
    if (const double c = cost(BM, 192, 0.77); c < best) { best = c; MT = 1; BN = 192; }
  }
  const int TM = MT * BM;
  // rows of the tensors as TMA sees them
  const int64_t a_rows = a.a_mn_major ? (grouped_k ? a.rows_total : a.Kc) : a.Mo;
  const int64_t b_rows = a.b_mn_major ? (grouped_k ? a.rows_total : (grouped_rows ? a.E * a.Kc : a.Kc))
                                      : (grouped_rows ? a.E * a.No : a.No);
  Maps tm{};
  const bool a3d = a.a_mn_major && a.Mo % 64 == 0, b3d = a.b_mn_major && a.No % 64 == 0;
  CUresult r = a3d ? make_tmap_mn3d(encode, &tm.a, a.a, a_rows, a.Mo, TM / 64)
             : a.a_mn_major ? make_tmap(encode, &tm.a, a.a, a_rows, a.Mo, 64, BK) : make_tmap(encode, &tm.a, a.a, a_rows, a.Kc, BK, TM);
  if (r == CUDA_SUCCESS)
    r = b3d ? make_tmap_mn3d(encode, &tm.b, a.b, b_rows, a.No, BN / 64)
      : a.b_mn_major ? make_tmap(encode, &tm.b, a.b, b_rows, a.No, 64, BK) : make_tmap(encode, &tm.b, a.b, b_rows, a.Kc, BK, BN);
  const uint64_t out_count = grouped_k ? static_cast<uint64_t>(a.E) : 1;
  if (r == CUDA_SUCCESS && a.c_f32) r = make_out_tmap(encode, &tm.f32, a.c_f32, out_count, a.Mo, a.No, 4);
  if (r == CUDA_SUCCESS && a.c_bf16) r = make_out_tmap(encode, &tm.bf16, a.c_bf16, out_count, a.Mo, a.No, 2);
  if (r != CUDA_SUCCESS) {
    *cu_err = r;
    return cudaErrorUnknown;
  }
  Bf16Params p{};
  p.Mo = static_cast<int>(a.Mo);
  p.No = static_cast<int>(a.No);
  p.Kc = static_cast<int>(a.Kc);
  p.offsets = a.offsets;
  p.E = static_cast<int>(a.E);
  p.rows_total = static_cast<int>(a.rows_total);
  p.a3d = a3d;
  p.b3d = b3d;
  p.col_fastest = a.group == 0 && a.Mo >= a.No;  // A (Mo x Kc) is the larger operand: re-read B, not A
  p.c_bf16 = a.c_bf16;
  p.c_f32 = a.c_f32;
  p.status = L.d_status;
  p.wait_limit_ns = L.wait_limit_ns ? L.wait_limit_ns : 2000000000ull;
  p.stop_after_stages = L.stop_after_stages;
  const int64_t n_tiles = (a.No + BN - 1) / BN;
  const int64_t m_tiles = (a.Mo + TM - 1) / TM;
  if (grouped_rows)  // each expert adds at most one partial row tile
    return launch_majors<kGroupedRows, 1, 256>(L, tm, p, (a.Mo / TM + a.E) * n_tiles, false, a.b_mn_major);
  if (grouped_k) return launch_majors<kGroupedContraction, 1, 256>(L, tm, p, a.E * m_tiles * n_tiles, true, true);
  const int64_t tiles = m_tiles * n_tiles;
  if (MT == 2) return launch_majors<kDense, 2, 256>(L, tm, p, tiles, a.a_mn_major, a.b_mn_major);
  if (BN == 192) return launch_majors<kDense, 1, 192>(L, tm, p, tiles, a.a_mn_major, a.b_mn_major);
  return launch_majors<kDense, 1, 256>(L, tm, p, tiles, a.a_mn_major, a.b_mn_major);
}

}  // namespace qarl
