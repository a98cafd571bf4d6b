// Router forward for up to a few thousand tokens: the one-launch router (router_fused_sm100.cu) with
// the experts of a 128-token tile split over the CTAs of a cluster.
//
// That kernel gives a token tile to one CTA: at M <= 2048 at most 16 of the 148 SMs work, and the call
// takes what one SM needs to walk the 128 x H x 128 tile and one thread needs to select a row -- 13.3 us
// at M = 1, 14.0 at M = 2048 (H = 2048, 128 experts, by graph replay; 8.2 and 12.7 here).  Here CTA c of a cluster computes the logits of experts
// [c NC, (c + 1) NC) with an MMA of N = NC columns (the same products in the same order per logit: the
// bits do not depend on N), every CTA sends the rows it does not own through distributed shared memory,
// and after one cluster barrier each CTA selects for its share of the rows, a warp per row.
//
// NC = 16 while the clusters (of 8 with 128 experts) fit the SMs at once, then 32: fewer columns per
// CTA mean a shorter walk, but each CTA re-reads the token tile (from L2), so a second round of clusters
// costs more than it saves.  More tokens than that go to the persistent kernel.
//
// Structure of a CTA (512 threads, one tile): warps 0-3 epilogue (thread = token row), warps 4 and 6
// TMA producers (per 64-element step a box of x, and a box of NC rows of W_r: for one token the walk is
// the time of issuing the loads), warp 5 MMA issuer; all 16 warps select.  Every barrier wait is bounded as in the other kernels; all threads reach the cluster
// barriers whatever happened before.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "router_select.cuh"

namespace qarl {
namespace {

using namespace ptx;

constexpr int RM = 128;   // tokens per tile (UMMA M)
constexpr int RN = 128;   // most experts
constexpr int RK = 64;    // contraction elements per stage: one 128-byte swizzle span of bf16
constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kTmaWarp = 4;
constexpr int kMmaWarp = 5;
constexpr int kTmaWarp2 = 6;
constexpr uint32_t kABytes = RM * RK * 2;
constexpr int kRowFloats = RN + 4;  // a gathered row, padded by one 16-byte chunk

constexpr int kMaxStages = 32;
constexpr size_t kSmemLimit = 227 * 1024;

struct Params {
  int M, H, E, k;
  int x_rows;  // rows of the x box: 128, or M rounded up to 8 when there is one tile.  The MMA then also multiplies what
               // lies behind the box (whole rows of zeros or of other stages): an output row depends on its own row only
  int stages;
  float* logits;
  int32_t* ids;
  float* wts;
  int* status;
  unsigned long long wait_limit_ns;
  int stop_after_stages;
};

struct __align__(8) Tail {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t done;
  uint64_t teardown;
  uint32_t tmem_addr;
  int abort_flag;
};

// rows a CTA gathers and selects for
__host__ __device__ constexpr int gather_rows(int cluster) { return (RM + cluster - 1) / cluster; }
__host__ __device__ constexpr uint32_t stage_bytes(int x_rows, int nc) { return static_cast<uint32_t>(x_rows + nc) * RK * 2; }

// shared memory besides the stages: alignment, the tail of the last token tile (see x_rows), gathered rows
size_t fixed_smem(int cluster) {
  return 1024 + kABytes + static_cast<size_t>(gather_rows(cluster)) * kRowFloats * 4 + sizeof(Tail);
}

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, Tail* s, const Params& p) {
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

template <int NC>
__global__ void __launch_bounds__(kThreads, 1)
router_cluster_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w, const Params p) {
  constexpr uint32_t kTmemCols = NC < 32 ? 32 : NC;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* gathered = reinterpret_cast<float*>(smem + static_cast<size_t>(p.stages) * stage_bytes(p.x_rows, NC) + kABytes);
  const int cluster = (p.E + NC - 1) / NC;
  Tail* s = reinterpret_cast<Tail*>(gathered + gather_rows(cluster) * kRowFloats);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int tile = blockIdx.x / cluster;
  const int KS = (p.H + RK - 1) / RK;  // a ragged last step reads zeros (TMA out-of-range fill)

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&s->full[i], 2);  // the two producers
      mbar_init(&s->empty[i], 1);
    }
    mbar_init(&s->done, 1);
    mbar_init(&s->teardown, 1);
    s->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kTmaWarp) {
    if (lane == 0) prefetch_tensormap(&tm_x);
    // the router's weights into L2 while the kernels before this one finish
    for (int ks = lane; ks < KS; ks += 32) tma_prefetch_2d(&tm_w, ks * RK, rank * NC);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&s->tmem_addr, kTmemCols);
    pdl_trigger();  // not before the allocation: see pdl_trigger
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  cluster_arrive();  // waited for before the first write into another CTA: by then it has started
  pdl_wait();
  const uint32_t tmem = s->tmem_addr;

  if (warp == kTmaWarp || warp == kTmaWarp2) {
    if (elect_one()) {
      const bool is_x = warp == kTmaWarp;
      const CUtensorMap* map = is_x ? &tm_x : &tm_w;
      const uint32_t bytes = stage_bytes(p.x_rows, NC), x_bytes = stage_bytes(p.x_rows, 0);
      const int y = is_x ? tile * RM : rank * NC;
      int stage = 0;
      uint32_t phase = 0, armed = 0, armed_parity = 0;
      bool ok = true;
      for (int ks = 0; ks < KS; ++ks) {
        if (p.stop_after_stages >= 0 && ks >= p.stop_after_stages) { ok = false; break; }
        if (!wait_or_abort(&s->empty[stage], phase ^ 1, s, p)) { ok = false; break; }
        uint8_t* dst = smem + static_cast<size_t>(stage) * bytes + (is_x ? 0 : x_bytes);
        mbar_arrive_expect_tx(&s->full[stage], is_x ? x_bytes : bytes - x_bytes);
        tma_load_2d(dst, map, &s->full[stage], ks * RK, y);
        armed |= 1u << stage;
        armed_parity = (armed_parity & ~(1u << stage)) | (phase << stage);
        if (++stage == p.stages) { stage = 0; phase ^= 1; }
      }
      if (!ok) {  // let copies in flight land before the CTA's shared memory is released
        for (int i = 0; i < p.stages; ++i)
          if (armed & (1u << i)) mbar_wait_bounded(&s->full[i], (armed_parity >> i) & 1u, 20000000ull);
      }
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    if (elect_one()) {
      const uint32_t bytes = stage_bytes(p.x_rows, NC);
      constexpr uint32_t idesc = umma_idesc_bf16_f32_major(RM, NC, false, false);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int ks = 0; ks < KS; ++ks) {
        if (!wait_or_abort(&s->full[stage], phase, s, p)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t a_addr = smem_u32(smem + static_cast<size_t>(stage) * bytes);
        const uint64_t a_desc = umma_desc_k_sw128(a_addr);
        const uint64_t b_desc = umma_desc_k_sw128(a_addr + p.x_rows * RK * 2);
#pragma unroll
        for (int k4 = 0; k4 < RK / 16; ++k4)  // 16 elements further on: 32 bytes = 2 in the 16-byte address field
          umma_bf16(tmem, a_desc + 2 * k4, b_desc + 2 * k4, idesc, (ks > 0 || k4 > 0) ? 1u : 0u);
        umma_commit(&s->empty[stage]);
        if (++stage == p.stages) { stage = 0; phase ^= 1; }
      }
      if (ok) {
        umma_commit(&s->done);
      } else {  // nothing of this CTA's tensor work may be in flight when its TMEM and shared memory go away
        umma_commit(&s->teardown);
        mbar_wait_bounded(&s->teardown, 0, 20000000ull);
      }
    }
    __syncwarp();
  }
  __syncwarp();
  if (warp >= 4) cluster_wait();
  if (warp < 4) {
    const bool ok = __all_sync(0xFFFFFFFFu, wait_or_abort(&s->done, 0, s, p) ? 1 : 0) != 0;
    cluster_wait();
    if (ok) {
      tc_fence_after_sync();
      uint32_t v[NC / 16][16];
#pragma unroll
      for (int c = 0; c < NC / 16; ++c) tmem_ld_x16(tmem + (static_cast<uint32_t>(warp * 32) << 16) + 16 * c, v[c]);
      tmem_ld_wait();
      const int r = warp * 32 + lane;
      const int64_t row = static_cast<int64_t>(tile) * RM + r;
      if (row < p.M) {
        // row r is selected by CTA r % cluster, as its row r / cluster
        const uint32_t to = map_to_cta(smem_u32(gathered + (r / cluster) * kRowFloats + rank * NC), r % cluster);
        float* out = p.logits + row * p.E + rank * NC;
#pragma unroll
        for (int c = 0; c < NC / 4; ++c) {
          const uint32_t* u = &v[c / 4][4 * (c % 4)];
          st_cluster_v4(to + 16 * c, u[0], u[1], u[2], u[3]);
          if (rank * NC + 4 * c < p.E) *reinterpret_cast<uint4*>(out + 4 * c) = make_uint4(u[0], u[1], u[2], u[3]);
        }
      }
      tc_fence_before_sync();
    }
  }
  __syncwarp();
  cluster_sync();  // the rows of this CTA are complete; nobody writes to another CTA any more
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
  }
  const int first = tile * RM;
  for (int i = warp; i * cluster + rank < RM; i += kWarps) {
    const int64_t row = first + i * cluster + rank;
    if (row >= p.M) break;
    float v[RN / 32];
#pragma unroll
    for (int j = 0; j < RN / 32; ++j) v[j] = lane + 32 * j < p.E ? gathered[i * kRowFloats + lane + 32 * j] : -INFINITY;
    select_topk<RN / 32>(v, p.E, p.k, lane, p.ids + row * p.k, p.wts + row * p.k);
  }
}

// Tensor map of a row-major bf16 matrix [rows, cols]: box of 64 columns x box_rows rows, 128-byte swizzle.
CUresult make_tmap(EncodeTiledFn encode, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {RK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

int tiles_of(int64_t M) { return static_cast<int>((M + RM - 1) / RM); }

// Sets the shared-memory limit of the kernel and returns how many clusters of this size run at once (they
// stay inside a GPC, so SMs are left over), 0 on failure.
template <int NC>
int resident_clusters(const Launch& L, int cluster) {
  static std::atomic<int> known[64][RN / NC + 1];  // value + 1; 0: not asked yet.  Set idempotently
  std::atomic<int>& slot = known[L.device & 63][cluster];
  const int have = slot.load(std::memory_order_acquire);
  if (have) return have - 1;
  int n = 0;
  if (cudaFuncSetAttribute(router_cluster_kernel<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmemLimit)) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(cluster));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, router_cluster_kernel<NC>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
  }
  slot.store(n + 1, std::memory_order_release);
  return n;
}

// Columns per CTA: the fewest for which the clusters of all token tiles run at once, 0 if none.
int pick_nc(const Launch& L, int64_t M, int64_t E) {
  if (tiles_of(M) <= resident_clusters<16>(L, static_cast<int>((E + 15) / 16))) return 16;
  if (tiles_of(M) <= resident_clusters<32>(L, static_cast<int>((E + 31) / 32))) return 32;
  return 0;
}

template <int NC>
cudaError_t launch(const Launch& L, const CUtensorMap& tx, const CUtensorMap& tw, Params p) {
  const int cluster = (p.E + NC - 1) / NC;
  const size_t fixed = fixed_smem(cluster), per = stage_bytes(p.x_rows, NC);
  p.stages = static_cast<int>(std::min<size_t>({kMaxStages, static_cast<size_t>((p.H + RK - 1) / RK), (kSmemLimit - fixed) / per}));
  ++*L.launches;
  return launch_pdl_cluster(router_cluster_kernel<NC>, static_cast<unsigned>(tiles_of(p.M) * cluster),
                            static_cast<unsigned>(cluster), kThreads, fixed + p.stages * per, L.stream, tx, tw, p);
}

}  // namespace

bool router_cluster_applies(const Launch& L, int64_t M, int64_t E) { return E <= RN && pick_nc(L, M, E) != 0; }

cudaError_t launch_router_cluster(const Launch& L, EncodeTiledFn encode, const uint16_t* x, int64_t M, int64_t H,
                                  const uint16_t* wr, int64_t E, int64_t k, float* logits, int32_t* ids, float* wts,
                                  CUresult* cu_err) {
  *cu_err = CUDA_SUCCESS;
  const int nc = pick_nc(L, M, E);
  Params p{};
  p.M = static_cast<int>(M);
  p.H = static_cast<int>(H);
  p.E = static_cast<int>(E);
  p.k = static_cast<int>(k);
  p.x_rows = static_cast<int>(std::min<int64_t>(RM, (M + 7) / 8 * 8));
  p.logits = logits;
  p.ids = ids;
  p.wts = wts;
  p.status = L.d_status;
  p.wait_limit_ns = L.wait_limit_ns ? L.wait_limit_ns : 2000000000ull;
  p.stop_after_stages = L.stop_after_stages;
  CUtensorMap tx, tw;
  CUresult r = make_tmap(encode, &tx, x, static_cast<uint64_t>(M), static_cast<uint64_t>(H), static_cast<uint32_t>(p.x_rows));
  if (r == CUDA_SUCCESS) r = make_tmap(encode, &tw, wr, static_cast<uint64_t>(E), static_cast<uint64_t>(H), static_cast<uint32_t>(nc));
  if (r != CUDA_SUCCESS) {
    *cu_err = r;
    return cudaErrorUnknown;
  }
  return nc == 16 ? launch<16>(L, tx, tw, p) : launch<32>(L, tx, tw, p);
}

}  // namespace qarl
