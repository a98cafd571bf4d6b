// Router of the MoE block: top-k experts of every token from its fp32 logits (ties to the lower
// expert id, descending order) and the softmax over the selected logits.  One warp per token; lane l
// keeps experts l, l + 32, ... in registers; k rounds of a warp arg-max.  The logits come from the
// bf16 tensor-core GEMM (x . W_r^T, fp32 accumulation in a fixed order), so a token's routing
// depends only on that token's row -- the same invariance the expert GEMMs have (App. C).
#include "router_select.cuh"

namespace qarl {
namespace {

// PER = experts per lane (E <= 32 PER).
template <int PER>
__global__ void __launch_bounds__(256) router_topk_kernel(const float* __restrict__ logits, int64_t M, int E, int k,
                                                          int32_t* __restrict__ ids, float* __restrict__ wts) {
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t m = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  if (m >= M) return;
  const float* row = logits + m * E;
  float v[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = lane + 32 * j;
    v[j] = e < E ? row[e] : -INFINITY;
  }
  select_topk<PER>(v, E, k, lane, ids + m * k, wts + m * k);
}

}  // namespace

cudaError_t launch_router_topk(const Launch& L, const float* logits, int64_t M, int64_t E, int64_t k, int32_t* ids,
                               float* wts) {
  if (M == 0) return cudaSuccess;
  ++*L.launches;
  const unsigned grid = static_cast<unsigned>((M * 32 + 255) / 256);
  const int Ei = static_cast<int>(E), ki = static_cast<int>(k);
  const int per = static_cast<int>((E + 31) / 32);
  if (per <= 1) return launch_pdl(router_topk_kernel<1>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
  if (per <= 2) return launch_pdl(router_topk_kernel<2>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
  if (per <= 4) return launch_pdl(router_topk_kernel<4>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
  if (per <= 8) return launch_pdl(router_topk_kernel<8>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
  if (per <= 16) return launch_pdl(router_topk_kernel<16>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
  return launch_pdl(router_topk_kernel<32>, grid, 256, 0, L.stream, logits, M, Ei, ki, ids, wts);
}

}  // namespace qarl
