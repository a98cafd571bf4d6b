// TBPO sequence-level surrogate (Sec. 3.2; ratio and weight as written out in the appendix
// "Detail of TBPO") over B packed responses: for response i with tokens [off[i], off[i+1]) of the
// flat fp32 arrays,
//   a = mean_t (lp_cur - lp_old_learner),  r = exp(a);   b = mean_t (lp_old_learner - lp_old_sampler),  w = exp(b)
//   w~ = exp(clip(b, -log c, log c));  r~ = clip(r, 0, 1 + eps_h) if A >= 0 else clip(r, 1 - delta_l, 1 + delta_h)
//   J = w~ r~ A;   loss = -mean_i J;   d loss / d lp_cur[t] = -(w~ A r) / (L B) if r is inside its band, else 0.
// HBM-bound: 12 bytes read and 4 written per token.  Two launches:
//   partial  (warp per 512 tokens)  the 12 loads of a lane are issued before anything else; for every response that
//                                   overlaps the piece, the sums of the two token differences over the
//                                   overlap, in double, to slot (response + piece) -- unique, because both
//                                   indices only grow along the token axis.  No block barrier, whatever the lengths.
//   finish   (CTA per 4096 tokens)  for every response that overlaps the chunk: its partials added (lane l takes
//                                   every 32nd, then a butterfly), r, w, J, flags and the gradient value its
//                                   tokens share, in double -- repeated by each chunk of a response, written out
//                                   by the chunk that holds its first token --, then the gradient streamed over
//                                   the chunk; the last CTA to finish adds all J in index order: loss = -mean J
// The response of a token is found by a 32-way search of the offsets.  Every sum has a fixed order: results do not
// depend on the grid or on timing.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace qarl {
namespace {

constexpr int kPiece = 512;    // tokens per warp of the partial kernel: 16 per lane
constexpr int kChunk = 4096;   // tokens per CTA of the finish kernel
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

struct TbpoParams {
  const float* lp_cur;
  const float* lp_old;
  const float* lp_smp;
  const int64_t* off;
  const float* adv;
  int64_t B, T;
  double eps_h, delta_l, delta_h, log_cap;
  double* r_seq;
  double* w_seq;
  double* j_seq;
  int32_t* flags;
  float* grad;
  double* loss;
  double2* partial;      // [B + pieces]
  unsigned int* ticket;  // CTAs of the finish kernel that are done
};

__device__ __forceinline__ int64_t clamp_off(const TbpoParams& p, int64_t i) {
  return min(max(p.off[i], int64_t(0)), p.T);
}

// The response that holds token t (whole warp; B >= 1): the last i with off[i] <= t.  Malformed offsets give some
// index in [0, B - 1], never an out-of-range access.
__device__ __forceinline__ int64_t response_of(const TbpoParams& p, int64_t t, int lane) {
  int64_t at = 0, n = p.B;
  while (n > 1) {
    const int64_t step = (n + 31) / 32;
    const bool below = lane * step < n && __ldg(p.off + at + lane * step) <= t;
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, below);
    const int c = max(__popc(m) - 1, 0);
    at += c * step;
    n = min(step, n - c * step);
  }
  return at;
}

__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xFFFFFFFFu, v.x, o);
    v.y += __shfl_xor_sync(0xFFFFFFFFu, v.y, o);
  }
  return v;
}

// VEC: the three arrays are 16-byte aligned
template <bool VEC>
__global__ void __launch_bounds__(kThreads) tbpo_partial_kernel(const TbpoParams p) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.ticket = 0;
  const int lane = threadIdx.x & 31;
  const int64_t k = static_cast<int64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  const int64_t lo = k * kPiece, hi = min(lo + kPiece, p.T);
  if (lo >= p.T) return;
  // token of this lane's element (j, u): lo + 4 (32 j + lane) + u
  float c[16], o[16], q[16];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int64_t t = lo + 4 * (32 * j + lane);
    if (VEC && t + 4 <= hi) {
      const float4 a = __ldcs(reinterpret_cast<const float4*>(p.lp_cur + t));
      const float4 b = __ldcs(reinterpret_cast<const float4*>(p.lp_old + t));
      const float4 d = __ldcs(reinterpret_cast<const float4*>(p.lp_smp + t));
      c[4 * j] = a.x, c[4 * j + 1] = a.y, c[4 * j + 2] = a.z, c[4 * j + 3] = a.w;
      o[4 * j] = b.x, o[4 * j + 1] = b.y, o[4 * j + 2] = b.z, o[4 * j + 3] = b.w;
      q[4 * j] = d.x, q[4 * j + 1] = d.y, q[4 * j + 2] = d.z, q[4 * j + 3] = d.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = t + u < hi;
        c[4 * j + u] = in ? __ldcs(p.lp_cur + t + u) : 0.0f;
        o[4 * j + u] = in ? __ldcs(p.lp_old + t + u) : 0.0f;
        q[4 * j + u] = in ? __ldcs(p.lp_smp + t + u) : 0.0f;
      }
    }
  }
  for (int64_t i = response_of(p, lo, lane); i < p.B; ++i) {
    const int64_t t0 = clamp_off(p, i);
    if (t0 >= hi) break;
    const int64_t s0 = max(t0, lo), s1 = min(clamp_off(p, i + 1), hi);
    if (s1 <= s0) continue;
    double2 acc = make_double2(0.0, 0.0);
    if (s0 == lo && s1 == lo + kPiece) {
#pragma unroll
      for (int e = 0; e < 16; ++e) {  // differences formed in double: exact
        acc.x += static_cast<double>(c[e]) - static_cast<double>(o[e]);
        acc.y += static_cast<double>(o[e]) - static_cast<double>(q[e]);
      }
    } else {
      const int a0 = static_cast<int>(s0 - lo) - 4 * lane, a1 = static_cast<int>(s1 - lo) - 4 * lane;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const int at = 128 * (e >> 2) + (e & 3);
        if (at >= a0 && at < a1) {
          acc.x += static_cast<double>(c[e]) - static_cast<double>(o[e]);
          acc.y += static_cast<double>(o[e]) - static_cast<double>(q[e]);
        }
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) p.partial[i + k] = acc;
  }
}

// Everything about response i (tokens [t0, t1), t1 > t0) from its two sums; returns the gradient value its tokens
// share, and writes the per-response outputs if `write`.
__device__ __forceinline__ float finish_response(const TbpoParams& p, int64_t i, int64_t t0, int64_t t1, double2 sum, bool write) {
  const double L = static_cast<double>(t1 - t0);
  const double a = sum.x / L, b = sum.y / L;
  const double r = exp(a);
  int f = 0;
  double bc = b;
  if (bc > p.log_cap) { bc = p.log_cap; f |= 2; }
  if (bc < -p.log_cap) { bc = -p.log_cap; f |= 2; }
  const double wt = exp(bc);
  const double A = static_cast<double>(__ldg(p.adv + i));
  const double band_lo = A >= 0.0 ? 0.0 : 1.0 - p.delta_l;
  const double band_hi = A >= 0.0 ? 1.0 + p.eps_h : 1.0 + p.delta_h;
  double rt = r;
  if (rt < band_lo) { rt = band_lo; f |= 1; }
  if (rt > band_hi) { rt = band_hi; f |= 1; }
  if (write) {
    p.r_seq[i] = r;
    p.w_seq[i] = (f & 2) ? exp(b) : wt;
    p.j_seq[i] = wt * rt * A;
    p.flags[i] = f;
  }
  return (f & 1) ? 0.0f : static_cast<float>(-(wt * A * r) / (L * static_cast<double>(p.B)));
}

__global__ void __launch_bounds__(kThreads) tbpo_finish_kernel(const TbpoParams p) {
  __shared__ double part[kThreads];
  __shared__ double2 sums[kThreads];
  __shared__ float gval[kThreads];
  __shared__ int64_t bound[kThreads + 1];  // clamped offsets of the responses in hand
  __shared__ bool last;
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t lo = static_cast<int64_t>(blockIdx.x) * kChunk, hi = min(lo + kChunk, p.T);
  // empty responses: J = 0, still counted in B
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kThreads + tid; i < p.B; i += static_cast<int64_t>(gridDim.x) * kThreads)
    if (clamp_off(p, i + 1) <= clamp_off(p, i)) {
      p.r_seq[i] = 1.0;
      p.w_seq[i] = 1.0;
      p.j_seq[i] = 0.0;
      p.flags[i] = 4;
    }
  if (lo < hi) {
    // up to kThreads responses at a time
    for (int64_t i0 = response_of(p, lo, lane); i0 < p.B; i0 += kThreads) {
      for (int j = tid; j <= kThreads; j += kThreads) bound[j] = i0 + j <= p.B ? clamp_off(p, i0 + j) : p.T;
      __syncthreads();
      if (bound[0] >= hi) break;  // (the same for every thread)
      for (int j = warp; j < kThreads && i0 + j < p.B && bound[j] < hi; j += kWarps) {
        const int64_t t0 = bound[j], t1 = bound[j + 1];
        if (t1 <= max(t0, lo)) continue;
        const int64_t k0 = t0 / kPiece, k1 = (t1 + kPiece - 1) / kPiece;
        double2 s = make_double2(0.0, 0.0);
        for (int64_t kk = k0 + lane; kk < k1; kk += 32) {
          const double2 v = p.partial[i0 + j + kk];
          s.x += v.x;
          s.y += v.y;
        }
        s = warp_sum(s);
        if (lane == 0) sums[j] = s;
      }
      __syncthreads();
      if (i0 + tid < p.B && bound[tid] < hi && bound[tid + 1] > max(bound[tid], lo))
        gval[tid] = finish_response(p, i0 + tid, bound[tid], bound[tid + 1], sums[tid], bound[tid] >= lo);
      __syncthreads();
      if (p.grad) {
        const bool vec = (reinterpret_cast<uintptr_t>(p.grad) & 15u) == 0;
        for (int j = 0; j < kThreads && i0 + j < p.B && bound[j] < hi; ++j) {
          const int64_t s0 = max(bound[j], lo), s1 = min(bound[j + 1], hi);
          if (s1 <= s0) continue;
          const float g = gval[j];
          const int64_t v0 = vec ? min((s0 + 3) & ~int64_t(3), s1) : s1, v1 = vec ? max(s1 & ~int64_t(3), v0) : s1;
          for (int64_t t = s0 + tid; t < v0; t += kThreads) p.grad[t] = g;
          for (int64_t t = v0 + 4 * tid; t < v1; t += 4 * kThreads) *reinterpret_cast<float4*>(p.grad + t) = make_float4(g, g, g, g);
          for (int64_t t = v1 + tid; t < s1; t += kThreads) p.grad[t] = g;
        }
      }
      if (bound[kThreads] >= hi) break;
      __syncthreads();
    }
  }
  // The last CTA to get here adds every J in one fixed order (thread j takes j, j + 256, ...; then a
  // tree): which CTA that is varies, what it computes does not.
  __syncthreads();
  if (tid == 0) {
    __threadfence();  // after the barrier: covers what the CTA's threads wrote
    last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0;
  for (int64_t j = tid; j < p.B; j += kThreads) s += __ldcg(p.j_seq + j);
  part[tid] = s;
  __syncthreads();
  for (int o = kThreads / 2; o > 0; o >>= 1) {
    if (tid < o) part[tid] += part[tid + o];
    __syncthreads();
  }
  if (tid == 0) *p.loss = -part[0] / static_cast<double>(p.B);
}

__global__ void tbpo_zero_loss_kernel(const TbpoParams p) {
  pdl_trigger();
  pdl_wait();
  *p.loss = 0.0;
}

}  // namespace

namespace {
int64_t pieces_of(int64_t T) { return (T + kPiece - 1) / kPiece; }
size_t ticket_at(int64_t B, int64_t T) { return (static_cast<size_t>(B + pieces_of(T)) * sizeof(double2) + 255) / 256 * 256; }
}  // namespace

size_t tbpo_workspace_bytes(int64_t B, int64_t T) { return ticket_at(B, T) + 256; }

cudaError_t launch_tbpo(const Launch& L, const TbpoArgs& a) {
  TbpoParams p{};
  p.lp_cur = a.lp_cur;
  p.lp_old = a.lp_old_learner;
  p.lp_smp = a.lp_old_sampler;
  p.off = a.offsets;
  p.adv = a.adv;
  p.B = a.B;
  p.T = a.T;
  p.eps_h = a.eps_h;
  p.delta_l = a.delta_l;
  p.delta_h = a.delta_h;
  p.log_cap = log(a.cap);
  p.r_seq = a.r_seq;
  p.w_seq = a.w_seq;
  p.j_seq = a.j_seq;
  p.flags = a.flags;
  p.grad = a.grad;
  p.loss = a.loss;
  uint8_t* ws = static_cast<uint8_t*>(a.workspace);
  p.partial = reinterpret_cast<double2*>(ws);
  p.ticket = reinterpret_cast<unsigned int*>(ws + ticket_at(a.B, a.T));
  if (a.B == 0) {  // no responses: the loss of an empty batch is 0
    ++*L.launches;
    return launch_pdl(tbpo_zero_loss_kernel, 1u, 1u, 0, L.stream, p);
  }
  const bool vec = ((reinterpret_cast<uintptr_t>(a.lp_cur) | reinterpret_cast<uintptr_t>(a.lp_old_learner) |
                     reinterpret_cast<uintptr_t>(a.lp_old_sampler)) & 15u) == 0;
  const unsigned partial_blocks = static_cast<unsigned>(std::max<int64_t>(1, (pieces_of(a.T) + kWarps - 1) / kWarps));
  const unsigned finish_blocks = static_cast<unsigned>(std::max<int64_t>(1, (a.T + kChunk - 1) / kChunk));
  *L.launches += 2;
  const cudaError_t e = launch_pdl(vec ? tbpo_partial_kernel<true> : tbpo_partial_kernel<false>, partial_blocks, kThreads, 0, L.stream, p);
  if (e != cudaSuccess) return e;
  return launch_pdl(tbpo_finish_kernel, finish_blocks, kThreads, 0, L.stream, p);
}

}  // namespace qarl
