// TBPO sequence-level surrogate (Sec. 3.2; ratio and weight as written out in the appendix
// "Detail of TBPO") over B packed responses: for response i with tokens [off[i], off[i+1]) of the
// flat fp32 arrays,
//   a = mean_t (lp_cur - lp_old_learner),  r = exp(a);   b = mean_t (lp_old_learner - lp_old_sampler),  w = exp(b)
//   w~ = exp(clip(b, -log c, log c));  r~ = clip(r, 0, 1 + eps_h) if A >= 0 else clip(r, 1 - delta_l, 1 + delta_h)
//   J = w~ r~ A;   loss = -mean_i J;   d loss / d lp_cur[t] = -(w~ A r) / (L B) if r is inside its band, else 0.
// HBM-bound: 12 bytes read and 4 written per token.  Two launches:
//   partial  (warp per piece, all pieces at once: T / 2368 tokens, at least 512)  walks its piece in steps of 512
//                                   tokens with the next step's loads in flight; for every response that
//                                   overlaps the piece, the sums of the two token differences over the
//                                   overlap, in double, to slot (response + piece) -- unique, because both
//                                   indices only grow along the token axis.  No block barrier, whatever the lengths.
//   finish   (CTA per 1024 to 16384 tokens)  for every response that overlaps the chunk: its partials added (lane l takes
//                                   every 32nd, then a butterfly), r, w, J, flags and the gradient value its
//                                   tokens share, in double -- repeated by each chunk of a response, written out
//                                   by the chunk that holds its first token --, then the gradient streamed over
//                                   the chunk; the last CTA to finish adds all J in index order: loss = -mean J
// The response of a token is found by a 32-way search of the offsets.  Every sum has a fixed order: results do not
// depend on the grid or on timing.  1024 responses, 4.2 M tokens (67 MB) on the device: 31.7 us as four launches (response
// map, CTA per 8192 tokens with a block sum per response, statistics, gradient), 22.5 us so, of which 13.6 are the partial
// kernel (3.7 TB/s: ~4 us of its time is launch and first-load latency).
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace qarl {
namespace {

constexpr int kStep = 512;     // tokens a warp of the partial kernel takes at a time: 16 per lane
constexpr int kPieces = 2368;  // most pieces of a call: 16 warps on each of 148 SMs (a fixed number: the cut depends on T alone)
// Tokens per CTA of the finish kernel: the smallest power of two from kMinChunk that is half an average response or more and leaves the
// call kFinishCtas CTAs or fewer, at most kMaxChunk: calls over 592 x 16384 tokens have more CTAs, responses of over 32768 tokens on
// average more chunks each.  A CTA takes the responses of its chunk one after the other, so a call of few tokens in short responses wants short
// chunks (64 responses, 32,768 tokens: 22.4 us with 8192, 13.0 with 1024; 300 responses, 233,100 tokens: 21.4 and 12.9), while every
// chunk of a response repeats its statistics (64 responses, 393,216 tokens: 10.1 with 8192, 10.6 with 1024; 1024 responses, 4.2 M tokens:
// 22.2 with 8192, 25.9 with 4096; 2048 responses, 12.6 M: 51.9 with 8192, 49.6 with 16384).
constexpr int kMinChunk = 1024, kMaxChunk = 16384, kFinishCtas = 592;
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
  int64_t piece;         // tokens per piece
  int64_t chunk;         // tokens per CTA of the finish kernel
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

struct Step {
  float c[16], o[16], q[16];
};
// Loads of the step at token `base`; element e of a lane is token base + 4 lane + 128 (e / 4) + e % 4.
// VEC: the three arrays are 16-byte aligned.  They are read evict-first whatever their size: left in the L2, inputs that fit it cost
// a call on other inputs more (4.2 M tokens 24.0 -> 25.5 us) than they save one on the same (22.2 -> 20.2).
template <bool VEC>
__device__ __forceinline__ void load_step(const TbpoParams& p, Step& s, int64_t base, int64_t hi, int lane) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int64_t t = base + 4 * (32 * j + lane);
    if (VEC && t + 4 <= hi) {
      const float4 a = __ldcs(reinterpret_cast<const float4*>(p.lp_cur + t));
      const float4 b = __ldcs(reinterpret_cast<const float4*>(p.lp_old + t));
      const float4 d = __ldcs(reinterpret_cast<const float4*>(p.lp_smp + t));
      s.c[4 * j] = a.x, s.c[4 * j + 1] = a.y, s.c[4 * j + 2] = a.z, s.c[4 * j + 3] = a.w;
      s.o[4 * j] = b.x, s.o[4 * j + 1] = b.y, s.o[4 * j + 2] = b.z, s.o[4 * j + 3] = b.w;
      s.q[4 * j] = d.x, s.q[4 * j + 1] = d.y, s.q[4 * j + 2] = d.z, s.q[4 * j + 3] = d.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = t + u < hi;
        s.c[4 * j + u] = in ? __ldcs(p.lp_cur + t + u) : 0.0f;
        s.o[4 * j + u] = in ? __ldcs(p.lp_old + t + u) : 0.0f;
        s.q[4 * j + u] = in ? __ldcs(p.lp_smp + t + u) : 0.0f;
      }
    }
  }
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads, 2) tbpo_partial_kernel(const TbpoParams p) {
  pdl_wait();
  pdl_trigger();  // after the wait: the finish kernel may read the call's inputs before its own wait
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.ticket = 0;
  const int lane = threadIdx.x & 31;
  const int64_t k = static_cast<int64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5);
  const int64_t lo = k * p.piece, hi = min(lo + p.piece, p.T);
  if (lo >= p.T) return;
  Step s[2];
  load_step<VEC>(p, s[0], lo, hi, lane);
  int64_t i = response_of(p, lo, lane);
  int64_t t0 = clamp_off(p, i), t1 = clamp_off(p, i + 1);
  double2 acc = make_double2(0.0, 0.0);
  auto flush = [&]() {
    acc = warp_sum(acc);
    if (lane == 0) p.partial[i + k] = acc;
    acc = make_double2(0.0, 0.0);
  };
  auto consume = [&](const Step& s, int64_t base) -> bool {  // false: no response left
    const int64_t end = min(base + kStep, hi);
    for (;;) {
      if (t0 <= base && t1 >= base + kStep && end == base + kStep) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {  // differences formed in double: exact
          acc.x += static_cast<double>(s.c[e]) - static_cast<double>(s.o[e]);
          acc.y += static_cast<double>(s.o[e]) - static_cast<double>(s.q[e]);
        }
      } else {
        const int a0 = static_cast<int>(max(t0, base) - base) - 4 * lane;
        const int a1 = static_cast<int>(max(min(t1, end), base) - base) - 4 * lane;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int at = 128 * (e >> 2) + (e & 3);
          if (at >= a0 && at < a1) {
            acc.x += static_cast<double>(s.c[e]) - static_cast<double>(s.o[e]);
            acc.y += static_cast<double>(s.o[e]) - static_cast<double>(s.q[e]);
          }
        }
      }
      if (t1 > end) return true;  // goes on in the next step (or piece)
      if (t1 > max(t0, lo)) flush();
      if (++i >= p.B) return false;
      t0 = clamp_off(p, i);
      t1 = clamp_off(p, i + 1);
      if (t0 >= end) return true;
    }
  };
  bool more = true;
  for (int64_t base = lo; more && base < hi; base += 2 * kStep) {
    if (base + kStep < hi) load_step<VEC>(p, s[1], base + kStep, hi, lane);
    more = consume(s[0], base);
    if (more && base + kStep < hi) {
      if (base + 2 * kStep < hi) load_step<VEC>(p, s[0], base + 2 * kStep, hi, lane);
      more = consume(s[1], base + kStep);
    }
  }
  if (more && t0 < hi && t1 > hi) flush();
}

// Everything about response i (tokens [t0, t1), t1 > t0) from its two sums; returns the gradient value its tokens
// share, and writes the per-response outputs if `write`.
__device__ __forceinline__ float finish_response(const TbpoParams& p, int64_t i, int64_t t0, int64_t t1, double2 sum, float adv, bool write) {
  const double L = static_cast<double>(t1 - t0);
  const double a = sum.x / L, b = sum.y / L;
  const double r = exp(a);
  int f = 0;
  double bc = b;
  if (bc > p.log_cap) { bc = p.log_cap; f |= 2; }
  if (bc < -p.log_cap) { bc = -p.log_cap; f |= 2; }
  const double wt = exp(bc);
  const double A = static_cast<double>(adv);
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
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t lo = static_cast<int64_t>(blockIdx.x) * p.chunk, hi = min(lo + p.chunk, p.T);
  // Offsets and advantages are inputs of the call and the partial kernel started this one after its own wait: they may
  // be read ahead of this kernel's wait, while the last pieces are still being summed.
  int64_t first = 0;
  float adv = 0.0f;  // of response i0 + tid
  if (lo < hi) {
    first = response_of(p, lo, lane);
    for (int j = tid; j <= kThreads; j += kThreads) bound[j] = first + j <= p.B ? clamp_off(p, first + j) : p.T;
    if (first + tid < p.B) adv = __ldg(p.adv + first + tid);
  }
  pdl_wait();
  // empty responses: J = 0, still counted in B
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kThreads + tid; i < p.B; i += static_cast<int64_t>(gridDim.x) * kThreads)
    if (clamp_off(p, i + 1) <= clamp_off(p, i)) {
      p.r_seq[i] = 1.0;
      p.w_seq[i] = 1.0;
      p.j_seq[i] = 0.0;
      p.flags[i] = 4;
    }
  // Counted once the CTA's J are written: the last CTA to get here adds every J at its end, in one fixed order
  // (thread j takes j, j + 256, ...; then a tree): which CTA that is varies, what it computes does not.
  auto count = [&]() {
    __syncthreads();
    if (tid == 0) {
      __threadfence();  // after the barrier: covers what the CTA's threads wrote
      last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
    }
  };
  if (lo < hi) {
    // up to kThreads responses at a time
    for (int64_t i0 = first; i0 < p.B; i0 += kThreads) {
      if (i0 > first) {
        for (int j = tid; j <= kThreads; j += kThreads) bound[j] = i0 + j <= p.B ? clamp_off(p, i0 + j) : p.T;
        if (i0 + tid < p.B) adv = __ldg(p.adv + i0 + tid);
      }
      __syncthreads();
      for (int j = warp; j < kThreads && i0 + j < p.B && bound[j] < hi; j += kWarps) {
        const int64_t t0 = bound[j], t1 = bound[j + 1];
        if (t1 <= max(t0, lo)) continue;
        const bool small = p.T + p.piece < (int64_t(1) << 32);  // (a 64-bit division takes several times as long)
        const uint32_t d = static_cast<uint32_t>(p.piece);
        const int64_t k0 = small ? static_cast<uint32_t>(t0) / d : t0 / p.piece;
        const int64_t k1 = small ? static_cast<uint32_t>(t1 + p.piece - 1) / d : (t1 + p.piece - 1) / p.piece;
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
        gval[tid] = finish_response(p, i0 + tid, bound[tid], bound[tid + 1], sums[tid], adv, bound[tid] >= lo);
      const bool final = i0 + kThreads >= p.B || bound[kThreads] >= hi;  // no further round
      if (final) count();
      else __syncthreads();
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
      if (final) break;
      __syncthreads();
    }
  } else {
    count();
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
int64_t piece_of(int64_t T) { return std::max<int64_t>(kStep, ((T + kPieces - 1) / kPieces + 127) / 128 * 128); }
int64_t pieces_of(int64_t T) { return (T + piece_of(T) - 1) / piece_of(T); }
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
  p.piece = piece_of(a.T);
  p.chunk = kMinChunk;
  while (p.chunk < kMaxChunk && ((a.T + p.chunk - 1) / p.chunk > kFinishCtas || 2 * p.chunk * a.B < a.T)) p.chunk *= 2;
  p.partial = reinterpret_cast<double2*>(ws);
  p.ticket = reinterpret_cast<unsigned int*>(ws + ticket_at(a.B, a.T));
  if (a.B == 0) {  // no responses: the loss of an empty batch is 0
    ++*L.launches;
    return launch_pdl(tbpo_zero_loss_kernel, 1u, 1u, 0, L.stream, p);
  }
  const bool vec = ((reinterpret_cast<uintptr_t>(a.lp_cur) | reinterpret_cast<uintptr_t>(a.lp_old_learner) |
                     reinterpret_cast<uintptr_t>(a.lp_old_sampler)) & 15u) == 0;
  const unsigned partial_blocks = static_cast<unsigned>(std::max<int64_t>(1, (pieces_of(a.T) + kWarps - 1) / kWarps));
  const unsigned finish_blocks = static_cast<unsigned>(std::max<int64_t>(1, (a.T + p.chunk - 1) / p.chunk));
  *L.launches += 2;
  const cudaError_t e = launch_pdl(vec ? tbpo_partial_kernel<true> : tbpo_partial_kernel<false>, partial_blocks, kThreads, 0, L.stream, p);
  if (e != cudaSuccess) return e;
  return launch_pdl(tbpo_finish_kernel, finish_blocks, kThreads, 0, L.stream, p);
}

}  // namespace qarl
