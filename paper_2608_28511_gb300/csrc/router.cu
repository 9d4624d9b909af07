// Router kernels: top-K with renormalised probabilities, and
// the router backward dz = p (dp - sum_k p_k dp_k) on the chosen set.
#include <math_constants.h>

#include "common.cuh"
#include "launch.h"
#include "select.cuh"

namespace moe {

// One warp or a few lanes per token (select.cuh): the K largest logits, ties to
// the lower expert index (reading R2), NaN as -inf, ordered by descending logit.
// The probabilities are exp(z_k - z_max) normalised over the K chosen logits,
// which equals the full softmax renormalised over the chosen set (reading R1).
template <int V, int G>
__global__ void __launch_bounds__(256) topk_kernel(const float* __restrict__ logits, int64_t T, int E, int K,
                                                   int32_t* __restrict__ idx, float* __restrict__ prob) {
  constexpr int TW = 32 / G, P = sel::kPerLane<V, G>;
  __shared__ uint2 slots[8][TW][kMaxK];
  const int warp = threadIdx.x >> 5, sub = (threadIdx.x & 31) / G, l = threadIdx.x % G;
  const int64_t t0 = ((int64_t)blockIdx.x * 8 + warp) * TW, t = t0 + sub;
  if (t0 >= T) return;  // the whole warp
  const float* row = logits + t * E;
  float z[V];
#pragma unroll
  for (int v = 0; v < V; ++v) z[v] = t < T && v * G + l < E ? __ldg(row + v * G + l) : 0.f;
  const uint2* slot = slots[warp][sub];
  sel::token_topk<V, G>(
      [&](int v) { return v * G + l < E ? sel::key_of(z[v]) : __uint_as_float(sel::kAbsent); }, E, K, l,
      slots[warp][sub]);
  const float best = __uint_as_float(slot[0].x);
  float w[P];
#pragma unroll
  for (int p = 0; p < P; ++p) w[p] = p * G + l < K ? expf(__uint_as_float(slot[p * G + l].x) - best) : 0.f;
  const float inv = 1.0f / sel::sum_chosen<P, G>(w, K);
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int k = p * G + l;
    if (k < K && t < T) {
      idx[t * K + k] = (int)(slot[k].y & 255u);
      prob[t * K + k] = w[p] * inv;
    }
  }
}

cudaError_t launch_topk(const Ctx& c, const float* logits, int64_t T, int E, int K, int32_t* idx, float* prob) {
  if (T == 0) return cudaSuccess;
  KernelScope ks("topk", c.stream);
  auto run = [&](auto v, auto g) {
    constexpr int G = decltype(g)::value, per = 8 * 32 / G;  // tokens per block
    topk_kernel<decltype(v)::value, G>
        <<<(unsigned)((T + per - 1) / per), 256, 0, c.stream>>>(logits, T, E, K, idx, prob);
  };
  // 17 to 32 experts: while the GPU holds all warps at once, the shorter chain of a
  // warp per token is faster (E = 32, warm, groups of eight lanes -> warps: T = 1024,
  // K = 4 2.2 -> 1.8 us, K = 8 2.7 -> 1.9; T = 16384, K = 4 3.5 -> 4.0)
  if (E > 16 && E <= 32 && T <= 4096) run(std::integral_constant<int, 1>(), std::integral_constant<int, 32>());
  else sel::for_experts(E, run);
  return cudaGetLastError();
}

// One warp per token: dz[t, e] = p_k (dp_k - c) if e = idx[t, k], else 0,
// with c = sum_k p_k dp_k.  Every entry of the row is written once.
__global__ void __launch_bounds__(256) route_dz_kernel(const int32_t* __restrict__ idx,
                                                       const float* __restrict__ prob,
                                                       const float* __restrict__ dprob, int64_t T, int E, int K,
                                                       float* __restrict__ dz, bf16* __restrict__ dz_bf16,
                                                       int64_t ld16) {
  const int lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= T) return;
  int my_e = -1;
  float my_p = 0.f, my_dp = 0.f;
  if (lane < K) {
    my_e = idx[t * K + lane];
    my_p = prob[t * K + lane];
    my_dp = dprob[t * K + lane];
  }
  float cdot = my_p * my_dp;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) cdot += __shfl_xor_sync(0xffffffffu, cdot, off);
  const float my_dz = my_p * (my_dp - cdot);
  for (int e0 = 0; e0 < E; e0 += 32) {
    const int e = e0 + lane;
    float val = 0.f;
    for (int k = 0; k < K; ++k) {
      const int ek = __shfl_sync(0xffffffffu, my_e, k);
      const float dk = __shfl_sync(0xffffffffu, my_dz, k);
      if (ek == e) val = dk;
    }
    if (e < E) {
      dz[t * E + e] = val;
      if (dz_bf16) dz_bf16[t * ld16 + e] = __float2bfloat16_rn(val);
    }
  }
}

cudaError_t launch_route_dz(const Ctx& c, const int32_t* idx, const float* prob, const float* dprob, int64_t T,
                            int E, int K, float* dz, void* dz_bf16, int64_t ld16) {
  if (T == 0) return cudaSuccess;
  const int warps = 8;
  dim3 grid((unsigned)((T + warps - 1) / warps)), block(32 * warps);
  KernelScope ks("route_dz", c.stream);
  route_dz_kernel<<<grid, block, 0, c.stream>>>(idx, prob, dprob, T, E, K, dz, (bf16*)dz_bf16,
                                                 ld16 > 0 ? ld16 : E);
  return cudaGetLastError();
}

// Deterministic reduction of split-K partial products: each output is the
// in-order sum of its S partials.
__global__ void __launch_bounds__(256) sum_splits_kernel(const float4* __restrict__ part, int S, int64_t n4,
                                                         float4* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    float4 a = __ldcs(part + i);
    for (int s = 1; s < S; ++s) {
      const float4 b = __ldcs(part + (int64_t)s * n4 + i);
      a.x += b.x;
      a.y += b.y;
      a.z += b.z;
      a.w += b.w;
    }
    out[i] = a;
  }
}

cudaError_t launch_sum_splits(const Ctx& c, const float* part, int S, int64_t n, float* out) {
  const int64_t n4 = n / 4;
  const int64_t want = (n4 + 255) / 256;
  const int blocks = (int)(want < (int64_t)c.num_sms * 8 ? want : (int64_t)c.num_sms * 8);
  KernelScope ks("sum_splits", c.stream);
  sum_splits_kernel<<<blocks, 256, 0, c.stream>>>((const float4*)part, S, n4, (float4*)out);
  return cudaGetLastError();
}

}  // namespace moe
