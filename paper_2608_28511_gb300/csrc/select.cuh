// Top-K selection over the E experts of each token, shared by the softmax
// router (keys = logits) and the sigmoid router (keys = sigmoid scores + expert
// bias).  One warp per token: lane l holds experts l, l + 32, ... as a short
// list sorted in registers; each of the K rounds takes the largest list head
// with one warp reduction (redux.sync.max.f32), and the lane whose head it is
// records it and drops it.
//
// Rounds assume that all chosen keys differ, and the end checks it: one head
// taken per round, no two taken keys equal, none left equal to the last one.
// Otherwise the token is chosen again by rounds that resolve equal keys to the
// lower expert.  -0 ties with +0 and NaN keys count as -inf.
//
// Bound by the compare / select pipe, then by the chain of K reductions.  At
// T = 30011, E = 128, K = 8 the top-K kernel takes 14.3 us; four threads per
// token with sorted insertion lists took 29.7, rounds that track each owner's
// expert by vote and shuffle 18.3.
#pragma once

#include <math_constants.h>

#include "common.cuh"

namespace moe {
namespace sel {

// The key that is compared for a value; NaN marks an absent expert.
__device__ __forceinline__ float key_of(float v) { return fmaxf(v, -CUDART_INF_F) + 0.f; }
constexpr uint32_t kAbsent = 0x7fffffffu;

// The largest value of the warp that is not NaN.
__device__ __forceinline__ float warp_max(float v) {
  float m;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
  return m;
}

// Lists of 32 experts that E takes, and a bound on K, as compile-time sizes.
inline int lists_of(int E) { return E <= 32 ? 1 : E <= 64 ? 2 : E <= 128 ? 4 : 8; }

// Comparators that sort V keys (Batcher's odd-even merge sort).
template <int V>
__device__ __forceinline__ void sort_lists(float (&key)[V], uint32_t (&id)[V]) {
#pragma unroll
  for (int p = 1; p < V; p <<= 1) {
#pragma unroll
    for (int k = p; k >= 1; k >>= 1) {
#pragma unroll
      for (int j = k % p; j + k < V; j += 2 * k) {
#pragma unroll
        for (int i = 0; i < k; ++i) {
          if (i + j + k < V && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
            const bool up = key[i + j + k] > key[i + j];  // false if either is absent: those stay last
            const float a = key[i + j], b = key[i + j + k];
            const uint32_t ia = id[i + j], ib = id[i + j + k];
            key[i + j] = up ? b : a;
            key[i + j + k] = up ? a : b;
            id[i + j] = up ? ib : ia;
            id[i + j + k] = up ? ia : ib;
          }
        }
      }
    }
  }
}

// The rounds for keys that may be equal: ties go to the lower expert.
template <int V>
__device__ __noinline__ uint2 topk_with_ties(const float* row, int E, int K, int lane) {
  // row: the warp's keys in shared or global memory, expert by expert
  float key[V];
#pragma unroll
  for (int v = 0; v < V; ++v)
    key[v] = v * 32 + lane < E ? key_of(row[v * 32 + lane]) : __uint_as_float(kAbsent);
  uint2 r = make_uint2(0u, 0u);
  for (int k = 0; k < K; ++k) {
    float h = key[0];
    unsigned he = (unsigned)lane;
#pragma unroll
    for (int v = 1; v < V; ++v) {
      if (key[v] > h || h != h) {  // strictly larger: the lower expert keeps a tie
        h = key[v];
        he = (unsigned)(v * 32 + lane);
      }
    }
    const float m = warp_max(h);
    const unsigned e = __reduce_min_sync(0xffffffffu, h == m ? he : 0xffffffffu);
    if (lane == k) r = make_uint2(__float_as_uint(m), e);
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (e == (unsigned)(v * 32 + lane)) key[v] = __uint_as_float(kAbsent);
  }
  return r;
}

// The K <= 16 best of a token's E keys: key[v] = key_of(expert 32 v + lane's),
// absent where there is none.  slot: 16 entries of shared memory of this warp's
// own; row(): the same keys in memory (read only where keys are equal).  Lane
// k < K returns the k-th best's key and expert, the other lanes 0 and 0; *best
// is the best key, in every lane.  The whole warp calls.
template <int V, typename Row>
__device__ __forceinline__ void warp_topk(float (&key)[V], int E, int K, int lane, uint2* slot, Row row,
                                          float* my_key, int* my_e, float* best) {
  const float absent = __uint_as_float(kAbsent);
  uint32_t id[V];
#pragma unroll
  for (int v = 0; v < V; ++v) id[v] = (uint32_t)(v * 32 + lane);
  sort_lists<V>(key, id);
  // the list's experts, a byte each, first to last: dropping the head is a shift
  uint32_t lo = 0, hi = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (v < 4) lo |= id[v] << (8 * v);
    else hi |= id[v] << (8 * (v - 4));
  }
  int taken = 0;
  float m = 0.f;
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    m = warp_max(key[0]);
    if (key[0] == m) {
      slot[k] = make_uint2(__float_as_uint(m), lo);
      ++taken;
#pragma unroll
      for (int v = 0; v + 1 < V; ++v) key[v] = key[v + 1];
      key[V - 1] = absent;
      if (V > 4) {
        lo = __funnelshift_r(lo, hi, 8);
        hi >>= 8;
      } else {
        lo >>= 8;
      }
    }
  }
  __syncwarp();
  uint2 r = make_uint2(0u, 0u);
  if (lane < K) r = slot[lane];
  r.y &= 255u;
  const float mine = __uint_as_float(r.x), next = __shfl_down_sync(0xffffffffu, mine, 1);
  // m is NaN if the keys ran out, which takes an earlier round that took several
  const bool tie = key[0] == m || m != m || (lane + 1 < K && mine == next);
  if (__reduce_add_sync(0xffffffffu, (unsigned)taken) != (unsigned)K || __any_sync(0xffffffffu, tie))
    r = topk_with_ties<V>(row(), E, K, lane);
  *my_key = __uint_as_float(r.x);
  *my_e = (int)r.y;
  *best = __shfl_sync(0xffffffffu, *my_key, 0);
  __syncwarp();  // the slots are read before the next token's rounds write them
}

// The sum of the values of lanes 0 .. K - 1, added in that order (best expert
// first), in every lane: a probability is a function of its chosen keys alone,
// not of how the lanes are paired.
__device__ __forceinline__ float sum_chosen(float v, int K) {
  float s = 0.f;
#pragma unroll 4
  for (int k = 0; k < K; ++k) s += __shfl_sync(0xffffffffu, v, k);
  return s;
}

}  // namespace sel
}  // namespace moe
