// Top-K selection over the E experts of each token, shared by the softmax
// router (keys = logits) and the sigmoid router (keys = sigmoid scores + expert
// bias).  More than 32 experts: one warp per token; lane l holds experts l,
// l + 32, ... as a short list sorted in registers; each of the K rounds takes the
// largest list head with one warp reduction (redux.sync.max.f32), and the lane
// whose head it is records it and drops it.  Up to 32 experts: four or eight
// lanes per token (below).
//
// Rounds assume that all chosen keys differ.  The first one shows whether the
// best key is in several lanes, and the end checks the rest: one head taken per
// round, no two taken keys equal, none left equal to the last one.  Otherwise the
// token is chosen again by rounds that take every key equal to the largest one
// left, in the order of the experts.  -0 ties with +0 and NaN keys count as -inf.
//
// Bound by the compare / select pipe, then by the chain of K reductions.  At
// T = 30011, E = 128, K = 8 the top-K kernel takes 14.3 us; four threads per
// token with sorted insertion lists took 29.7, rounds that track each owner's
// expert by vote and shuffle 18.3.  Equal keys (logits of a router that starts at
// zero, scores that saturate), T = 16384, E = 256, K = 8, inputs in L2: all equal
// 8.9 us, one equal pair 15.2, none 9.2; with all K rounds first and then rounds
// that take one key each 20.5, 20.5 and 9.3.
#pragma once

#include <math_constants.h>

#include <type_traits>

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

// Runs f with the lists per lane (V) and lanes per token (G) for E experts.
template <typename F>
inline void for_experts(int E, F f) {
  if (E <= 4) f(std::integral_constant<int, 1>(), std::integral_constant<int, 4>());
  else if (E <= 8) f(std::integral_constant<int, 1>(), std::integral_constant<int, 8>());
  else if (E <= 16) f(std::integral_constant<int, 2>(), std::integral_constant<int, 8>());
  else if (E <= 32) f(std::integral_constant<int, 4>(), std::integral_constant<int, 8>());
  else if (E <= 64) f(std::integral_constant<int, 2>(), std::integral_constant<int, 32>());
  else if (E <= 128) f(std::integral_constant<int, 4>(), std::integral_constant<int, 32>());
  else f(std::integral_constant<int, 8>(), std::integral_constant<int, 32>());
}

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

// The K <= 16 best of a token's E keys: lane l holds the keys of experts l,
// l + 32, ..., keys(v) being key_of(expert 32 v + l's), absent where there is
// none (called again where keys are equal).  slot: 16 entries of shared memory of
// this warp's own, of which 0 .. K - 1 receive the best ones' keys and (in the low
// byte) experts, best first.  The whole warp calls, and calls __syncwarp() between
// reading the slots and the next token.
template <int V, typename Keys>
__device__ __forceinline__ void warp_topk(Keys keys, int K, int lane, uint2* slot) {
  const float absent = __uint_as_float(kAbsent);
  float key[V];
  uint32_t id[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    key[v] = keys(v);
    id[v] = (uint32_t)(v * 32 + lane);
  }
  sort_lists<V>(key, id);
  // the list's experts, a byte each, first to last: dropping the head is a shift
  uint32_t lo = 0, hi = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (v < 4) lo |= id[v] << (8 * v);
    else hi |= id[v] << (8 * (v - 4));
  }
  float m = warp_max(key[0]);
  const unsigned heads = __ballot_sync(0xffffffffu, key[0] == m);
  bool ties = (heads & (heads - 1u)) != 0u;
  if (!ties) {
    int taken = 0;
#pragma unroll 2
    for (int k = 0;;) {
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
      if (++k == K) break;
      m = warp_max(key[0]);
    }
    __syncwarp();
    const float mine = lane < K ? __uint_as_float(slot[lane].x) : 0.f;
    const float next = __shfl_down_sync(0xffffffffu, mine, 1);
    // m is NaN if the keys ran out, which takes an earlier round that took several
    const bool tie = key[0] == m || m != m || (lane + 1 < K && mine == next);
    ties = __reduce_add_sync(0xffffffffu, (unsigned)taken) != (unsigned)K || __any_sync(0xffffffffu, tie);
  }
  if (ties) {
    // keys that may be equal: each round takes every key that equals the largest
    // one left, in the order of the experts, so equal keys cost one round together
#pragma unroll
    for (int v = 0; v < V; ++v) key[v] = keys(v);
    __syncwarp();
    int got = 0;
    for (int k = 0; k < K && got < K; ++k) {
      float h = key[0];
#pragma unroll
      for (int v = 1; v < V; ++v) h = fmaxf(h, key[v]);
      m = warp_max(h);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const bool eq = key[v] == m;
        const unsigned b = __ballot_sync(0xffffffffu, eq);
        if (eq) {
          const int at = got + __popc(b & ((1u << lane) - 1u));
          if (at < K) slot[at] = make_uint2(__float_as_uint(m), (unsigned)(v * 32 + lane));
          key[v] = absent;
        }
        got += __popc(b);
      }
    }
    __syncwarp();
  }
}

// Tokens of up to 32 experts: G lanes each (32 / G tokens at once), lane l of a
// group holding experts l, l + G, ...  A warp per token leaves lanes without an
// expert and costs the same for 8 experts as for 32; T = 16384, K = 2, inputs in L2:
// E = 8 3.7 -> 2.1 us, 16 3.7 -> 2.6, 32 3.7 -> 2.8 (four threads per token with
// sorted lists 2.4, 2.7, 3.4); T = 65536, E = 8 10.3 -> 3.9.
//
// group_ranks: every lane counts the keys that come before each of its own, and
// the chosen ones go to their places; the cost does not depend on K.
template <int V, int G, typename Keys>
__device__ __forceinline__ void group_ranks(Keys keys, int E, int K, int l, uint2* slot) {
  float key[V];
  int rank[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    key[v] = keys(v);
    rank[v] = 0;
  }
#pragma unroll
  for (int u = 0; u < V; ++u) {
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const float kj = __shfl_sync(0xffffffffu, key[u], j, G);
#pragma unroll
      for (int v = 0; v < V; ++v)  // false for an absent kj
        if (u < v ? kj >= key[v] : kj > key[v] || (u == v && kj == key[v] && j < l)) ++rank[v];
    }
  }
#pragma unroll
  for (int v = 0; v < V; ++v)
    if (v * G + l < E && rank[v] < K) slot[rank[v]] = make_uint2(__float_as_uint(key[v]), (unsigned)(v * G + l));
  __syncwarp();
}

// group_rounds: K rounds, each the group's best key (the lower expert of equal
// ones) by shuffles.  For lists of four it is cheaper than counting up to K = 6
// (T = 16384, E = 32: K = 2 2.8 us against 4.2, K = 4 3.5 against 4.2, K = 8 5.0
// against 4.3), for lists of two up to K = 2.
template <int V, int G, typename Keys>
__device__ __forceinline__ void group_rounds(Keys keys, int K, int l, uint2* slot) {
  float key[V];
#pragma unroll
  for (int v = 0; v < V; ++v) key[v] = keys(v);
  for (int k = 0; k < K; ++k) {
    float m = key[0];
    int e = l;
#pragma unroll
    for (int v = 1; v < V; ++v) {
      if (key[v] > m || m != m) {  // strictly larger: the lower expert keeps a tie
        m = key[v];
        e = v * G + l;
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, m, o);
      const int oe = __shfl_xor_sync(0xffffffffu, e, o);
      if (om > m || m != m || (om == m && oe < e)) {
        m = om;
        e = oe;
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (e == v * G + l) {
        slot[k] = make_uint2(__float_as_uint(m), (unsigned)e);
        key[v] = __uint_as_float(kAbsent);
      }
    }
  }
  __syncwarp();
}

template <int V, int G, typename Keys>
__device__ __forceinline__ void token_topk(Keys keys, int E, int K, int l, uint2* slot) {
  if constexpr (G == 32) {
    warp_topk<V>(keys, K, l, slot);
  } else {
    if (V == 4 ? K <= 6 : V == 2 && K <= 2) group_rounds<V, G>(keys, K, l, slot);
    else group_ranks<V, G>(keys, E, K, l, slot);
  }
}

// Chosen experts per lane of a group: lane l has the k-th for k = l, l + G, ...
template <int V, int G>
constexpr int kPerLane = V * G <= G || G >= kMaxK ? 1 : (kMaxK + G - 1) / G;

// The sum of a group's K chosen terms, w[p] of lane l being the (p G + l)-th's (0
// from the K-th on), in that order (best expert first), in every lane: a
// probability is a function of its chosen keys alone, not of how the lanes are
// paired.  The shuffles of a size are in flight together; a loop to K takes them
// one by one (8192 sequences of one token, E = 64, K = 6 90 us, now 77).
template <int N, int P, int G>
__device__ __forceinline__ float sum_first(const float (&w)[P]) {
  float u[N];
#pragma unroll
  for (int k = 0; k < N; ++k) u[k] = __shfl_sync(0xffffffffu, w[k / G], k % G, G);
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < N; ++k) s += u[k];
  return s;
}
template <int P, int G>
__device__ __forceinline__ float sum_chosen(const float (&w)[P], int K) {
  constexpr int N = P * G < kMaxK ? P * G : kMaxK;  // K is at most this
  if (N <= 4 || K <= 4) return sum_first<(N < 4 ? N : 4), P, G>(w);
  if (N <= 8 || K <= 8) return sum_first<(N < 8 ? N : 8), P, G>(w);
  return sum_first<N, P, G>(w);
}

}  // namespace sel
}  // namespace moe
