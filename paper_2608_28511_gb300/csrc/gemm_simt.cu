// CUDA-core grouped GEMM (fp32 FMA, no TF32): the all-fp32 path and the
// reference engine for every GemmDesc shape the tensor-core engine handles.
//
// C(m, n) = sum_k A(m, k) B(n, k) with arbitrary element strides, grouped
// along M (per-expert row ranges), along K (per-expert or equal reduction
// ranges) or dense, plus the router / SwiGLU epilogues, and the row gathers of
// GemmDesc.  256 threads per BM x BN tile in a 16 x 16 arrangement; a thread
// owns BM / 16 rows (in groups of up to 4, 64 apart) and BN / 16 columns (the
// same), so that in a 128-column tile a packed gate column and its up column
// (64 apart) land in the same thread.
//
// Both operands are staged in shared memory as [k][m] and [k][n], two buffers:
// the next k-tile's global loads are issued before the current one is
// multiplied and written to the other buffer after it, one barrier per k-tile.
// The products are packed fp32 FMAs on two adjacent columns (fma.rn.f32x2, each
// half rounded as a scalar FMA), in the order of k.  The SwiGLU backward is an
// epilogue of dA's product: 174 us at T = 3001 for 160 and 18.6 as a pass of its
// own.
//
// Bound by the FMA pipe and its issue slots.  Measured on an fp32 layer of
// T = 3001, D = 512, E = 12, K = 3, F = 768: GEMM-1 (14.2 GFLOP) 526 us on the
// single-buffered 64 x 128 x 16 tiles used before, 358 us with scalar FMAs here,
// 304 us with packed ones (47 TFLOP/s; 92 % of the tile rows real).  A k-tile of
// 8 (363 us) or 32 (336 us, spills), one block per SM with more registers
// (365 us), and in the 32 x 32 tile k split over four groups of threads, are
// slower.
#include "common.cuh"
#include "launch.h"

namespace moe {

namespace {

template <typename T>
__device__ __forceinline__ float ldf(const T* p) {
  return to_f32<T>(__ldg(p));
}
// Four consecutive elements (16-byte aligned fp32, 8-byte aligned bf16).
__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 ld4(const bf16* p) {
  const uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(bf16* p, const float* v) {
  uint2 w;
  w.x = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[0])) |
        ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[1])) << 16);
  w.y = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[2])) |
        ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[3])) << 16);
  *reinterpret_cast<uint2*>(p) = w;
}

__device__ __forceinline__ float silu_f(float v) { return v / (1.0f + __expf(-v)); }

// One operand tile, ROWS (m or n) x BK, staged as s[k * ROWS + (row ^ swz(k))].
// swz spreads the scalar stores of a k-contiguous operand (4 k values of one
// row per thread, 32 / (BK / 4) rows and all BK / 4 k-chunks per warp) over
// all 32 banks; it is a multiple of 4, so 4-row vectors stay whole.
template <int BK>
__device__ __forceinline__ constexpr int swz(int k) {
  return ((k >> 2) % (BK / 4)) * (32 / (BK / 4));
}

template <typename T, int ROWS, int BK>
struct Loader {
  static constexpr int NV = ROWS * BK / 4 / 256;  // 4-element vectors per thread
  static_assert(NV >= 1 && ROWS * BK == NV * 1024, "whole vectors per thread");
  const T* p;            // the operand, advanced to this tile's group
  int64_t s_r, s_k;      // element strides of the row and of k
  int64_t r0, r_end;     // the tile's first row and the end of its rows
  const int32_t* gat_r;  // row indirection of the rows / of k (or NULL)
  const int32_t* gat_k;
  bool kfast;            // s_k == 1: vectors along k; else along the rows
  bool vec;              // vectors may be read whole (alignment)
  // the fast path: this thread's vectors of the next whole k-tile, each either
  // inside the operand or (bit clear) past its rows
  const T* ptr[NV];
  uint32_t in;
  bool fast;

  __device__ __forceinline__ int row_of(int j) const {
    const int i = (int)threadIdx.x + j * 256;
    return kfast ? i / (BK / 4) : (i % (ROWS / 4)) * 4;
  }
  __device__ __forceinline__ int k_of(int j) const {
    const int i = (int)threadIdx.x + j * 256;
    return kfast ? (i % (BK / 4)) * 4 : i / (ROWS / 4);
  }
  __device__ __forceinline__ void init(const T* base, int64_t sr, int64_t sk, int64_t row0, int64_t row_end,
                                       int64_t kbeg, const int32_t* gr, const int32_t* gk) {
    p = base;
    s_r = sr;
    s_k = sk;
    r0 = row0;
    r_end = row_end;
    gat_r = gr;
    gat_k = gk;
    kfast = sk == 1;
    // whole vectors start at a multiple of 4 along the unit-stride dimension
    const int64_t pitch = kfast ? sr : sk, origin = kfast ? kbeg : row0;
    vec = (kfast || sr == 1) && pitch % 4 == 0 && origin % 4 == 0 &&
          (reinterpret_cast<uintptr_t>(base) & (4 * sizeof(T) - 1)) == 0;
    fast = vec && !gr && !gk;
    in = 0;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int64_t r = row0 + row_of(j);
      ptr[j] = base + r * sr + (kbeg + k_of(j)) * sk;
      if (r < row_end) in |= 1u << j;
      if (!kfast && r < row_end && r + 4 > row_end) fast = false;  // a vector across the last row
    }
  }
  // The k-tile [k0, k0 + BK) cut at kend; called for consecutive k-tiles.
  __device__ __forceinline__ void load(int64_t k0, int64_t kend, float (&v)[NV][4]) {
    if (fast && k0 + BK <= kend) {
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in >> j & 1u) q = ld4(ptr[j]);
        ptr[j] += (int64_t)BK * s_k;
        v[j][0] = q.x; v[j][1] = q.y; v[j][2] = q.z; v[j][3] = q.w;
      }
      return;
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int64_t r = r0 + row_of(j), k = k0 + k_of(j);
#pragma unroll
      for (int u = 0; u < 4; ++u) v[j][u] = 0.f;
      if (r >= r_end || k >= kend) continue;
      if (kfast) {
        const T* row = p + (gat_r ? (int64_t)__ldg(gat_r + r) : r) * s_r;
        if (vec && !gat_k && k + 4 <= kend) {
          const float4 q = ld4(row + k);
          v[j][0] = q.x; v[j][1] = q.y; v[j][2] = q.z; v[j][3] = q.w;
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (k + u < kend) v[j][u] = ldf<T>(row + (gat_k ? (int64_t)__ldg(gat_k + k + u) : k + u));
        }
      } else {
        const T* col = p + (gat_k ? (int64_t)__ldg(gat_k + k) : k) * s_k;
        if (vec && !gat_r && r + 4 <= r_end) {
          const float4 q = ld4(col + r);
          v[j][0] = q.x; v[j][1] = q.y; v[j][2] = q.z; v[j][3] = q.w;
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (r + u < r_end) v[j][u] = ldf<T>(col + (gat_r ? (int64_t)__ldg(gat_r + r + u) : r + u) * s_r);
        }
      }
    }
  }
  __device__ __forceinline__ void store(float* s, const float (&v)[NV][4]) const {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int r = row_of(j), k = k_of(j);
      const int rs = r ^ swz<BK>(k);  // k .. k + 3 of a k-contiguous vector share it
      if (kfast) {
#pragma unroll
        for (int u = 0; u < 4; ++u) s[(k + u) * ROWS + rs] = v[j][u];
      } else {
        *reinterpret_cast<float4*>(s + k * ROWS + rs) = make_float4(v[j][0], v[j][1], v[j][2], v[j][3]);
      }
    }
  }
};

// A thread's N = TILE / 16 positions of one tile dimension: t in 0 .. 15.
template <int N>
__device__ __forceinline__ int pos(int t, int i) {
  return N >= 4 ? (i >> 2) * 64 + t * 4 + (i & 3) : t * N + i;
}
template <int N>
__device__ __forceinline__ void frag(const float* row, int t, int sw, float (&f)[N]) {
  if (N >= 4) {
#pragma unroll
    for (int g = 0; g < N / 4; ++g) {
      const float4 q = *reinterpret_cast<const float4*>(row + ((g * 64 + t * 4) ^ sw));
      f[4 * g] = q.x; f[4 * g + 1] = q.y; f[4 * g + 2] = q.z; f[4 * g + 3] = q.w;
    }
  } else {
    const float2 q = *reinterpret_cast<const float2*>(row + ((t * 2) ^ sw));
    f[0] = q.x; f[1] = q.y;
  }
}

// The problems of one launch: problem i's blocks start at first[i], tiles[i] of
// them per group of a Group::K problem.
template <int NP>
struct Problems {
  GemmDesc d[NP];
  unsigned first[NP];
  unsigned tiles[NP];
};

template <typename TA, typename TB, typename TC, int BM, int BN, int BK, int NP>
__global__ void __launch_bounds__(256, BM * BN >= 8192 ? 2 : 3)
    simt_gemm_kernel(const __grid_constant__ Problems<NP> ps) {
  int pi = 0;
#pragma unroll
  for (int i = 1; i < NP; ++i)
    if (blockIdx.x >= ps.first[i]) pi = i;
  const GemmDesc& d = ps.d[pi];
  const unsigned block = blockIdx.x - ps.first[pi];
  constexpr int TM = BM / 16, TN = BN / 16;
  extern __shared__ __align__(16) float smem[];  // two A tiles, then two B tiles
  auto As = [&](int b) { return smem + b * BK * BM; };
  auto Bs = [&](int b) { return smem + 2 * BK * BM + b * BK * BN; };
  __shared__ int s_wsum[8];
  __shared__ int s_g;
  __shared__ int s_row0, s_rend;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const unsigned tiles_n = (unsigned)((d.N + BN - 1) / BN);
  const unsigned tile = d.group == Group::K ? block % ps.tiles[pi] : block;
  const int mt = (int)(tile / tiles_n);  // a row tile's column tiles are consecutive blocks
  const int64_t n0 = (int64_t)(tile % tiles_n) * BN;

  int g = 0;
  int64_t row0 = (int64_t)mt * BM, row_end = d.M, kbeg = 0, kend = d.K;
  if (d.group == Group::M) {
    // the expert whose tiles include this one: thread e counts expert e's
    // tiles, an exclusive scan over the (at most 256) experts places them
    const int lane = tid & 31, warp = tid >> 5;
    int lo = 0, hi = 0;
    if (tid < d.num_groups) {
      lo = __ldg(d.offsets + tid);
      hi = __ldg(d.offsets + tid + 1);
    }
    const int nt = (hi - lo + BM - 1) / BM;
    int inc = nt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s_wsum[warp] = inc;
    if (tid == 0) s_g = -1;
    __syncthreads();
    int base = 0;
    for (int w = 0; w < warp; ++w) base += s_wsum[w];
    const int first = base + inc - nt;
    if (mt >= first && mt < first + nt) {
      s_g = tid;
      s_row0 = lo + (mt - first) * BM;
      s_rend = hi;
    }
    __syncthreads();
    g = s_g;
    if (g < 0) return;
    row0 = s_row0;
    row_end = s_rend;
  } else if (d.group == Group::K) {
    g = (int)(block / ps.tiles[pi]);
    if (d.offsets) {
      kbeg = d.offsets[g];
      kend = d.offsets[g + 1];
    } else {
      kbeg = d.split_rows * g / d.num_groups;
      kend = d.split_rows * (g + 1) / d.num_groups;
    }
  }
  if (row0 >= row_end || n0 >= d.N) return;

  Loader<TA, BM, BK> la;
  Loader<TB, BN, BK> lb;
  la.init(static_cast<const TA*>(d.A), d.sa_m, d.sa_k, row0, row_end, kbeg,
          d.group == Group::M ? d.gather : nullptr, nullptr);
  lb.init(static_cast<const TB*>(d.B) + (int64_t)g * d.sb_g, d.sb_n, d.sb_k, n0, d.N, kbeg,
          nullptr, d.group == Group::K ? d.gather : nullptr);

  unsigned long long acc2[TM][TN / 2];  // two adjacent columns per 64-bit pair
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc2[i][j] = 0ull;

  float va[Loader<TA, BM, BK>::NV][4], vb[Loader<TB, BN, BK>::NV][4];
  la.load(kbeg, kend, va);
  lb.load(kbeg, kend, vb);
  la.store(As(0), va);
  lb.store(Bs(0), vb);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
    const bool more = k0 + BK < kend;
    if (more) {
      la.load(k0 + BK, kend, va);
      lb.load(k0 + BK, kend, vb);
    }
    const float* as = As(buf);
    const float* bs = Bs(buf);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
      frag<TM>(as + k * BM, ty, swz<BK>(k), a);
      frag<TN>(bs + k * BN, tx, swz<BK>(k), b);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        unsigned long long aa;
        asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a[i]));
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
          unsigned long long bb;
          asm("mov.b64 %0, {%1, %2};" : "=l"(bb) : "f"(b[2 * j]), "f"(b[2 * j + 1]));
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[i][j]) : "l"(aa), "l"(bb));
        }
      }
    }
    if (more) {
      la.store(As(buf ^ 1), va);
      lb.store(Bs(buf ^ 1), vb);
      __syncthreads();
      buf ^= 1;
    }
  }

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[i][2 * j]), "=f"(acc[i][2 * j + 1]) : "l"(acc2[i][j]));
  TC* C = static_cast<TC*>(d.C) + (d.group == Group::K ? (int64_t)g * d.sc_g : 0);
  const bool vec_c = d.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C) & (4 * sizeof(TC) - 1)) == 0;
  constexpr int CG = TN >= 4 ? 4 : TN;  // consecutive columns of a thread
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t gm = row0 + pos<TM>(ty, i);
    if (gm >= row_end) continue;
    TC* crow = C + gm * d.ldc;
#pragma unroll
    for (int j0 = 0; j0 < TN; j0 += CG) {
      const int64_t gn = n0 + pos<TN>(tx, j0);
      if (gn >= d.N) continue;
      const bool whole = CG == 4 && vec_c && gn + 4 <= d.N;
      float v[CG];
#pragma unroll
      for (int u = 0; u < CG; ++u) {
        v[u] = acc[i][j0 + u];
        if (d.epi == Epi::StoreBias && d.bias && gn + u < d.N) v[u] += d.bias[gn + u];
        if (d.epi == Epi::Accum && gn + u < d.N) v[u] = to_f32<TC>(crow[gn + u]) + v[u];
      }
      if (d.epi == Epi::SwigluBwd) {
        // dA at columns gn ..: the gate block of h / dH at 128 (gn / 64) + gn mod 64,
        // the up block 64 further (N is a multiple of 64)
        const int64_t o = gm * d.ldc + (gn >> 6) * 128 + (gn & 63);
        const TC* h = static_cast<const TC*>(d.aux) + o;
        float dg[CG], du[CG];
#pragma unroll
        for (int u = 0; u < CG; ++u) {
          const float gate = to_f32<TC>(__ldg(h + u)), up = to_f32<TC>(__ldg(h + 64 + u));
          const float sg = __frcp_rn(1.0f + __expf(-gate));
          dg[u] = v[u] * up * sg * (1.0f + gate * (1.0f - sg));
          du[u] = v[u] * gate * sg;
        }
        if constexpr (CG == 4) {
          st4(C + o, dg);
          st4(C + o + 64, du);
        } else {
#pragma unroll
          for (int u = 0; u < CG; ++u) {
            C[o + u] = from_f32<TC>(dg[u]);
            C[o + 64 + u] = from_f32<TC>(du[u]);
          }
        }
        continue;
      }
      if (whole) {
        if constexpr (CG == 4) st4(crow + gn, v);
      } else {
#pragma unroll
        for (int u = 0; u < CG; ++u)
          if (gn + u < d.N) crow[gn + u] = from_f32<TC>(v[u]);
      }
      if (d.epi == Epi::ReluSqFwd) {
#pragma unroll
        for (int u = 0; u < CG; ++u) {
          const float r = fmaxf(v[u], 0.f);
          if (gn + u < d.N) static_cast<TC*>(d.aux)[gm * d.ldc + gn + u] = from_f32<TC>(r * r);
        }
      }
      if constexpr (TN == 8) {
        // gate at tile columns c < 64, up at c + 64 (the same thread, index + 4)
        if (d.epi == Epi::SwigluFwd && j0 == 0) {
          TC* arow = static_cast<TC*>(d.aux) + gm * (d.N / 2) + n0 / 2 + tx * 4;
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = silu_f(v[u]) * acc[i][4 + u];
          st4(arow, v);  // N is a multiple of 128: aligned
        }
      }
    }
  }
}

template <typename TA, typename TB, typename TC, int BM, int BN, int BK, int NP>
cudaError_t run_tile(const Ctx& c, const GemmDesc (&ds)[NP]) {
  Problems<NP> ps;
  int64_t blocks = 0;
  for (int i = 0; i < NP; ++i) {
    const GemmDesc& d = ds[i];
    const int64_t tiles_n = (d.N + BN - 1) / BN;
    const int64_t tiles_m =
        d.group == Group::M ? (d.max_rows + BM - 1) / BM + d.num_groups : (d.M + BM - 1) / BM;
    const int64_t tiles = tiles_m * tiles_n;
    const int groups = d.group == Group::K ? d.num_groups : 1;
    if (tiles <= 0 || groups <= 0) return NP == 1 ? cudaSuccess : cudaErrorInvalidValue;
    ps.d[i] = d;
    ps.first[i] = (unsigned)blocks;
    ps.tiles[i] = (unsigned)tiles;
    blocks += tiles * groups;
    if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;
  }
  constexpr int kSmem = 2 * (BM + BN) * BK * 4;
  static_assert(kSmem <= 48 * 1024, "fits without opting in to more shared memory");
  simt_gemm_kernel<TA, TB, TC, BM, BN, BK, NP><<<(unsigned)blocks, 256, kSmem, c.stream>>>(ps);
  return cudaGetLastError();
}

// Tiles of a BM x BN tiling that hold rows (an upper estimate for Group::M,
// whose experts' row counts only the device knows).
template <int NP>
int64_t tiles_of(const GemmDesc (&ds)[NP], int bm, int bn) {
  int64_t sum = 0;
  for (const GemmDesc& d : ds) {
    const int64_t nt = (d.N + bn - 1) / bn;
    if (d.group == Group::M) {
      const int64_t groups = d.max_rows < d.num_groups ? d.max_rows : d.num_groups;
      sum += nt * (d.max_rows / bm + (groups + 1) / 2);
    } else {
      sum += nt * ((d.M + bm - 1) / bm) * (d.group == Group::K ? d.num_groups : 1);
    }
  }
  return sum;
}

template <typename TA, typename TB, typename TC, int NP>
cudaError_t run(const Ctx& c, const GemmDesc (&ds)[NP]) {
  const bool swiglu = ds[0].epi == Epi::SwigluFwd;  // needs gate and up columns in one 128-column tile
  int64_t widest = 0;
  for (const GemmDesc& d : ds) widest = d.N > widest ? d.N : widest;
  // a split reduction onto at most 32 rows (router_splits_simt sizes the splits for
  // this tile): a taller tile is half empty.  fp32, E = 12, Din = 1024, T = 4096 35.0
  // us on 64 x 64 tiles, 31.5 here; Din = 2048 53 and 45
  if (NP == 1 && ds[0].group == Group::K && ds[0].M <= 32) return run_tile<TA, TB, TC, 32, 32, 32>(c, ds);
  if constexpr (sizeof(TA) == 4 && sizeof(TB) == 4) {
    // the largest tile that still gives every SM work: at T = 256, D = 128, E = 8,
    // K = 2, F = 256 the small tiles take GEMM-1's dgrad from 102 to 17 us
    if (widest > 64) {
      if (tiles_of(ds, 128, 128) >= c.num_sms) return run_tile<TA, TB, TC, 128, 128, 16>(c, ds);
      if (tiles_of(ds, 64, 128) >= c.num_sms) return run_tile<TA, TB, TC, 64, 128, 16>(c, ds);
      if (swiglu) return run_tile<TA, TB, TC, 32, 128, 32>(c, ds);
    }
    // (three problems of unequal length: several blocks per SM, or the longest is
    // left alone; the same case on 64 x 64 tiles 29 us, on 32 x 32 18)
    if (tiles_of(ds, 64, 64) >= NP * c.num_sms && widest > 32) return run_tile<TA, TB, TC, 64, 64, 32>(c, ds);
    return run_tile<TA, TB, TC, 32, 32, 32>(c, ds);
  } else {
    if (swiglu || (widest > 64 && tiles_of(ds, 64, 128) >= c.num_sms))
      return run_tile<TA, TB, TC, 64, 128, 16>(c, ds);
    return run_tile<TA, TB, TC, 32, 32, 32>(c, ds);
  }
}

}  // namespace

cudaError_t launch_gemm_simt(const Ctx& c, const GemmDesc& d, const char* name) {
  KernelScope ks(name, c.stream);
  const GemmDesc ds[1] = {d};
  const int key = (int)d.a_type * 4 + (int)d.b_type * 2 + (int)d.c_type;
  switch (key) {
    case 0: return run<bf16, bf16, bf16>(c, ds);
    case 1: return run<bf16, bf16, float>(c, ds);
    case 2 + 0: return run<bf16, float, bf16>(c, ds);
    case 4 + 0: return run<float, bf16, bf16>(c, ds);
    case 4 + 1: return run<float, bf16, float>(c, ds);
    case 4 + 2 + 1: return run<float, float, float>(c, ds);
    default: return cudaErrorNotSupported;
  }
}

cudaError_t launch_gemm_simt_f32x3(const Ctx& c, const GemmDesc (&ds)[3], const char* name) {
  KernelScope ks(name, c.stream);
  return run<float, float, float>(c, ds);
}

}  // namespace moe
