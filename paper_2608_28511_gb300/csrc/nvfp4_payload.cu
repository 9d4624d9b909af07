// NVFP4 dispatch payload (Sec. 1, the precision lever b_x of Eq. 1; Sec. 6
// names FP8 and NVFP4): every dispatched row travels as E2M1 codes (two per
// byte, element 2j in the low nibble of byte j), one E4M3 scale per block of
// 16 elements and one power-of-two scale g per row:
//   g   = the smallest 2^e (e >= -126) with max |x| <= 6 * 448 * g;
//   s_b = E4M3 nearest to max_{i in b} |x_i| / (6 g)   (fp32 ratio);
//   q_i = E2M1 nearest to x_i / (s_b g)                (fp32 ratio);
// both roundings to nearest, ties to even, saturating.  The receiver's
// q * s_b * g is exact in bf16.
#include <cuda_fp4.h>
#include <cuda_fp8.h>
#include <math_constants.h>

#include <type_traits>

#include "common.cuh"
#include "launch.h"

namespace moe {

namespace {

constexpr int kBlk = 16;  // elements per block scale

// Exponent of the row scale for a row maximum amax (finite, >= 0): the
// smallest e with amax <= 6 * 448 * 2^e, where 6 * 448 = 2688 is
// 0.65625 * 2^12.
__device__ __forceinline__ int nvfp4_row_exp(float amax) {
  if (!(amax > 0.f)) return 0;
  int k;
  const float m = frexpf(amax, &k);  // amax = m 2^k, m in [0.5, 1)
  const int e = k - 12 + (m > 0.65625f ? 1 : 0);
  return e < -126 ? -126 : e;
}

__device__ __forceinline__ float e4m3_to_float(uint8_t c) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)c, __NV_E4M3);
  return __half2float(*reinterpret_cast<const __half*>(&h));
}

// E2M1 code pairs of f / den, rounded to nearest even, 8 bytes: quot(v) is the
// quotient for one element.
template <typename Q>
__device__ __forceinline__ uint2 e2m1_codes(const float (&f)[kBlk], Q quot) {
  uint32_t w[2] = {0u, 0u};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = 8 * h + 2 * j;
      const __nv_fp4x2_storage_t b =
          __nv_cvt_float2_to_fp4x2(make_float2(quot(f[i]), quot(f[i + 1])), __NV_E2M1, cudaRoundNearest);
      w[h] |= (uint32_t)b << (8 * j);
    }
  }
  return make_uint2(w[0], w[1]);
}

// One 16-element block (two 16-byte vectors of bf16) -> its E4M3 scale code
// and 8 bytes of E2M1 codes.  The quotients v / den, den = s_b g, were what bound
// the dispatch as one fp32 division per element.  They are taken as
// v rh + v rl with rh + rl = 1 / den to about 2^-47: the fused sum rounds a value
// within 2^-47 of v / den, so a quotient that is an E2M1 midpoint (a few bits,
// exact in fp32) comes out exactly, and any other differs from every midpoint by
// more than 2^-12 of it (v has 8 significant bits, midpoint times den at most 7):
// the codes are those of the exact quotient.  T = 8191, K = 6, D = 2048: 23.7 ->
// 19.3 us.  rl has to be a normal number, so a den outside 2^-100 .. 2^100 takes
// the division, and so does a block with an infinity (inf rh + inf rl is NaN for
// rl <= 0).  The sign is v's: -0 rh + -0 rl is +0 for rl < 0.
__device__ __forceinline__ void quantize_block(const uint4& v0, const uint4& v1, float six_g, float g,
                                               uint8_t* scode, uint2* codes) {
  float f[kBlk];
  unpack16<bf16>(v0, f);
  unpack16<bf16>(v1, f + 8);
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < kBlk; ++i) amax = fmaxf(amax, fabsf(f[i]));
  const __nv_fp8_storage_t sc = __nv_cvt_float_to_fp8(amax / six_g, __NV_SATFINITE, __NV_E4M3);
  *scode = (uint8_t)sc;
  const float sb = e4m3_to_float((uint8_t)sc);
  uint2 w = make_uint2(0u, 0u);
  if (sb > 0.f) {
    const float den = sb * g;  // exact: an E4M3 value times a power of two
    if (den >= 0x1p-100f && den <= 0x1p100f && amax < CUDART_INF_F) {
      const float rh = 1.0f / den;
      const float rl = fmaf(-rh, den, 1.0f) * rh;
      w = e2m1_codes(f, [&](float v) { return copysignf(fmaf(v, rh, v * rl), v); });
    } else {
      w = e2m1_codes(f, [&](float v) { return v / den; });
    }
  }
  *codes = w;
}

// One warp per token: the row maximum and scale, then every block's scale and
// codes, written to each of the token's K rows (row_of_slot).  NB > 0: a lane's
// (at most NB) blocks are read once, into registers; wider rows are read twice.
// T = 8191, K = 6, D = 2048, dispatch and arrival: 69.8 -> 67.8 us.  NB is no larger
// than the row needs, since the unused blocks cost their share of the code (with
// the permutation, warm, T = 8191, K = 6: D = 256 read twice 15.9 us, NB = 4 18.1,
// NB = 1 14.2; D = 1024 18.5, 20.7, NB = 2 18.0).
template <int KM, int NB>
__global__ void __launch_bounds__(256) dispatch_nvfp4_kernel(const uint4* __restrict__ x,
                                                             const int32_t* __restrict__ row_of_slot, int64_t T,
                                                             int K, int vpr, uint2* __restrict__ xq,
                                                             uint8_t* __restrict__ bscale, float* __restrict__ rscale,
                                                             uint32_t* err) {
  const int lane = threadIdx.x & 31;
  const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= T) return;
  const uint4* row = x + t * vpr;
  const int nblk = vpr / 2;  // 16-element blocks per row
  float amax = 0.f;
  uint4 raw[NB > 0 ? 2 * NB : 1];
  if (NB > 0) {
    // the lane's NB blocks stay in registers, all loads in flight at once
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int b = lane + 32 * j;
      raw[2 * j] = b < nblk ? ld_stream(row + 2 * b) : make_uint4(0, 0, 0, 0);
      raw[2 * j + 1] = b < nblk ? ld_stream(row + 2 * b + 1) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < 2 * NB; ++j) {
      float f[8];
      unpack16<bf16>(raw[j], f);
#pragma unroll
      for (int u = 0; u < 8; ++u) amax = fmaxf(amax, fabsf(f[u]));
    }
  } else {
    for (int i = lane; i < vpr; i += 32) {
      float f[8];
      unpack16<bf16>(__ldg(row + i), f);
#pragma unroll
      for (int j = 0; j < 8; ++j) amax = fmaxf(amax, fabsf(f[j]));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  const int e = nvfp4_row_exp(amax);
  const float g = ldexpf(1.0f, e);
  const float six_g = 6.0f * g;  // exact
  int64_t dst[KM];
#pragma unroll
  for (int k = 0; k < KM; ++k) {
    dst[k] = k < K ? (int64_t)__ldg(row_of_slot + t * K + k) : -1;
    if (dst[k] >= T * K) {  // a row outside [0, TK): recorded and skipped
      set_error(err, kErrIndex);
      dst[k] = -1;
    }
  }
  if (lane < K) {
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k == lane && dst[k] >= 0) rscale[dst[k]] = g;
  }
  auto put = [&](int b, const uint4& v0, const uint4& v1) {
    uint8_t sc;
    uint2 q;
    quantize_block(v0, v1, six_g, g, &sc, &q);
#pragma unroll
    for (int k = 0; k < KM; ++k) {
      if (dst[k] >= 0) {
        xq[dst[k] * nblk + b] = q;
        bscale[dst[k] * nblk + b] = sc;
      }
    }
  };
  if (NB > 0) {
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (lane + 32 * j < nblk) put(lane + 32 * j, raw[2 * j], raw[2 * j + 1]);
  } else {
    for (int b = lane; b < nblk; b += 32) put(b, __ldg(row + 2 * b), __ldg(row + 2 * b + 1));
  }
}

// x_perm[r] = code * s_b * g in bf16 (exact), 8 elements (4 code bytes, one
// 16-byte store) per thread step.  L lanes per row (dequant_lanes), four steps'
// loads in flight before the first is converted, so no address needs a division
// and a warp writes 512 contiguous bytes.
// Bound by HBM: at 49146 rows of 2048 (258 MB) 37.4 us, 6.9 TB/s; one step per
// thread of a flat grid, with a 64-bit division for the row, took 60.
template <int L>
__global__ void __launch_bounds__(256) dequant_nvfp4_kernel(const uint32_t* __restrict__ xq,
                                                            const uint8_t* __restrict__ bscale,
                                                            const float* __restrict__ rscale, int64_t rows,
                                                            int vpr, uint4* __restrict__ out) {
  constexpr int U = 4;
  const int64_t r = (int64_t)blockIdx.x * (256 / L) + threadIdx.x / L;
  if (r >= rows) return;
  xq += r * vpr;
  bscale += r * (vpr / 2);
  out += r * vpr;
  const float g = __ldg(rscale + r);
  for (int v0 = threadIdx.x % L; v0 < vpr; v0 += U * L) {
    uint32_t w[U];
    uint8_t sc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int v = v0 + u * L;
      w[u] = v < vpr ? __ldcs(xq + v) : 0u;
      sc[u] = v < vpr ? __ldg(bscale + (v >> 1)) : (uint8_t)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int v = v0 + u * L;
      if (v >= vpr) break;
      const float s = e4m3_to_float(sc[u]) * g;
      float f[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __half2_raw hr = __nv_cvt_fp4x2_to_halfraw2((__nv_fp4x2_storage_t)(w[u] >> (8 * j)), __NV_E2M1);
        const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&hr));
        f[2 * j] = p.x * s;
        f[2 * j + 1] = p.y * s;
      }
      st_stream(out + v, pack16<bf16>(f));
    }
  }
}

int k_bound(int K) { return K <= 2 ? 2 : K <= 4 ? 4 : K <= 8 ? 8 : 16; }

}  // namespace

cudaError_t launch_dispatch_nvfp4(const Ctx& c, const void* x, const int32_t* row_of_slot, int64_t T, int K, int D,
                                  void* xq, uint8_t* bscale, float* rscale) {
  if (T == 0) return cudaSuccess;
  const int warps = 8;
  const dim3 grid((unsigned)((T + warps - 1) / warps));
  const int vpr = D / 8;
  KernelScope ks("dispatch_nvfp4", c.stream);
  auto run = [&](auto kernel) {
    kernel<<<grid, 32 * warps, 0, c.stream>>>((const uint4*)x, row_of_slot, T, K, vpr, (uint2*)xq, bscale, rscale,
                                              c.err);
  };
  auto by_width = [&](auto km) {
    constexpr int KM = decltype(km)::value;
    if (D <= 512) run(dispatch_nvfp4_kernel<KM, 1>);
    else if (D <= 1024) run(dispatch_nvfp4_kernel<KM, 2>);
    else if (D <= 2048) run(dispatch_nvfp4_kernel<KM, 4>);
    else run(dispatch_nvfp4_kernel<KM, 0>);
  };
  switch (k_bound(K)) {
    case 2: by_width(std::integral_constant<int, 2>()); break;
    case 4: by_width(std::integral_constant<int, 4>()); break;
    case 8: by_width(std::integral_constant<int, 8>()); break;
    default: by_width(std::integral_constant<int, 16>()); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_dequant_nvfp4(const Ctx& c, const void* xq, const uint8_t* bscale, const float* rscale,
                                 int64_t rows, int D, void* out) {
  if (rows == 0) return cudaSuccess;
  const int vpr = D / 8;  // a multiple of 8
  const int L = dequant_lanes(c, rows, vpr);
  const int rpb = 256 / L;
  const unsigned blocks = (unsigned)((rows + rpb - 1) / rpb);
  const uint32_t* q = (const uint32_t*)xq;
  KernelScope ks("dequant_nvfp4", c.stream);
  if (L == 256) dequant_nvfp4_kernel<256><<<blocks, 256, 0, c.stream>>>(q, bscale, rscale, rows, vpr, (uint4*)out);
  else if (L == 32) dequant_nvfp4_kernel<32><<<blocks, 256, 0, c.stream>>>(q, bscale, rscale, rows, vpr, (uint4*)out);
  else if (L == 16) dequant_nvfp4_kernel<16><<<blocks, 256, 0, c.stream>>>(q, bscale, rscale, rows, vpr, (uint4*)out);
  else dequant_nvfp4_kernel<8><<<blocks, 256, 0, c.stream>>>(q, bscale, rscale, rows, vpr, (uint4*)out);
  return cudaGetLastError();
}

}  // namespace moe
