// FP8 E4M3 storage of S with one power-of-two scale per 128 x 128 tile
// (the setup step before the solver streams S; the paper runs FP32 only, so
// this storage format is this library's).  One CTA per tile: the tile is
// read once into registers, its largest magnitude fixes the scale, then the
// codes are written.  The FP64 sum of squares of the unquantised tile is
// written beside the scale so the caller can form ||S||_F^2 of the source.
#include <cuda_bf16.h>

#include "epi_common.cuh"
#include "symnmf_internal.h"

namespace symnmf {
namespace {

// 256 threads: warp w covers rows 16 w .. 16 w + 15, lane l columns 4 l .. 4 l + 3.
// Bound by HBM (source read once, codes written once).  The sum of squares
// of the thread's 64 entries is kept in FP32 words with FP64 accuracy (SqSum;
// FP64 per entry bounded the kernel by the FP64 pipe; n=12000 FP32: 626 -> 182
// us); vsrc / vdst: 4-entry loads and 4-code stores, when base and pitch are
// aligned to them.
template <int SRC>
__global__ void __launch_bounds__(256) quantize_kernel(const void *src, int64_t rows, int64_t cols,
                                                       int64_t ld_src, uint8_t *q, int64_t ldq,
                                                       float *scales, int64_t ld_scales,
                                                       double *tile_sumsq, bool vsrc, bool vdst) {
  __shared__ float wmax[8];
  __shared__ double wsum[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = (int64_t)blockIdx.y * kTileRows, c0 = (int64_t)blockIdx.x * kTileRows;
  const int64_t c = c0 + lane * 4;
  float v[16][4];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int64_t r = r0 + warp * 16 + i;
    const int64_t at = r * ld_src + c;
    if (vsrc && r < rows && c + 4 <= cols) {
      if constexpr (SRC == 0) {
        const float4 x = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(src) + at));
        v[i][0] = x.x;
        v[i][1] = x.y;
        v[i][2] = x.z;
        v[i][3] = x.w;
      } else {
        const uint2 x = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(src) + at));
        v[i][0] = __uint_as_float(x.x << 16);
        v[i][1] = __uint_as_float(x.x & 0xFFFF0000u);
        v[i][2] = __uint_as_float(x.y << 16);
        v[i][3] = __uint_as_float(x.y & 0xFFFF0000u);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i][j] = (r < rows && c + j < cols) ? s_entry<SRC>(src, at + j) : 0.f;
    }
  }
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) m = fmaxf(m, fabsf(v[i][j]));
  double ss = 0.0;
  if (tile_sumsq) {
    SqSum<SRC == 1> s;
    if (m == 0.f || s.raise(m)) {
#pragma unroll
      for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s.put(v[i][j]);
      s.flush();
      ss = s.acc;
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ss = fma((double)v[i][j], (double)v[i][j], ss);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (tile_sumsq) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
  if (lane == 0) {
    wmax[warp] = m;
    wsum[warp] = ss;
  }
  __syncthreads();
  float amax = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) amax = fmaxf(amax, wmax[w]);
  const float sc = e4m3_tile_scale(amax), inv = 1.f / sc;
  if (threadIdx.x == 0) {
    scales[(int64_t)blockIdx.y * ld_scales + blockIdx.x] = sc;
    if (tile_sumsq) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += wsum[w];
      tile_sumsq[(int64_t)blockIdx.y * ld_scales + blockIdx.x] = t;
    }
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int64_t r = r0 + warp * 16 + i;
    if (r >= rows) break;
    const uint32_t w =
        (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(v[i][0] * inv, v[i][1] * inv),
                                           __NV_SATFINITE, __NV_E4M3) |
        ((uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(v[i][2] * inv, v[i][3] * inv),
                                            __NV_SATFINITE, __NV_E4M3) << 16);
    uint8_t *dst = q + r * ldq + c;
    if (vdst && c + 4 <= cols) {
      *reinterpret_cast<uint32_t *>(dst) = w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c + j < cols) dst[j] = (uint8_t)(w >> (8 * j));
    }
  }
}

}  // namespace

cudaError_t launch_quantize_fp8(const void *src, int src_dtype, int64_t rows, int64_t cols,
                                int64_t ld_src, uint8_t *q, int64_t ldq, float *scales,
                                int64_t ld_scales, double *tile_sumsq, cudaStream_t s) {
  const dim3 grid((unsigned)((cols + kTileRows - 1) / kTileRows),
                  (unsigned)((rows + kTileRows - 1) / kTileRows));
  const bool vsrc = reinterpret_cast<uintptr_t>(src) % (src_dtype == 0 ? 16 : 8) == 0 && ld_src % 4 == 0;
  const bool vdst = reinterpret_cast<uintptr_t>(q) % 4 == 0 && ldq % 4 == 0;
  if (src_dtype == 0)
    quantize_kernel<0><<<grid, 256, 0, s>>>(src, rows, cols, ld_src, q, ldq, scales, ld_scales,
                                            tile_sumsq, vsrc, vdst);
  else
    quantize_kernel<1><<<grid, 256, 0, s>>>(src, rows, cols, ld_src, q, ldq, scales, ld_scales,
                                            tile_sumsq, vsrc, vdst);
  return cudaGetLastError();
}

}  // namespace symnmf
