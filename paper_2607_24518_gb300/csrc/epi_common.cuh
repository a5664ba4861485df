// Device helpers shared by the stand-alone epilogue and reduction kernels
// and the fused epilogue of the tensor-core kernels: number formats of the
// MMA copy of H, the stream-K slot arithmetic, and fixed-order summation.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_fp16.h>

#include "../../include/symnmf.h"
#include "symnmf_internal.h"

namespace symnmf {

// Launch as a programmatic dependent of the kernel before it in the stream:
// the kernel executes griddepcontrol.wait before it touches what that one
// writes, and always before it ends.
template <class... P, class... A>
cudaError_t launch_dependent(void (*f)(P...), dim3 grid, int threads, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, f, args...);
}

__device__ __forceinline__ uint16_t bf16_bits(float x) {
  __nv_bfloat16 b = __float2bfloat16_rn(x);
  return *reinterpret_cast<uint16_t *>(&b);
}
__device__ __forceinline__ float bf16_val(uint16_t u) {
  __nv_bfloat16 b = *reinterpret_cast<__nv_bfloat16 *>(&u);
  return __bfloat162float(b);
}
// tf32 value of x >= 0 with the 13 low mantissa bits cleared
__device__ __forceinline__ float tf32_trunc(float x) {
  return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
}
// x >= 0 rounded to the nearest tf32 value (ties away from zero)
__device__ __forceinline__ float tf32_round(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

// OCP E4M3 code of x, round to nearest even, saturating at +-448
__device__ __forceinline__ uint8_t e4m3_bits(float x) {
  return (uint8_t)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ float e4m3_val(uint8_t u) {
  return __half2float(__half(__nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)u, __NV_E4M3)));
}
// smallest power of two d with amax / d <= 448 (1 for amax = 0 or not
// finite).  With amax = m 2^E, m in [0.5, 1): amax / 448 = (m / 1.75)
// 2^(E-8), so d = 2^(E-9) when m <= 0.875 and 2^(E-8) otherwise; frexpf
// is exact, so the decision is exact.
__device__ __forceinline__ float e4m3_tile_scale(float amax) {
  if (!(amax > 0.f) || !isfinite(amax)) return 1.f;
  int E;
  const float m = frexpf(amax, &E);
  int e = E - 9 + (m > 0.875f ? 1 : 0);
  if (e < -100) e = -100;
  return ldexpf(1.f, e);
}
// two-piece E4M3 form of h at tile factor d: h ~ d (hi + lo), hi the
// E4M3 value of h / d and lo that of the remainder h / d - hi (exact in
// FP32), both rounded to nearest even
__device__ __forceinline__ void e4m3_pieces(float h, float inv_d, uint8_t &hi, uint8_t &lo) {
  const float x = h * inv_d;
  hi = e4m3_bits(x);
  lo = e4m3_bits(x - e4m3_val(hi));
}

// CTA of a stream-K launch whose unit range [b W / G, (b+1) W / G) holds x
__device__ __forceinline__ int64_t sk_cta(int64_t x, int64_t W, int64_t G) {
  int64_t b = x * G / W;
  while (b + 1 < G && (b + 1) * W / G <= x) ++b;
  while (b > 0 && b * W / G > x) --b;
  return b;
}

// Partials of a product launch that ran without the fused epilogue (slots are
// 128 x KP row-major blocks): with the stream-K layout (skG > 0) CTAs b0..b1
// hold row position p's partials in slots b + p; the SIMT layout has nsplit
// column shares per position, slot share * nlist + p.  They are added in that
// order.
__device__ __forceinline__ void part_range(int p, int skG, int ncols, int nlist, int64_t &b0,
                                           int64_t &b1) {
  b0 = b1 = 0;
  if (skG > 0) {
    const int64_t W = (int64_t)nlist * ncols;
    b0 = sk_cta((int64_t)p * ncols, W, skG);
    b1 = sk_cta((int64_t)p * ncols + ncols - 1, W, skG);
  }
}
// num / (sqrt(v) + eps), the AdaGrad / RMSprop step (Sec. 2.2), in
// straight-line code: PTX sqrt.approx.f32 (relative error at most 2^-23)
// and div.full.f32 (at most 2 ulp over the full range).  With no
// out-of-line special-case path the columns of a row overlap in flight.  The
// sum, and what callers do with the quotient, are rounded on their own: the
// assembler may otherwise fuse them with the last multiplication inside the
// square root or the quotient, in one kernel and not in another.
__device__ __forceinline__ float adaptive_step(float num, float v, float eps) {
  float r, q;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  asm("div.full.f32 %0, %1, %2;" : "=f"(q) : "f"(num), "f"(__fadd_rn(r, eps)));
  return q;
}

// Row order of every Gram partial (H_tile^T H_tile over a 128-row tile):
// entry (c, d) is (s_0 + s_1) + (s_2 + s_3), s_g the FMA chain over the rows
// r = 4 i + g, i = 0..31 in order, starting from zero.  gram_entry forms it
// from a tile in shared memory; gram_quad_sum adds the four s_g held by the
// lanes 4 q + g of a quad (every lane of the quad gets the same bits).
template <int KP>
__device__ __forceinline__ float gram_entry(const float (*Hn)[KP + 1], int c, int d) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int i = 0; i < kTileRows / 4; ++i)
#pragma unroll
    for (int g = 0; g < 4; ++g) s[g] = fmaf(Hn[4 * i + g][c], Hn[4 * i + g][d], s[g]);
  return (s[0] + s[1]) + (s[2] + s[3]);
}
__device__ __forceinline__ float gram_quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// (hi, lo) += (hi, lo) of lane ^ o for non-overlapping float pairs: the
// high parts by Knuth's TwoSum (exact: s + err = a + b), the low parts and
// err added and renormalised by Fast2Sum.  Relative error near 2^-44; both
// lanes of the pair get the same bits.
__device__ __forceinline__ void ff_xor_add(float &hi, float &lo, int o) {
  const float bh = __shfl_xor_sync(0xffffffffu, hi, o);
  const float bl = __shfl_xor_sync(0xffffffffu, lo, o);
  const float s = __fadd_rn(hi, bh);
  const float v = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(bh, v));
  const float t = __fadd_rn(__fadd_rn(lo, bl), err);
  hi = __fadd_rn(s, t);
  lo = __fsub_rn(t, __fsub_rn(hi, s));
}

// Running sum of squares as a float-float pair: the product is split exactly
// by an FMA and the high parts are added by Knuth's TwoSum, so only the low
// part (near 2^-23 of the sum) is rounded.  FP64 runs at two operations per
// SM and cycle on this part; a run of 64 entries summed this way (rounding
// near 2^-47) takes three FP64 operations instead of 128 and more.
struct SqRun {
  float h = 0.f, l = 0.f, m = 0.f;  // sum = h + l, m = largest magnitude
  // SHORT: v has at most 12 significant bits, so its square is exact
  template <bool SHORT = false>
  __device__ __forceinline__ void add(float v) {
    const float p = __fmul_rn(v, v);
    const float t = __fadd_rn(h, p), b = __fsub_rn(t, h);
    float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(p, b));
    if constexpr (!SHORT) e = __fadd_rn(e, fmaf(v, v, -p));
    l = __fadd_rn(l, e);
    h = t;
    m = fmaxf(m, fabsf(v));
  }
  // squares that neither overflow nor lose bits to underflow; otherwise the
  // caller sums the run in FP64
  __device__ __forceinline__ bool in_range() const {
    return m < 0x1p56f && (m == 0.f || m > 0x1p-40f);
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

// entry i of S (FP8: the code's value, without its tile scale)
template <int DT>
__device__ __forceinline__ float s_entry(const void *S, int64_t i) {
  if constexpr (DT == 0) return __ldg(reinterpret_cast<const float *>(S) + i);
  else if constexpr (DT == 1) return bf16_val(__ldg(reinterpret_cast<const uint16_t *>(S) + i));
  else return e4m3_val(__ldg(reinterpret_cast<const uint8_t *>(S) + i));
}
// a lane's 16 entries of columns c0 .. c0 + 511 of a row of S, in 16-byte
// groups one warp apart (vec: every row starts on a 16-byte boundary), else
// element by element; entries from column n on are 0.  FP8: the 16 entries
// are consecutive, so they share a tile scale.
template <int DT>
__device__ __forceinline__ void load16(const void *S, int64_t rowbase, int64_t c0, int64_t n,
                                       bool vec, int lane, float (&v)[16]) {
  constexpr int W = DT == 0 ? 4 : DT == 1 ? 8 : 16;  // entries of a 16-byte group
#pragma unroll
  for (int i = 0; i < 16 / W; ++i) {
    const int64_t c = c0 + (i * 32 + lane) * W;
    if (vec && c + W <= n) {
      const uint4 x = __ldg(reinterpret_cast<const uint4 *>(
          reinterpret_cast<const uint8_t *>(S) + (rowbase + c) * (16 / W)));
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if constexpr (DT == 0) {
          v[4 * i + j] = __uint_as_float(w[j]);
        } else if constexpr (DT == 1) {
          v[8 * i + 2 * j] = __uint_as_float(w[j] << 16);
          v[8 * i + 2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
        } else {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float2 f = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(
                (__nv_fp8x2_storage_t)(w[j] >> (16 * u)), __NV_E4M3)));
            v[4 * j + 2 * u] = f.x;
            v[4 * j + 2 * u + 1] = f.y;
          }
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < W; ++j) v[i * W + j] = c + j < n ? s_entry<DT>(S, rowbase + c + j) : 0.f;
    }
  }
}

// the lane's entries of columns [c0, c1) (as load16 deals them) summed in FP64
template <int DT>
__device__ __noinline__ double row_sumsq_lane64(const void *S, int64_t rowbase, int64_t c0,
                                                int64_t c1, int64_t n, const float *scales,
                                                int lane) {
  constexpr int W = DT == 0 ? 4 : DT == 1 ? 8 : 16;
  double acc = 0.0;
  for (int64_t c = c0 + lane * W; c < c1; c += 32 * W)
    for (int j = 0; j < W && c + j < n; ++j) {
      double x = (double)s_entry<DT>(S, rowbase + c + j);
      if constexpr (DT == 2) x *= (double)scales[(c + j) / kTileRows];
      acc = fma(x, x, acc);
    }
  return acc;
}

// One lane's share of sum_j S_rj^2 over row r: runs of 64 entries in
// float-float form, the runs in FP64.  FP8: a power-of-two tile scale (all
// that symnmf_quantize_fp8 writes) is exact in FP32; other scales and values
// out of SqRun's range take the FP64 sum.  `scales`: the row's tile scales.
template <int DT>
__device__ __forceinline__ double row_sumsq_lane(const void *S, int64_t rowbase, int64_t n,
                                                 const float *scales, bool vec, int lane) {
  double acc = 0.0;
  for (int64_t c0 = 0; c0 < n; c0 += 2048) {
    SqRun s;
    bool exact = true;
    // loads in flight per lane: one chunk of FP32 is four, of FP8 one
#pragma unroll (DT == 0 ? 1 : DT == 1 ? 2 : 4)
    for (int i = 0; i < 4; ++i) {
      const int64_t cc = c0 + 512 * i;
      if (DT != 2 && cc >= n) break;
      float v[16], sc = 1.f;
      load16<DT>(S, rowbase, cc, n, vec, lane, v);
      if constexpr (DT == 2) {
        sc = __ldg(scales + min(cc + 16 * lane, n - 1) / kTileRows);
        exact = exact && (__float_as_uint(sc) & 0x7FFFFFu) == 0u;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) s.template add<(DT == 2)>(DT == 2 ? v[j] * sc : v[j]);
    }
    if (exact && s.in_range()) acc += s.value();
    else acc += row_sumsq_lane64<DT>(S, rowbase, c0, min(c0 + 2048, n), n, scales, lane);
  }
  return acc;
}

}  // namespace symnmf
