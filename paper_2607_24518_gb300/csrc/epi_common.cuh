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
// tf32 value of x with the 13 low mantissa bits cleared
__device__ __forceinline__ float tf32_trunc(float x) {
  return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
}
// x rounded to the nearest tf32 value (ties away from zero)
__device__ __forceinline__ float tf32_round(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}
// leading tf32 piece of an entry of H, whose remainder is the lower piece.  At
// kp = 64 the product S_lo H_lo is left out (bt_fmt 1, S_hi and S_hi H_lo cover
// the rest), and truncated pieces, all of one sign, would leave out as much
// from every term: to nearest, unless that overflows.  Gradient error of FP32
// at k = 33 .. 64, n = 1000 / 4096 / 9000 / 20000, mean of eight inputs, relative
// to the size of its terms: 9.4 / 9.3 / 9.6 / 11.1e-8 truncated (0.3% less with
// S H_lo in an accumulator of its own), 8.5 / 8.5 / 8.8 / 10.5e-8 to nearest.
template <int KP>
__device__ __forceinline__ float tf32_lead(float x) {
  const uint32_t a = __float_as_uint(x) & 0x7FFFFFFFu;
  return KP == 64 && a < 0x7F7FF000u ? tf32_round(x) : tf32_trunc(x);
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

// Sum of x over the warp in FP64, every lane the same bits: the values as
// 64-bit integers in units of 2^-34 of the largest one's last place, so that an
// integer tree adds them exactly (24 + 34 bits and 5 for 32 lanes); what lies
// below that unit, 2^-57 of the largest value, is cut off.  An integer tree
// takes two shuffles and two additions a level, as many shuffles as and fewer
// operations than float-float pairs, which hold 48 bits.  Infinities and NaN:
// the FP32 sum.
__device__ __forceinline__ double warp_sum64(float x) {
  const uint32_t u = __float_as_uint(x), a = u & 0x7FFFFFFFu;
  const uint32_t top = __reduce_max_sync(0xffffffffu, a);
  if (top >= 0x7F800000u) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return (double)x;
  }
  // exponent fields, 1 for subnormals as for the smallest normal numbers
  const int et = max((int)(top >> 23), 1), ex = max((int)(a >> 23), 1);
  int64_t m = (int64_t)((a & 0x7FFFFFu) | (a >= 0x800000u ? 0x800000u : 0u)) << 34;
  m = et - ex < 58 ? m >> (et - ex) : 0;
  if (u >> 31) m = -m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, (long long)m, o);
  return (double)m * __hiloint2double((et - 150 - 34 + 1023) << 20, 0);
}

// Running sum of squares of FP32 values with FP64 accuracy and few FP64
// operations (two per SM and cycle on this part): a run of up to 64 values in
// three FP32 words, joined in FP64 by flush().  With |v| <= cap (a power of
// two) the words start at anchors, H at A = 64 cap^2 and L at 1.5 * 2^-16 A.
// p = v^2 is below A / 64, so H stays in [A, 2 A), is never smaller than what
// is added and Fast2Sum (Dekker 1971) gives the exact error of H + p in two
// operations; that error and the product's own (one FMA) are at most 2^-24 A
// and go into L in the same way, 2^-18 A in all; what L rounds off is at most
// 2^-40 A each time and is added up in T.  Only those additions round, 2^-51 A
// for a run at the very most.  ||S||^2 of uniform FP32 entries, n = 2048: off by
// at most 2e-16 of itself (FP64 per entry 7e-16; two words without the third
// 5e-15).  A larger value flushes and raises cap; what leaves [2^-40, 2^56],
// where squares would lose bits or overflow, is summed in FP64.  EXACT: v has at
// most 12 significant bits, so p is exact.
template <bool EXACT = false>
struct SqSum {
  float H = 0.f, L = 0.f, T = 0.f, cap = 0.f;
  double acc = 0.0;  // the sum, once flushed
  __device__ __forceinline__ static float hi(float c) { return 64.f * c * c; }
  __device__ __forceinline__ static float lo(float c) { return 0x1.8p-10f * c * c; }
  __device__ __forceinline__ void put(float v) {
    const float p = __fmul_rn(v, v);
    const float t = __fadd_rn(H, p), e = __fsub_rn(p, __fsub_rn(t, H));
    H = t;
    low(e);
    if constexpr (!EXACT) low(fmaf(v, v, -p));
  }
  __device__ __forceinline__ void low(float e) {
    const float t = __fadd_rn(L, e);
    T = __fadd_rn(T, __fsub_rn(e, __fsub_rn(t, L)));
    L = t;
  }
  // H - A and L - 1.5 * 2^-16 A are exact; after at most 64 values
  __device__ __forceinline__ void flush() {
    acc += (double)__fsub_rn(H, hi(cap));
    acc += (double)__fsub_rn(L, lo(cap));
    acc += (double)T;
    H = hi(cap);
    L = lo(cap);
    T = 0.f;
  }
  // ready for values up to m (m > cap); false: they have to be summed in FP64
  __device__ __forceinline__ bool raise(float m) {
    if (!(m > 0x1p-40f && m < 0x1p56f)) return false;
    if (H != 0.f) flush();  // (nothing but zeros before)
    cap = __uint_as_float((__float_as_uint(m) & 0x7F800000u) + 0x00800000u);
    H = hi(cap);
    L = lo(cap);
    return true;
  }
  template <int N>
  __device__ __forceinline__ void add(const float (&v)[N]) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) m = fmaxf(m, fabsf(v[i]));
    if (m > cap && !raise(m)) {
#pragma unroll
      for (int i = 0; i < N; ++i) acc = fma((double)v[i], (double)v[i], acc);
      return;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) put(v[i]);
  }
};

// entry i of S (FP8: the code's value, without its tile scale)
template <int DT>
__device__ __forceinline__ float s_entry(const void *S, int64_t i) {
  if constexpr (DT == 0) return __ldg(reinterpret_cast<const float *>(S) + i);
  else if constexpr (DT == 1) return bf16_val(__ldg(reinterpret_cast<const uint16_t *>(S) + i));
  else return e4m3_val(__ldg(reinterpret_cast<const uint8_t *>(S) + i));
}
// 16 E4M3 codes of a row from column c on (vec: the row starts on a 16-byte
// boundary, c is a multiple of 16), 0 from column n on; and their values
__device__ __forceinline__ uint4 load_codes(const void *S, int64_t rowbase, int64_t c, int64_t n,
                                            bool vec) {
  const uint8_t *p = reinterpret_cast<const uint8_t *>(S) + rowbase + c;
  if (vec && c + 16 <= n) return __ldg(reinterpret_cast<const uint4 *>(p));
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if (c + j < n) w[j / 4] |= (uint32_t)__ldg(p + j) << (8 * (j % 4));
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ void e4m3_vals(const uint4 &x, float (&v)[16]) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float2 f = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(
          (__nv_fp8x2_storage_t)(w[j] >> (16 * u)), __NV_E4M3)));
      v[4 * j + 2 * u] = f.x;
      v[4 * j + 2 * u + 1] = f.y;
    }
}
// a lane's 16 entries of columns c0 .. c0 + 511 of a row of S (FP32, BF16), in
// 16-byte groups one warp apart (vec: every row starts on a 16-byte boundary),
// else element by element; entries from column n on are 0
template <int DT>
__device__ __forceinline__ void load16(const void *S, int64_t rowbase, int64_t c0, int64_t n,
                                       bool vec, int lane, float (&v)[16]) {
  constexpr int W = DT == 0 ? 4 : 8;  // entries of a 16-byte group
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
        } else {
          v[8 * i + 2 * j] = __uint_as_float(w[j] << 16);
          v[8 * i + 2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < W; ++j) v[i * W + j] = c + j < n ? s_entry<DT>(S, rowbase + c + j) : 0.f;
    }
  }
}

// One lane's share of sum_j S_rj^2 over row r, in runs of 64 entries.  FP8: a
// code's square has at most 8 significant bits, none below 2^-18, and 64 of
// them stay below 2^24, so with H from 2^24 on (ulp 2) and L (at most one per
// code, multiples of 2^-18) a run is exact in two words and four operations per
// code; the tile scale enters in FP64, whenever it changes (`scales`: the row's
// tile scales).  n = 12000, ||S||^2: FP32 111, BF16 106, FP8 48 us (two words,
// which hold 48 bits: 100, 105 and 72, and 1220 with scales that are no powers
// of two; FP64 per entry: 555, 556 and 1068).
template <int DT>
__device__ __forceinline__ double row_sumsq_lane(const void *S, int64_t rowbase, int64_t n,
                                                 const float *scales, bool vec, int lane) {
  if constexpr (DT == 2) {
    double acc = 0.0, s2 = 1.0;
    float H = 0x1p24f, L = 0.f, scale = 1.f;
    auto flush = [&]() {
      acc = fma(s2, (double)__fsub_rn(H, 0x1p24f) + (double)L, acc);
      H = 0x1p24f;
      L = 0.f;
    };
    auto add = [&](const uint4 &x) {
      float v[16];
      e4m3_vals(x, v);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float t = fmaf(v[j], v[j], H);
        L = __fadd_rn(L, fmaf(v[j], v[j], -__fsub_rn(t, H)));
        H = t;
      }
    };
    for (int64_t c0 = 16 * lane; c0 < n + 16 * lane; c0 += 2048) {
      uint4 x[4];
      float sc[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {  // all loads of a run first
        const int64_t c = c0 + 512 * i;
        x[i] = load_codes(S, rowbase, c, n, vec);
        sc[i] = __ldg(scales + min(c, n - 1) / kTileRows);
      }
      if (sc[0] == scale && sc[1] == scale && sc[2] == scale && sc[3] == scale) {
#pragma unroll
        for (int i = 0; i < 4; ++i) add(x[i]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (sc[i] != scale) {
            flush();
            scale = sc[i];
            s2 = (double)scale * (double)scale;
          }
          add(x[i]);
        }
      }
      flush();
    }
    return acc;
  } else {
    SqSum<(DT == 1)> s;
    for (int64_t c0 = 0; c0 < n; c0 += 2048) {
      // loads in flight per lane: one chunk of FP32 is four, of BF16 two
#pragma unroll (DT == 0 ? 1 : 2)
      for (int i = 0; i < 4; ++i) {
        const int64_t cc = c0 + 512 * i;
        if (cc >= n) break;
        float v[16];
        load16<DT>(S, rowbase, cc, n, vec, lane, v);
        s.add(v);
      }
      s.flush();
    }
    return s.acc;
  }
}

}  // namespace symnmf
