// Dependence matrix on the GPU (Sec. 3: the absolute correlation matrix and
// the empirical TPDM), the step before the solver.  Both are unit-diagonal
// normalisations of a Gram matrix of the n variables over T observations:
//   S_ij = |G_ij| / sqrt(G_ii G_jj),   G = Y^T Y,
// with Y the observations with centred columns (correlation) or the
// exceedance angles Omega (TPDM; the n / n_exc factor cancels).
//
// Kernels:
//   dep_prep    one CTA per 32 variables: column means (centring), the FP64
//               sum d_i of the squares of the FP32 centred values c_ti, and
//               the transposed operand P = [hi | lo] (n x 2 Tp, FP16): with
//               s_i the power of two that brings sqrt(d_i) into [2^14, 2^15),
//               hi = fp16(s_i c), lo = fp16(s_i c - hi), both to nearest, so
//               hi + lo keeps 22 bits of c (entries below 2^-17 sqrt(d_i):
//               2^-39 sqrt(d_i) absolute); Tp = T rounded up to 32
//   dep_gemm    persistent, one CTA per SM over the 128 x 256 tiles of G on
//               or above the diagonal, on tcgen05 (kind::f16, M = 128, N =
//               256, two accumulators in tensor memory taken in turn, so a
//               tile's epilogue overlaps the next tile's MMAs): each stage
//               holds a 32-column chunk of A_hi, A_lo, B_hi and B_lo (64-byte
//               swizzle, fetched from P by TMA) and feeds the three products
//               hi hi, lo hi and hi lo (the dropped lo lo term is below
//               2^-24 relative), so every staged byte serves two products;
//               the epilogue normalises, clamps to [0, 1], writes 1 on the
//               diagonal and stores S as FP32, BF16 (round to nearest) or
//               E4M3 with one power-of-two scale per 128 x 128 tile, plus
//               the CTA's FP64 sum of squares (FP8: of the values before
//               quantisation).  Only 128 x 128 tiles on or above the
//               diagonal are computed; each one above it is also stored
//               transposed, so S is exactly symmetric and the tensor work is
//               halved
//   dep_sum     fixed-order FP64 sum of the CTA partials -> ||S||^2
// FP16 pieces hold as many bits as tf32 ones (11) in half the bytes and at
// twice the tensor rate, and a dot product takes half as many chained
// accumulations; the column scales remove FP16's narrow range.  n = 20000,
// T = 500: FP32 / BF16 / FP8 output 548 / 462 / 442 us (tf32 pieces, four
// epilogue warps with per-entry tests and stores: 1348 / 1349 / 2102 us),
// error of S 1.8e-6 instead of 4.5e-6.  The FP8 figure is the operand
// stream's (4.8 GB from L2, 11 TB/s); the wider outputs add their stores.
// Every mbarrier wait is bounded (2 s); on expiry the CTA records an error
// code, drains its own copies, frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "../../include/symnmf.h"
#include "epi_common.cuh"
#include "symnmf_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>

namespace symnmf {
namespace {

using namespace tc;

constexpr int kDepStages = 4;
constexpr int kDepKC = 32;                             // halves per staged row (64 bytes)
constexpr uint32_t kDepA = 128 * 64;                   // 128 rows x 32 halves
constexpr uint32_t kDepB = 256 * 64;                   // 256 rows x 32 halves
constexpr uint32_t kDepStage = 2 * kDepA + 2 * kDepB;  // A_hi, A_lo, B_hi, B_lo: 48 KB
constexpr size_t kDepSmem = 1024 + (size_t)kDepStages * kDepStage + 256 + 256 * 4 + 64 * 8;
constexpr int kDepThreads = 320;  // warp 0 TMA, warp 1 MMA, warps 2-9 epilogue
constexpr int kDepGroup = 16;     // row tiles that sweep the column blocks together

// s += v; returns the exact error (Knuth's TwoSum)
__device__ __forceinline__ float two_sum(float &s, float v) {
  const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b));
  s = t;
  return e;
}

// One CTA per 32 variables, 32 x 16 threads: thread (x, y) sums variable
// i0 + x over the observations y, y + 16, ...  Runs of 64 observations are
// kept in three FP32 words (TwoSum, SqSum), the runs are added in FP64 and the
// 16 threads of a variable in order.  Bound by HBM once Y is read; FP64 per
// entry in one thread per variable was bound by latency and the FP64 pipe.
constexpr int kPrepY = 16;   // threads per variable
constexpr int kPrepT = 128;  // observations transposed together
__global__ void __launch_bounds__(32 * kPrepY, 2)
    dep_prep_kernel(const float *Y, int64_t T, int64_t n, int64_t ldy, int center, int Tp,
                    float *inv_d, __half *P) {
  __shared__ double part[kPrepY][33];
  __shared__ float tile[kPrepT][33];
  __shared__ float mean[32];
  __shared__ int sexp[32];
  const int x = threadIdx.x, y = threadIdx.y;
  const int64_t i0 = (int64_t)blockIdx.x * 32, i = i0 + x;
  const bool have = i < n;
  const float *col = Y + (have ? i : i0);
  // the variable's partial sums, added in order by thread (x, 0)
  auto total = [&](double v) -> double {
    part[y][x] = v;
    __syncthreads();
    double s = 0.0;
    if (y == 0)
      for (int k = 0; k < kPrepY; ++k) s += part[k][x];
    __syncthreads();
    return s;
  };
  // (T is at most 2^30)
  constexpr int kRun = 64 * kPrepY;
  const int Ti = (int)T;
  const int64_t step = (int64_t)kPrepY * ldy;
  float mf = 0.f;
  if (center) {
    double m = 0.0;
    for (int t = y; t < Ti; t += kRun) {
      float h = 0.f, l = 0.f, r = 0.f;  // what h and l round off goes one word down
      const float *p = col + t * ldy;
      const int e = min(Ti, t + kRun);
#pragma unroll 8
      for (int tt = t; tt < e; tt += kPrepY, p += step) r = __fadd_rn(r, two_sum(l, two_sum(h, __ldg(p))));
      if (isfinite(h + l)) {
        m += (double)h;
        m += (double)l;
        m += (double)r;
      } else {  // levels from about FLT_MAX / 64 overflow the run's high word
        p = col + t * ldy;
        for (int tt = t; tt < e; tt += kPrepY, p += step) m += (double)__ldg(p);
      }
    }
    m = total(m);
    if (y == 0) mean[x] = (float)(m / (double)T);
    __syncthreads();
    mf = mean[x];
  }
  SqSum<> sq;
  for (int t = y; t < Ti; t += kRun) {
    const float *p = col + t * ldy;
    for (int t8 = t; t8 < min(Ti, t + kRun); t8 += 8 * kPrepY) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u, p += step) v[u] = t8 + u * kPrepY < Ti ? __ldg(p) - mf : 0.f;
      sq.add(v);
    }
    sq.flush();
  }
  double d = sq.acc;
  d = total(d);
  if (y == 0) {
    // s = 2^e with s sqrt(d) in [2^14, 2^15); 1 for a column without a norm
    int e = 0;
    double inv = 0.0;
    if (d > 0.0 && d <= 1.7976931348623157e308) {
      frexp(sqrt(d), &e);
      e = 15 - e;
      inv = ldexp(1.0 / sqrt(d), -e);  // of the scaled column
    }
    sexp[x] = e;
    if (have) inv_d[i] = (float)inv;
  }
  __syncthreads();
  // P row i: hi at [0, Tp), lo at [Tp, 2 Tp); warp y writes variables y and
  // y + 16, two observations per lane
  const int64_t pitch = 2 * (int64_t)Tp;
  const int se = sexp[x];
  for (int64_t t0 = 0; t0 < Tp; t0 += kPrepT) {
#pragma unroll
    for (int k = 0; k < kPrepT / kPrepY; ++k) {
      const int64_t t = t0 + y + k * kPrepY;
      tile[y + k * kPrepY][x] = t < T ? ldexpf(__ldg(col + t * ldy) - mf, se) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 32 / kPrepY; ++v) {
      const int iv = y + v * kPrepY;
#pragma unroll
      for (int k = 0; k < kPrepT / 64; ++k) {
        const int tt = k * 64 + 2 * x;
        if (i0 + iv < n && t0 + tt < Tp) {  // Tp is even
          const float c0 = tile[tt][iv], c1 = tile[tt + 1][iv];
          const __half2 hi = __floats2half2_rn(c0, c1);
          const float2 hf = __half22float2(hi);
          __half2 *dst = reinterpret_cast<__half2 *>(P + (i0 + iv) * pitch + t0 + tt);
          dst[0] = hi;
          dst[Tp / 2] = __floats2half2_rn(c0 - hf.x, c1 - hf.y);
        }
      }
    }
    __syncthreads();
  }
}

struct DepArgs {
  int64_t n;
  int Tp;
  int natoms;       // Tp / 32 staged chunks per tile
  int nib, njb;     // 128-row tiles, 256-column blocks
  int ntiles;       // tiles on or above the diagonal
  const float *inv_d;  // 1 / (s_i sqrt(d_i))
  void *S;
  int64_t lds;
  int out;          // 0 FP32, 1 BF16, 2 E4M3
  float *scales;
  int64_t ld_scales;
  double *sq;       // per CTA
  int *err;
  bool w8;          // every row of S starts on a 32-byte boundary
  int exact_sq;     // F32 / BF16: run sums of squares as float-float pairs
};

// The tile list: groups of kDepGroup row tiles that sweep the column blocks
// together (the operand rows they share stay in L2), of each group the tiles
// (ib, jb) with 2 jb + 1 >= ib: in the group from row tile g0 (a multiple of
// 16, R of its rows exist), block g0 / 2 + x holds min(2 x + 2, R) tiles for
// x < 8 and R from there on.
__host__ __device__ inline int dep_group_tiles(int g0, int nib, int njb) {
  const int R = nib - g0 < kDepGroup ? nib - g0 : kDepGroup;
  const int cols = njb - g0 / 2;
  int m = 0;
  for (int x = 0; x < kDepGroup / 2 && x < cols; ++x) m += 2 * x + 2 < R ? 2 * x + 2 : R;
  return cols > kDepGroup / 2 ? m + (cols - kDepGroup / 2) * R : m;
}
struct DepTiles {  // walks the list forward
  int g0 = 0, base = 0, size;
  __device__ __forceinline__ DepTiles(const DepArgs &a) : size(dep_group_tiles(0, a.nib, a.njb)) {}
  __device__ __forceinline__ void at(const DepArgs &a, int t, int &ib, int &jb) {
    while (t >= base + size) {
      base += size;
      g0 += kDepGroup;
      size = dep_group_tiles(g0, a.nib, a.njb);
    }
    const int R = a.nib - g0 < kDepGroup ? a.nib - g0 : kDepGroup;
    int k = t - base, x = 0;
    for (; x < kDepGroup / 2; ++x) {
      const int c = 2 * x + 2 < R ? 2 * x + 2 : R;
      if (k < c) break;
      k -= c;
    }
    if (x == kDepGroup / 2) {
      x += k / R;
      k %= R;
    }
    ib = g0 + k;
    jb = g0 / 2 + x;
  }
};

// the same verdict for the 128 epilogue threads of column half h: whether
// all of them have ok (a warp that gave up alone would leave the others at
// the next barrier)
__device__ __forceinline__ bool dep_all(int h, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %2, 0;\n bar.red.and.pred q, %1, 128, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(1 + h), "r"((uint32_t)ok)
      : "memory");
  return r != 0;
}
// 32 bytes of one row, on a 32-byte boundary when w8, else on a 16-byte one.
// The rows of a warp lie in 32 lines; a 16-byte store is a partial sector to
// L2, which bounded the wider outputs (n = 20000, T = 500, GEMM: FP32 684 ->
// 548 us, BF16 535 -> 462, FP8 462 -> 442; streaming and write-through hints
// changed nothing).
__device__ __forceinline__ void dep_store32(void *dst, bool w8, uint32_t a, uint32_t b, uint32_t c,
                                            uint32_t d, uint32_t e, uint32_t f, uint32_t g,
                                            uint32_t h) {
  if (w8) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a),
                 "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h)
                 : "memory");
  } else {
    reinterpret_cast<uint4 *>(dst)[0] = make_uint4(a, b, c, d);
    reinterpret_cast<uint4 *>(dst)[1] = make_uint4(e, f, g, h);
  }
}
// barrier among the 128 epilogue threads of column half h
__device__ __forceinline__ void dep_bar(int h) {
  asm volatile("bar.sync %0, 128;" ::"r"(1 + h) : "memory");
}

// Persistent: CTA b takes tiles b, b + G, b + 2G, ... of the list.  Two
// accumulators of 256 TMEM columns alternate between tiles, so the
// epilogue of one tile overlaps the MMAs of the next.
__global__ void __launch_bounds__(kDepThreads, 1)
    dep_gemm_kernel(const __grid_constant__ CUtensorMap mP, const DepArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + kDepStages * kDepStage);
  uint64_t *empty = full + kDepStages;
  uint64_t *accf = empty + kDepStages;  // 2: accumulator ready for the epilogue
  uint64_t *acce = accf + 2;            // 2: accumulator free for the MMAs
  uint32_t *holder = reinterpret_cast<uint32_t *>(acce + 2);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(holder + 1);
  int *consumed = const_cast<int *>(abort_flag) + 1;
  float *invj = reinterpret_cast<float *>(smem + kDepStages * kDepStage + 256);
  double *red = reinterpret_cast<double *>(invj + 256);  // 64 doubles

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = gridDim.x;
  const int my_tiles = (a.ntiles - (int)blockIdx.x + G - 1) / G;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDepStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 8);
    }
    *abort_flag = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(holder, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = *holder;
  int issued = 0;

  if (warp == 0) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mP)) : "memory");
      DepTiles walk(a);
      int c = 0;  // chunks issued over all tiles
      bool stop = false;
      for (int lt = 0; lt < my_tiles && !stop; ++lt) {
        int ib, jb;
        walk.at(a, blockIdx.x + lt * G, ib, jb);
        for (int at = 0; at < a.natoms; ++at, ++c) {
          const int s = c % kDepStages;
          if (c >= kDepStages &&
              !mbar_wait(&empty[s], (uint32_t)((c / kDepStages - 1) & 1), abort_flag)) {
            set_err(a.err, 31);
            *abort_flag = 1;
            stop = true;
            break;
          }
          const int o = at * kDepKC;
          uint8_t *st = smem + (size_t)s * kDepStage;
          uint8_t *sb = st + 2 * kDepA;
          mbar_expect_tx(&full[s], kDepStage);
          tma_load_2d(st, &mP, &full[s], o, ib * 128);                    // A_hi
          tma_load_2d(st + kDepA, &mP, &full[s], a.Tp + o, ib * 128);     // A_lo
          tma_load_2d(sb, &mP, &full[s], o, jb * 256);                    // B_hi
          tma_load_2d(sb + kDepB / 2, &mP, &full[s], o, jb * 256 + 128);
          tma_load_2d(sb + kDepB, &mP, &full[s], a.Tp + o, jb * 256);     // B_lo
          tma_load_2d(sb + kDepB + kDepB / 2, &mP, &full[s], a.Tp + o, jb * 256 + 128);
          ++issued;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_f16(128, 256);
      int c = 0, done = 0;
      bool stop = false;
      for (int lt = 0; lt < my_tiles && !stop; ++lt) {
        const int b = lt & 1;
        if (lt >= 2 && !mbar_wait(&acce[b], (uint32_t)((lt / 2 - 1) & 1), abort_flag)) {
          set_err(a.err, 34);
          *abort_flag = 1;
          break;
        }
        fence_after();
        const uint32_t tacc = tbase + (uint32_t)(b * 256);
        for (int at = 0; at < a.natoms; ++at, ++c) {
          const int s = c % kDepStages;
          if (!mbar_wait(&full[s], (uint32_t)((c / kDepStages) & 1), abort_flag)) {
            set_err(a.err, 32);
            *abort_flag = 1;
            stop = true;
            break;
          }
          fence_after();
          const uint64_t ah = sdesc64(smem_u32(smem + (size_t)s * kDepStage));
          const uint64_t al = ah + (kDepA >> 4), bh = ah + (2 * kDepA >> 4), bl = bh + (kDepB >> 4);
#pragma unroll
          for (int ks = 0; ks < kDepKC / 16; ++ks) {  // K = 16 halves (32 bytes) per MMA
            const uint64_t o = (uint64_t)ks * 2u;     // descriptors count 16 bytes
            mma_f16(tacc, ah + o, bh + o, idesc, (at > 0 || ks > 0) ? 1u : 0u);
            mma_f16(tacc, al + o, bh + o, idesc, 1u);
            mma_f16(tacc, ah + o, bl + o, idesc, 1u);
          }
          mma_commit(&empty[s]);
          done = c + 1;
        }
        mma_commit(&accf[b]);
      }
      *consumed = done;
    }
  } else {
    // epilogue: thread row r of each tile; warps 2-5 take its 128-column
    // tile jt = 2 jb, warps 6-9 jt = 2 jb + 1.  Only the upper triangle is
    // computed: a tile with jt > ib is stored and mirrored to (jt, ib)
    // (lane = row, so the mirrored stores of a warp are 32 consecutive
    // entries of one row); in a tile with jt == ib the entries j >= i are
    // stored and those with j > i mirrored; jt < ib is left to its mirror.
    // Every stored pair S_ij, S_ji is one accumulator value, so S is exactly
    // symmetric.  A whole tile above the diagonal takes no per-entry test.
    const int q = warp & 3, r = q * 32 + lane, half = (warp - 2) >> 2;
    const int et = ((warp - 2) & 3) * 32 + lane;  // 0..127 within the half
    float *ij = invj + half * 128;
    double *rd = red + half * 32;
    double sq = 0.0;
    DepTiles walk(a);
    for (int lt = 0; lt < my_tiles; ++lt) {
      const int b = lt & 1;
      int ib, jb;
      walk.at(a, blockIdx.x + lt * G, ib, jb);
      const int jt = 2 * jb + half;
      const int64_t i = (int64_t)ib * 128 + r, j0 = (int64_t)jt * 128;
      const bool vrow = i < a.n;
      const int md = (j0 >= a.n || jt < ib) ? 0 : jt == ib ? 1 : 2;  // skip, diagonal, mirror
      const bool inner = md == 2 && j0 + 128 <= a.n && (int64_t)ib * 128 + 128 <= a.n;
      const float inv_i = vrow ? a.inv_d[i] : 0.f;
      dep_bar(half);  // every thread is done with the previous tile's invj
      ij[et] = j0 + et < a.n ? a.inv_d[j0 + et] : 0.f;
      dep_bar(half);
      const bool ok = warp_wait_idle(&accf[b], (uint32_t)((lt / 2) & 1), abort_flag);
      if (!ok && lane == 0) {
        set_err(a.err, 33);
        *abort_flag = 1;
      }
      if (!dep_all(half, ok)) break;
      fence_after();
      const uint32_t trow =
          tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * 256 + half * 128);
      // 32 accumulator columns from c0, normalised
      auto values = [&](int c0, float (&v)[32]) {
        uint32_t x[32];
#pragma unroll
        for (int u = 0; u < 4; ++u) tmem_ld8_nw(trow + c0 + 8 * u, x, 8 * u);
        tmem_wait_ld_all(x);
#pragma unroll
        for (int u = 0; u < 32; u += 4) {
          const float4 w = *reinterpret_cast<const float4 *>(ij + c0 + u);
          v[u] = fminf(1.f, fabsf(__uint_as_float(x[u])) * inv_i * w.x);
          v[u + 1] = fminf(1.f, fabsf(__uint_as_float(x[u + 1])) * inv_i * w.y);
          v[u + 2] = fminf(1.f, fabsf(__uint_as_float(x[u + 2])) * inv_i * w.z);
          v[u + 3] = fminf(1.f, fabsf(__uint_as_float(x[u + 3])) * inv_i * w.w);
        }
        if (!inner) {
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            const int64_t j = j0 + c0 + u;
            if (!vrow || j >= a.n) v[u] = 0.f;
            else if (j == i) v[u] = 1.f;
          }
        }
      };
      // how many stored entries the value of column c stands for (0, 1, 2)
      auto wgt = [&](int c) -> float {
        const int64_t j = j0 + c;
        return (inner || md == 2 || j > i) ? 2.f : (j == i ? 1.f : 0.f);
      };
      if (md && a.out == 2) {
        float amax = 0.f;
#pragma unroll 1
        for (int c0 = 0; c0 < 128; c0 += 32) {
          float v[32];
          values(c0, v);
#pragma unroll
          for (int u = 0; u < 32; ++u)
            if (inner || wgt(c0 + u) > 0.f) amax = fmaxf(amax, v[u]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        float *fr = reinterpret_cast<float *>(rd);
        if (lane == 0) fr[q] = amax;
        dep_bar(half);
        const float dsc = e4m3_tile_scale(fmaxf(fmaxf(fr[0], fr[1]), fmaxf(fr[2], fr[3])));
        const float isc = 1.f / dsc;
        if (et == 0) {
          a.scales[(int64_t)ib * a.ld_scales + jt] = dsc;
          if (md == 2) a.scales[(int64_t)jt * a.ld_scales + ib] = dsc;
        }
        uint8_t *S8 = reinterpret_cast<uint8_t *>(a.S);
        uint8_t *Srow = S8 + i * a.lds;
#pragma unroll 1
        for (int c0 = 0; c0 < 128; c0 += 32) {
          float v[32];
          values(c0, v);
          uint32_t w[8];
          float part = 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            w[u] = (uint32_t)__nv_cvt_float2_to_fp8x2(
                       make_float2(v[4 * u] * isc, v[4 * u + 1] * isc), __NV_SATFINITE, __NV_E4M3) |
                   ((uint32_t)__nv_cvt_float2_to_fp8x2(
                        make_float2(v[4 * u + 2] * isc, v[4 * u + 3] * isc), __NV_SATFINITE,
                        __NV_E4M3)
                    << 16);
#pragma unroll
          for (int u = 0; u < 32; ++u) part = fmaf(wgt(c0 + u) * v[u], v[u], part);
          sq += (double)part;
          if (inner) {
            dep_store32(Srow + j0 + c0, a.w8, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
            // mirror: 4 x 4 byte transposes among the lanes 4 p + z, after
            // which lane 4 p + z holds column c0 + 4 u + z of rows 4 p ..
            // 4 p + 3, one word of S's row j
            const int z = lane & 3;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const uint32_t o1 = __shfl_xor_sync(0xffffffffu, w[u], 1);
              const uint32_t t1 = (z & 1) ? __byte_perm(o1, w[u], 0x7351) : __byte_perm(w[u], o1, 0x6240);
              const uint32_t o2 = __shfl_xor_sync(0xffffffffu, t1, 2);
              const uint32_t t2 = (z & 2) ? __byte_perm(o2, t1, 0x7632) : __byte_perm(t1, o2, 0x5410);
              *reinterpret_cast<uint32_t *>(S8 + (j0 + c0 + 4 * u + z) * a.lds + i - z) = t2;
            }
          } else if (vrow) {
            for (int u = 0; u < 32 && j0 + c0 + u < a.n; ++u) {
              const int64_t j = j0 + c0 + u;
              const uint8_t code = (uint8_t)(w[u >> 2] >> (8 * (u & 3)));
              if (md == 2 || j >= i) Srow[j] = code;
              if (md == 2 || j > i) S8[j * a.lds + i] = code;
            }
          }
        }
      } else if (md) {
#pragma unroll 1
        for (int c0 = 0; c0 < 128; c0 += 32) {
          float v[32];
          values(c0, v);
          if (a.out == 1) {
#pragma unroll
            for (int u = 0; u < 32; ++u) v[u] = __bfloat162float(__float2bfloat16_rn(v[u]));
          }
          float ph = 0.f, pl = 0.f;
          if (a.exact_sq) {
            // the stored values' squares summed as a float-float pair
            // (products split exactly by an FMA, Knuth's TwoSum on the high
            // parts): the run's sum is exact to about 2^-44 before it joins
            // the FP64 total, so ||S||^2 from here stands in for a pass over
            // the stored matrix
#pragma unroll
            for (int u = 0; u < 32; ++u) {
              const float ws = wgt(c0 + u) * v[u];  // weight 0, 1 or 2: exact
              const float pr = __fmul_rn(ws, v[u]), pe = fmaf(ws, v[u], -pr);
              const float t = __fadd_rn(ph, pr), bv = __fsub_rn(t, ph);
              pl = __fadd_rn(pl, __fadd_rn(__fadd_rn(__fsub_rn(ph, __fsub_rn(t, bv)),
                                                     __fsub_rn(pr, bv)), pe));
              ph = t;
            }
          } else {
#pragma unroll
            for (int u = 0; u < 32; ++u) ph = fmaf(wgt(c0 + u) * v[u], v[u], ph);
          }
          sq += (double)ph + (double)pl;
          if (a.out == 0) {
            float *S32 = reinterpret_cast<float *>(a.S);
            float *Srow = S32 + i * a.lds + j0 + c0;
            if (inner) {
              float *Scol = S32 + (j0 + c0) * a.lds + i;
#pragma unroll
              for (int u = 0; u < 32; u += 8)
                dep_store32(Srow + u, a.w8, __float_as_uint(v[u]), __float_as_uint(v[u + 1]),
                            __float_as_uint(v[u + 2]), __float_as_uint(v[u + 3]),
                            __float_as_uint(v[u + 4]), __float_as_uint(v[u + 5]),
                            __float_as_uint(v[u + 6]), __float_as_uint(v[u + 7]));
#pragma unroll
              for (int u = 0; u < 32; ++u) Scol[u * a.lds] = v[u];
            } else if (vrow) {
              for (int u = 0; u < 32 && j0 + c0 + u < a.n; ++u) {
                const int64_t j = j0 + c0 + u;
                if (md == 2 || j >= i) Srow[u] = v[u];
                if (md == 2 || j > i) S32[j * a.lds + i] = v[u];
              }
            }
          } else {
            uint16_t *S16 = reinterpret_cast<uint16_t *>(a.S);
            uint16_t *Srow = S16 + i * a.lds + j0 + c0;
            if (inner) {
              uint32_t w[16];
#pragma unroll
              for (int u = 0; u < 16; ++u)
                w[u] = (__float_as_uint(v[2 * u]) >> 16) | (__float_as_uint(v[2 * u + 1]) & 0xFFFF0000u);
#pragma unroll
              for (int u = 0; u < 16; u += 8)
                dep_store32(Srow + 2 * u, a.w8, w[u], w[u + 1], w[u + 2], w[u + 3], w[u + 4],
                            w[u + 5], w[u + 6], w[u + 7]);
              // mirror: 2 x 2 transposes among lane pairs, then lane z of a
              // pair holds column c0 + 2 u + z of the pair's two rows
              const int z = lane & 1;
#pragma unroll
              for (int u = 0; u < 16; ++u) {
                const uint32_t o = __shfl_xor_sync(0xffffffffu, w[u], 1);
                const uint32_t t = z ? __byte_perm(o, w[u], 0x7632) : __byte_perm(w[u], o, 0x5410);
                *reinterpret_cast<uint32_t *>(S16 + (j0 + c0 + 2 * u + z) * a.lds + i - z) = t;
              }
            } else if (vrow) {
              for (int u = 0; u < 32 && j0 + c0 + u < a.n; ++u) {
                const int64_t j = j0 + c0 + u;
                const uint16_t code = (uint16_t)(__float_as_uint(v[u]) >> 16);
                if (md == 2 || j >= i) Srow[u] = code;
                if (md == 2 || j > i) S16[j * a.lds + i] = code;
              }
            }
          }
        }
      }
      // the accumulator goes back to the MMAs
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[b]);
    }
    // the CTA's sum of squares: xor tree per warp, warps in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[56 + (warp - 2)] = sq;
  }
  fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[56 + w];
    a.sq[blockIdx.x] = s;
  }
  if (warp == 0 && lane == 0 && *abort_flag) {
    // copies issued but never consumed (bounded)
    for (int c = *consumed; c < issued; ++c) {
      int dummy = 0;
      mbar_wait(&full[c % kDepStages], (uint32_t)((c / kDepStages) & 1),
                reinterpret_cast<volatile int *>(&dummy), 100000000ull);
    }
  }
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tbase, 512);
  }
}

// fixed-order FP64 sum: contiguous runs per thread, runs in order
__global__ void __launch_bounds__(256) dep_sum_kernel(const double *x, int64_t m, double *out) {
  __shared__ double red[8];
  const int tid = threadIdx.x;
  const int64_t per = (m + 255) / 256;
  double s = 0.0;
  for (int64_t k = tid * per; k < m && k < (tid + 1) * per; ++k) s += x[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    *out = t;
  }
}

}  // namespace

cudaError_t launch_dependence(const float *Y, int64_t T, int64_t n, int64_t ldy, int center,
                              int out, void *S, int64_t lds, float *scales, int64_t ld_scales,
                              double *normS2, int *err, int *herr, cudaStream_t s,
                              bool exact_norm, void *ws, size_t ws_bytes) {
  const int Tp = (int)((T + 31) / 32 * 32);
  const int nib = (int)((n + 127) / 128), njb = (int)((n + 255) / 256);
  if (nib >= 65536 || njb >= 65536) return cudaErrorInvalidValue;
  int64_t tiles = 0;
  for (int g0 = 0; g0 < nib; g0 += kDepGroup) tiles += dep_group_tiles(g0, nib, njb);
  const int ntiles = (int)tiles;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int G = std::max(1, std::min(sms, ntiles));
  // one scratch block: P, then the CTA sums, the error word and 1 / (s_i sqrt(d_i))
  const size_t bytesP = sizeof(__half) * (size_t)n * 2 * Tp;  // a multiple of 128
  const size_t bytes = bytesP + sizeof(double) * (G + 1) + sizeof(float) * (size_t)n;
  // (stream-ordered memory goes back to the system at every synchronisation,
  // so it is mapped anew by each call: about 150 us)
  uint8_t *scratch = reinterpret_cast<uint8_t *>(ws);
  const bool own = !ws || ws_bytes < bytes;
  if (own) {
    e = cudaMallocAsync((void **)&scratch, bytes, s);
    if (e != cudaSuccess) return e;
  }
  __half *P = reinterpret_cast<__half *>(scratch);
  double *sq = reinterpret_cast<double *>(scratch + bytesP);
  if (!err) err = reinterpret_cast<int *>(sq + G);
  float *inv_d = reinterpret_cast<float *>(sq + G + 1);
  e = cudaMemsetAsync(err, 0, sizeof(int), s);
  dep_prep_kernel<<<(unsigned)((n + 31) / 32), dim3(32, kPrepY), 0, s>>>(Y, T, n, ldy, center, Tp,
                                                                         inv_d, P);
  CUtensorMap mP;
  if (e == cudaSuccess &&
      !make_map_2d(&mP, P, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, (uint64_t)2 * Tp, (uint64_t)n,
                   (uint64_t)2 * Tp * 2, kDepKC, 128, 64)) {
    e = cudaErrorInvalidValue;
  } else if (e == cudaSuccess) {
    e = cudaFuncSetAttribute(dep_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kDepSmem);
  }
  if (e == cudaSuccess) {
    DepArgs a{};
    a.n = n;
    a.Tp = Tp;
    a.natoms = Tp / kDepKC;
    a.nib = nib;
    a.njb = njb;
    a.ntiles = ntiles;
    a.inv_d = inv_d;
    a.S = S;
    a.lds = lds;
    a.out = out;
    a.scales = scales;
    a.ld_scales = ld_scales;
    a.sq = sq;
    a.err = err;
    a.exact_sq = exact_norm ? 1 : 0;
    a.w8 = reinterpret_cast<uintptr_t>(S) % 32 == 0 && (lds * (out == 0 ? 4 : out == 1 ? 2 : 1)) % 32 == 0;
    dep_gemm_kernel<<<(unsigned)G, kDepThreads, kDepSmem, s>>>(mP, a);
    if (normS2) dep_sum_kernel<<<1, 256, 0, s>>>(sq, G, normS2);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  }
  const cudaError_t e2 = own ? cudaFreeAsync(scratch, s) : cudaSuccess;
  return e == cudaSuccess ? e2 : e;
}

}  // namespace symnmf
