// FP32 FMA product of a 128-row tile of S with H (n x KP), the core of the
// exact-FP32 product (k_prod_simt.cu) and of the objective without a handle
// (k_noalloc.cu).  It takes S of any pitch and alignment.
//
// Bound by the FMA rate together with the shared-memory reads that feed it: a
// thread holds 8 rows x 8 columns (KP = 8: 4 columns), so two columns of S
// cost 8 reads of 8 bytes and 4 of 16 for 128 FMAs (64 two-wide ones), about
// the balance of the two pipes.  KP / 8 x 16 threads cover the tile; the 256
// threads split each 32-column chunk among NG such groups, whose sums are
// added in group order at the end.  FP32 chunks arrive by cp.async in a ring
// of four (one chunk ahead in registers waited on HBM's latency: n = 10000,
// KP = 32 301 -> 244 us; rows on 16-byte boundaries in 16-byte pieces: 188 us);
// BF16 and FP8 entries, of any byte alignment, are loaded one chunk ahead into
// registers and widened there (staged as aligned words and widened in shared
// memory: n = 5001, KP = 32 60 -> 77 us).
#pragma once
#include "epi_common.cuh"

namespace symnmf {

// (d.x, d.y) += a * (b.x, b.y), two FP32 FMAs in one instruction
__device__ __forceinline__ void fma2(float2 &d, float a, float2 b) {
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %2};\n mov.b64 y, {%3, %4};\n mov.b64 z, {%0, %1};\n"
      " fma.rn.f32x2 z, x, y, z;\n mov.b64 {%0, %1}, z;\n}\n"
      : "+f"(d.x), "+f"(d.y)
      : "f"(a), "f"(b.x), "f"(b.y));
}

template <int DT, int KP>
struct Simt {
  static constexpr int BK = 32;                  // columns of S per chunk
  static constexpr int RING = 4;
  static constexpr int TN = KP == 8 ? 4 : 8;     // columns of H per thread
  static constexpr int CG = KP / TN;
  static constexpr int TPG = 16 * CG;            // threads per group
  static constexpr int NG = 256 / TPG;           // groups
  static constexpr int KG = BK / NG;             // columns of a chunk per group
  static constexpr int LD = BK + 4;              // FP32 rows: 16-byte aligned, no bank conflicts
  static constexpr int S_WORDS = 128 * LD;       // FP32 tile
  static constexpr int BUFS = DT == 0 ? RING : 2;
  static constexpr int H_WORDS = BK * KP;
  static constexpr int STAGE = S_WORDS + H_WORDS;  // S chunk, H chunk
  static constexpr int WORDS = BUFS * STAGE;
  static constexpr size_t SMEM = sizeof(float) * WORDS;
  static_assert(NG == (KP <= 16 ? 8 : 128 / KP), "simt_split");
  static_assert(KG % 2 == 0 && 128 * KP <= WORDS && STAGE % 4 == 0, "");
};

// 4 bytes to shared memory, the first `bytes` (0..4) from src and zeros after
__device__ __forceinline__ void cp_async4(float *dst, const void *src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}

// the same for 16 bytes (0..16 from src), both addresses on 16-byte boundaries
__device__ __forceinline__ void cp_async16(float *dst, const void *src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}

// sm: Simt<DT, KP>::SMEM bytes on a 16-byte boundary.  Rows r0 .. r0 + 127 of
// S times H over column tiles [cb, ce) of the list (col_list nullptr: in
// order); H: n rows of pitch ldh, columns from k on read as 0.  On return
// sm[r * KP + c] holds the tile's product (every thread may read it).
// scales: FP8, the tile scales of this row tile.
template <int DT, int KP>
__device__ __forceinline__ void simt_tile(float *sm, const void *S, int64_t lds, int64_t n,
                                          int64_t r0, const float *H, int64_t ldh, int k,
                                          const int *col_list, int cb, int ce,
                                          const float *scales) {
  using C = Simt<DT, KP>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid / C::TPG, t = tid % C::TPG, cg = t % C::CG, rg = t / C::CG;
  float2 acc[8][C::TN / 2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < C::TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int rows = (int)(n - r0 < kTileRows ? n - r0 : kTileRows);
  const int nq = (ce - cb) * 4;
  constexpr int HV = C::BK * KP / 256;
  // lane = column of the chunk, rows warp, warp + 8, ...
  auto col0 = [&](int q) -> int64_t {  // first column of chunk q
    const int ci = cb + (q >> 2);
    return (int64_t)(col_list ? col_list[ci] : ci) * kTileRows + (q & 3) * C::BK;
  };
  // FP32: chunk q into its stage of the ring, 16 bytes at a time where every
  // row of S (H) starts on such a boundary
  const bool svec = reinterpret_cast<uintptr_t>(S) % 16 == 0 && lds % 4 == 0;
  const bool hvec = reinterpret_cast<uintptr_t>(H) % 16 == 0 && ldh == KP && k == KP;
  auto issue = [&](int q) {
    if (q < nq) {
      const int64_t c0 = col0(q);
      const int cols = (int)(n - c0 < C::BK ? n - c0 : C::BK);  // may be <= 0
      float *st = sm + (q % C::RING) * C::STAGE, *hs = st + C::S_WORDS;
      const float *Sf = reinterpret_cast<const float *>(S);
      if (svec) {  // 4 columns per thread, rows tid / 8, + 32, ...
        const int c4 = 4 * (tid & 7);
        const int bytes = cols - c4 >= 4 ? 16 : cols > c4 ? 4 * (cols - c4) : 0;
        const float *p = Sf + (r0 + (tid >> 3)) * lds + c0 + c4;
#pragma unroll
        for (int i = 0; i < 4; ++i, p += 32 * lds) {
          const int r = (tid >> 3) + 32 * i;
          const int nb = r < rows ? bytes : 0;
          cp_async16(st + r * C::LD + c4, nb ? (const void *)p : S, nb);
        }
      } else {
        const float *p = Sf + (r0 + warp) * lds + c0 + lane;
#pragma unroll 4
        for (int r = warp; r < 128; r += 8, p += 8 * lds) {
          const bool in = r < rows && lane < cols;
          cp_async4(st + r * C::LD + lane, in ? (const void *)p : S, in ? 4 : 0);
        }
      }
      if (hvec) {
        for (int e = 4 * tid; e < C::H_WORDS; e += 1024) {
          const int r = e / KP, c = e % KP;
          cp_async16(hs + e, r < cols ? H + (c0 + r) * KP + c : H, r < cols ? 16 : 0);
        }
      } else {
#pragma unroll
        for (int i = 0; i < HV; ++i) {
          const int e = tid + 256 * i, r = e / KP, c = e % KP;
          const bool in = r < cols && c < k;
          cp_async4(hs + e, in ? H + (c0 + r) * ldh + c : H, in ? 4 : 0);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // BF16, FP8: chunk q into registers, from there into buffer q % 2
  constexpr int NV = DT == 0 ? 1 : 16, NH = DT == 0 ? 1 : HV;
  float sv[NV], hv[NH];
  auto load = [&](int q) {
    const int64_t c0 = col0(q), at = (r0 + warp) * lds + c0 + lane;
    float sc = 1.f;
    if constexpr (DT == 2) sc = __ldg(scales + c0 / kTileRows);
    if (rows == kTileRows && c0 + C::BK <= n) {
      int64_t x = at;
#pragma unroll
      for (int i = 0; i < NV; ++i, x += 8 * lds) sv[i] = s_entry<DT>(S, x);
    } else {
#pragma unroll
      for (int i = 0; i < NV; ++i)
        sv[i] = (c0 + lane < n && warp + 8 * i < rows) ? s_entry<DT>(S, at + (int64_t)(8 * i) * lds) : 0.f;
    }
    if constexpr (DT == 2) {
#pragma unroll
      for (int i = 0; i < NV; ++i) sv[i] *= sc;
    }
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      const int e = tid + 256 * i, r = e / KP, c = e % KP;
      hv[i] = (c0 + r < n && c < k) ? __ldg(H + (c0 + r) * ldh + c) : 0.f;
    }
  };
  auto store = [&](int q) {
    float *st = sm + (q & 1) * C::STAGE, *hs = st + C::S_WORDS;
#pragma unroll
    for (int i = 0; i < NV; ++i) st[(warp + 8 * i) * C::LD + lane] = sv[i];
#pragma unroll
    for (int i = 0; i < NH; ++i) hs[tid + 256 * i] = hv[i];
  };
  if constexpr (DT == 0) {
#pragma unroll
    for (int q = 0; q < C::RING - 1; ++q) issue(q);
  } else if (nq > 0) {
    load(0);
    store(0);
  }
  for (int q = 0; q < nq; ++q) {
    if constexpr (DT == 0) asm volatile("cp.async.wait_group %0;" ::"n"(C::RING - 2) : "memory");
    __syncthreads();  // chunk q is here, and every thread is done with q - 1
    if constexpr (DT == 0) issue(q + C::RING - 1);
    else if (q + 1 < nq) load(q + 1);
    const float *Ss = sm + (q % C::BUFS) * C::STAGE, *Hs = Ss + C::S_WORDS;
#pragma unroll
    for (int k2 = 0; k2 < C::KG; k2 += 2) {
      const int kk = grp * C::KG + k2;
      float a[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 v = *reinterpret_cast<const float2 *>(Ss + (rg + 16 * i) * C::LD + kk);
        a[i][0] = v.x;
        a[i][1] = v.y;
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        float2 b[C::TN / 2];
#pragma unroll
        for (int j = 0; j < C::TN; j += 4) {
          const float4 v = *reinterpret_cast<const float4 *>(Hs + (kk + x) * KP + cg * C::TN + j);
          b[j / 2] = make_float2(v.x, v.y);
          b[j / 2 + 1] = make_float2(v.z, v.w);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < C::TN / 2; ++j) fma2(acc[i][j], a[i][x], b[j]);
      }
    }
    if (DT != 0 && q + 1 < nq) store(q + 1);
  }
  __syncthreads();
  // groups in order into sm[r * KP + c]
#pragma unroll 1
  for (int g = 0; g < C::NG; ++g) {
    if (grp == g) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < C::TN; j += 4) {
          float4 *p = reinterpret_cast<float4 *>(sm + (rg + 16 * i) * KP + cg * C::TN + j);
          float4 v = make_float4(acc[i][j / 2].x, acc[i][j / 2].y, acc[i][j / 2 + 1].x, acc[i][j / 2 + 1].y);
          if (g > 0) {
            const float4 o = *p;
            v = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
          }
          *p = v;
        }
    }
    __syncthreads();
  }
}

// The number of column shares per row tile that ends soonest: `rows` CTAs per
// share on `slots` places, each share ceil(cols / s) column tiles long plus
// about one for its start and end.  A share's FP32 sums run over 1 / NG of its
// columns in a row; there are enough shares (of the `most` there may be) that
// none is longer than with `parts` shares and one group.  Without that limit the
// rule took a single share for 297 tiles at KP = 64: chains of 19008 FMAs where
// eight shares had 4864, and an objective off by 2e-8 of the trace, not 6e-10.
inline int simt_split(int rows, int cols, int kp, int slots, int most, int parts) {
  const int groups = kp <= 16 ? 8 : 128 / kp;  // Simt<DT, KP>::NG
  const int64_t longest = (int64_t)groups * ((cols + parts - 1) / parts);
  int best = 0;
  int64_t cost = INT64_MAX;
  for (int s = 1; s <= most && s <= cols; ++s) {
    if ((cols + s - 1) / s > longest && s < most) continue;
    const int64_t waves = ((int64_t)rows * s + slots - 1) / slots;
    const int64_t c = waves * ((cols + s - 1) / s + 1);
    if (c < cost) {
      cost = c;
      best = s;
    }
  }
  return best > 0 ? best : 1;
}

}  // namespace symnmf
