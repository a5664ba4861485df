// Per-tile epilogue of one solver iteration and the fixed-order reductions.
//
// For each 128-row tile I the epilogue forms the gradient rows
//   g_I = 4 (H_I Gram_t - (S H)_I)                          (Sec. 2.1)
// or the Row-SVRG / Block-SVRG estimates (Sec. 5.1; appendix), applies the
// AdaGrad or RMSprop update with the max(0, .) projection (appendix,
// Family 3; Sec. 2.4 "Projected space") into the other H buffer, writes the
// bf16 hi/lo MMA copy of the new rows, and produces the per-tile partials
// tr_I = sum H_I * (S H)_I (Eq. 2), ||grad_proj||^2_I (Eq. 6), sum(G)_I, the
// NaN/Inf count and the Gram partial H'_I^T H'_I.  Within a tile sums are
// FP32 in a fixed order; across tiles they are FP64 in tile order
// (launch_reduce), so every result is bit-reproducible run to run.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "../../include/symnmf.h"
#include "epi_common.cuh"
#include "tile_tail.cuh"
#include "symnmf_internal.h"

namespace symnmf {
namespace {

__device__ __forceinline__ double block_sum(double v, double *sh) {
  // fixed-order: xor tree within the warp, then warp 0 adds warps in order
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < nw; ++i) r += sh[i];
    sh[32] = r;
  }
  __syncthreads();
  return sh[32];
}

// A thread's 4 columns (from 4 cg) of RP rows (rg, rg + RS, ...): the rows of
// a warp's load or store of one of them are contiguous.
template <int KP>
struct EpiK {
  static constexpr int T = KP == 8 ? 256 : 512;
  static constexpr int CG = KP / 4;
  static constexpr int RS = T / CG;
  static constexpr int RP = kTileRows / RS;
  static constexpr size_t SMEM = sizeof(float) * (kTileRows * (KP + 1) + 3 + 2 * KP * KP);
};

// acc = (rows of Hs) M for the thread's entries, M (KP x KP) in shared
// memory, summed over d in order: RP scalar and one 16-byte read per 4 RP FMAs
template <int KP>
__device__ __forceinline__ void rows_times(const float (*Hs)[KP + 1], const float *M, int rg,
                                           int cg, float (&acc)[EpiK<KP>::RP][4]) {
  constexpr int RP = EpiK<KP>::RP, RS = EpiK<KP>::RS;
#pragma unroll
  for (int i = 0; i < RP; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll 8
  for (int d = 0; d < KP; ++d) {
    const float4 m = *reinterpret_cast<const float4 *>(M + d * KP + 4 * cg);
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const float h = Hs[rg + i * RS][d];
      acc[i][0] = fmaf(h, m.x, acc[i][0]);
      acc[i][1] = fmaf(h, m.y, acc[i][1]);
      acc[i][2] = fmaf(h, m.z, acc[i][2]);
      acc[i][3] = fmaf(h, m.w, acc[i][3]);
    }
  }
}

// the thread's entries of the summed partials of row position p, slots in
// order (part_range), four loads in flight
template <int KP>
__device__ __forceinline__ void parts_of(const float *P, int nsplit, int skG, int ncols, int nlist,
                                         int p, int rg, int cg, float (&v)[EpiK<KP>::RP][4]) {
  constexpr int RP = EpiK<KP>::RP, RS = EpiK<KP>::RS;
  int64_t b0, b1;
  part_range(p, skG, ncols, nlist, b0, b1);
  const int64_t first = skG > 0 ? b0 + p : p, step = skG > 0 ? 1 : nlist;
  const int count = skG > 0 ? (int)(b1 - b0) + 1 : nsplit;
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const float *src = P + (first * kTileRows + rg + i * RS) * KP + 4 * cg;
    const int64_t st = step * kTileRows * KP;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q0 = 0; q0 < count; q0 += 4) {
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = q0 + u < count ? __ldcg(reinterpret_cast<const float4 *>(src + (q0 + u) * st))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s[0] += x[u].x;
        s[1] += x[u].y;
        s[2] += x[u].z;
        s[3] += x[u].w;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) v[i][j] = s[j];
  }
}

// Stand-alone tile epilogue, one CTA per 128-row tile.  Bound by latency and
// shared-memory reads: the H Gram products are formed in 4-column register
// blocks and the state moves in 16-byte rows.  Multiply-adds are written out,
// so that every padded rank rounds the same way (restarts in one handle are
// bit-equal to separate handles).  n = 50000, kp = 64, block mode 337 -> 89
// us; n = 5001, kp = 32 33 -> 11; n = 3001, kp = 16 19 -> 8.9 (two shared
// reads per FMA and FP64 block sums before; exact warp sums instead of
// float-float trees take 0.6 us off the last).
template <int KP>
__global__ void __launch_bounds__(EpiK<KP>::T, KP == 64 ? 1 : 1024 / EpiK<KP>::T)
    epilogue_kernel(EpiArgs a) {
  using K = EpiK<KP>;
  constexpr int RP = K::RP, RS = K::RS, T = K::T;
  extern __shared__ __align__(16) float smem_epi[];
  float(*Hs)[KP + 1] = reinterpret_cast<float(*)[KP + 1]>(smem_epi);
  float *G1 = smem_epi + (kTileRows * (KP + 1) + 3) / 4 * 4, *G2 = G1 + KP * KP;
  __shared__ double red[T / 32][4];
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int cg = tid % K::CG, rg = tid / K::CG, c0 = 4 * cg;
  const int64_t r0 = (int64_t)tile * kTileRows;
  const int rows = (int)((a.n - r0) < kTileRows ? (a.n - r0) : kTileRows);
  const bool block = (a.mode == MODE_BLOCK);
  const bool rms = (a.method == SYMNMF_RMSPROP), admm = (a.method == SYMNMF_ADMM);
  int p1 = -1, p2 = -1, p3 = -1;
  if (a.mode == MODE_FULL || a.mode == MODE_GRAD_ONLY) {
    p1 = tile;
  } else {
    p1 = a.pos1[tile];
    if (block) {
      p2 = a.pos2[tile];
      p3 = a.pos3[tile];
    }
  }
  const int64_t base = (r0 + rg) * KP + c0;  // entry (i, j): base + i RS KP + j
  auto ld4 = [&](const float *src, int i) -> float4 {
    return rg + i * RS < rows ? __ldcg(reinterpret_cast<const float4 *>(src + base + (int64_t)i * RS * KP))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto st4 = [&](float *dst, int i, const float (&x)[4]) {
    if (rg + i * RS < rows)
      *reinterpret_cast<float4 *>(dst + base + (int64_t)i * RS * KP) = make_float4(x[0], x[1], x[2], x[3]);
  };
  float h[RP][4], g[RP][4], pv[RP][4];
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const float4 v = ld4(a.H, i);
    h[i][0] = v.x;
    h[i][1] = v.y;
    h[i][2] = v.z;
    h[i][3] = v.w;
  }
  const float *g1src = block ? a.gramJ : a.gram;
  for (int e = tid; e < KP * KP / 4; e += T) {
    reinterpret_cast<float4 *>(G1)[e] = reinterpret_cast<const float4 *>(g1src)[e];
    if (block) reinterpret_cast<float4 *>(G2)[e] = reinterpret_cast<const float4 *>(a.gramI)[e];
  }
#pragma unroll
  for (int i = 0; i < RP; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      Hs[rg + i * RS][c0 + j] = h[i][j];
      pv[i][j] = 0.f;
      g[i][j] = 0.f;
    }
  // block mode: a list whose column list was empty holds no partials; list 3
  // holds what lists 1 and 2 share
  float rv[RP][4];
  const bool has3 = p3 >= 0 && a.ncols3 > 0;
  if (has3) parts_of<KP>(a.R, a.nsplit3, a.skG3, a.ncols3, a.n3, p3, rg, cg, rv);
  if (p1 >= 0) {
    if (!block || a.ncols1 > 0)
      parts_of<KP>(a.P, a.nsplit, a.skG1, a.ncols1, a.n1, p1, rg, cg, pv);
    if (has3) {
#pragma unroll
      for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) pv[i][j] = rv[i][j] + pv[i][j];
    }
  }
  __syncthreads();  // Hs, G1 and G2 are complete

  // gradient estimate
  float tr = 0.f, kkt2 = 0.f, sumA = 0.f;
  int nonfin = 0;
  if (p1 >= 0) {
    float hg[RP][4];
    rows_times<KP>(Hs, G1, rg, cg, hg);
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        g[i][j] = __fmul_rn(a.coef, hg[i][j] - pv[i][j]);
        if (rg + i * RS < rows && c0 + j < a.k) tr = fmaf(h[i][j], pv[i][j], tr);
      }
  }
  if (p2 >= 0) {
    float hg[RP][4], qv[RP][4];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) qv[i][j] = 0.f;
    if (a.ncols2 > 0) parts_of<KP>(a.Q, a.nsplit2, a.skG2, a.ncols2, a.n2, p2, rg, cg, qv);
    rows_times<KP>(Hs, G2, rg, cg, hg);
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float q = has3 ? rv[i][j] + qv[i][j] : qv[i][j];
        g[i][j] = fmaf(a.coef, hg[i][j] - q, g[i][j]);
      }
  }
  if (p1 < 0 && p2 < 0) {
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const float4 v = ld4(a.mu, i);
      g[i][0] = v.x;
      g[i][1] = v.y;
      g[i][2] = v.z;
      g[i][3] = v.w;
    }
  }
  // outputs of the gradient
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const bool in = rg + i * RS < rows;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!in || c0 + j >= a.k) g[i][j] = 0.f;
      const float pg = (h[i][j] > 0.f) ? g[i][j] : fminf(0.f, g[i][j]);
      kkt2 = fmaf(pg, pg, kkt2);
      if (!isfinite(g[i][j])) ++nonfin;
      if (a.gcaller && in && c0 + j < a.k)
        a.gcaller[(r0 + rg + i * RS) * a.k + c0 + j] = g[i][j];
    }
    if (a.gout) st4(a.gout, i, g[i]);
    if (a.store_mu) st4(a.mu, i, g[i]);
  }
  if (a.update) {
    __syncthreads();  // every thread has read H_t from Hs
    float xv[RP][4];
    if (admm) {
      // H = rhs (2 W^T W + rho I)^-1 with rhs = 2 (S W) + rho (W - U), W' =
      // [H + U]_+, U' = U + H - W' (appendix, Family 6)
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        const float4 u = ld4(a.A, i);
        const float u4[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          Hs[rg + i * RS][c0 + j] = (rg + i * RS < rows && c0 + j < a.k)
                                        ? fmaf(a.rho, h[i][j] - u4[j], 2.f * pv[i][j])
                                        : 0.f;
      }
      for (int e = tid; e < KP * KP / 4; e += T)
        reinterpret_cast<float4 *>(G1)[e] = reinterpret_cast<const float4 *>(a.minv)[e];
      __syncthreads();
      rows_times<KP>(Hs, G1, rg, cg, xv);
      __syncthreads();  // every thread has read the right-hand sides
    }
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const float4 av4 = ld4(a.A, i);
      const float4 mv4 = rms ? ld4(a.M, i) : make_float4(0.f, 0.f, 0.f, 0.f);
      float av[4] = {av4.x, av4.y, av4.z, av4.w}, mv[4] = {mv4.x, mv4.y, mv4.z, mv4.w}, hn[4];
      const bool in = rg + i * RS < rows;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        hn[j] = 0.f;
        if (in && c0 + j < a.k) {
          const float gv = g[i][j];
          float x;
          if (admm) {
            x = xv[i][j] + av[j];
            hn[j] = (x > 0.f) ? x : 0.f;
            av[j] = x - hn[j];
            sumA += av[j];
          } else {
            if (rms) {
              av[j] = fmaf(a.alpha, av[j], __fmul_rn(1.f - a.alpha, __fmul_rn(gv, gv)));
              mv[j] = fmaf(a.mom, mv[j], adaptive_step(a.eta * gv, av[j], a.eps));
              x = h[i][j] - mv[j];
            } else {
              av[j] = fmaf(gv, gv, av[j]);
              x = __fsub_rn(h[i][j], adaptive_step(a.eta * gv, av[j], a.eps));
            }
            sumA += av[j];
            hn[j] = (x > 0.f) ? x : 0.f;
          }
        }
        Hs[rg + i * RS][c0 + j] = hn[j];
      }
      st4(a.A, i, av);
      if (rms) st4(a.M, i, mv);
      st4(a.Hn, i, hn);
    }
    __syncthreads();  // Hs holds the tile of H_{t+1}
    tile_tail<KP, T>(Hs, r0, a.Btn, a.bt_fmt, a.ldb, a.gram_part, tile);
  }
  // tile scalars: exact warp sums (FP64 trees would take 15 slow additions a
  // lane), warps in order in FP64
  const float sc[3] = {tr, kkt2, sumA};
  const unsigned nf = __reduce_add_sync(0xffffffffu, (unsigned)nonfin);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double v = warp_sum64(sc[i]);
    if ((tid & 31) == 0) red[tid >> 5][i] = v;
  }
  if ((tid & 31) == 0) red[tid >> 5][3] = (double)nf;
  __syncthreads();
  if (tid < 4 && a.slots) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < T / 32; ++w) s += red[w][tid];
    a.slots[(int64_t)tile * kSlotStride + tid] = s;
  }
}

template <int KP>
__global__ void __launch_bounds__(256) prepare_kernel(const float *H, int64_t n, void *Bt,
                                                      int bt_fmt, int64_t ldb, float *gram_part) {
  __shared__ float Hn[kTileRows][KP + 1];
  const int tile = blockIdx.x;
  const int64_t r0 = (int64_t)tile * kTileRows;
  const int rows = (int)((n - r0) < kTileRows ? (n - r0) : kTileRows);
  for (int e = threadIdx.x; e < kTileRows * KP; e += blockDim.x) {
    const int r = e / KP, c = e % KP;
    Hn[r][c] = (r < rows) ? H[(r0 + r) * KP + c] : 0.f;
  }
  __syncthreads();
  tile_tail<KP, 256>(Hn, r0, Bt, bt_fmt, ldb, gram_part, tile);
}

// Fixed-order FP64 reduction of an iteration's per-tile results (the 4
// scalar slots and the kp x kp Gram partial of every tile).  Block 0 forms the
// iteration record f = ||S||^2 - 2 tr + ||Gram_t||^2 (Eq. 2); every other
// block reduces 16 Gram entries, 16 threads to an entry: thread j adds the
// tiles j, j + 16, ... in order, the 16 sums are added in order.
//
// Latency-bound and on the path of every iteration: the next step's tile
// epilogues wait for it, and its blocks hold the SMs they run on, where the
// next step's CTAs (all registers of an SM) then start late.  It is launched
// early (programmatic dependent launch) and lets the next step launch once
// the step before it has completed: that step's rows of H are what the next
// step's stream reads before its own griddepcontrol.wait.  One level with a
// wide split instead of chunks of 32 tiles and a last arriver: an AdaGrad
// iteration at n = 512, k = 8 takes 18.9 instead of 26.8 us, at n = 20000,
// k = 32 290.6 instead of 294.2 us, k = 64 BF16 216 instead of 223 us.
template <int KP>
__global__ void __launch_bounds__(256) reduce_iter_kernel(ReduceArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ double red[256];
  const int tid = threadIdx.x;
  if (blockIdx.x > 0) {
    const int le = tid & 15, j = tid >> 4;
    const int e = ((int)blockIdx.x - 1) * 16 + le;
    const float *src = a.gram_part + e;
    double v = 0.0;
    for (int t0 = j; t0 < a.ntiles; t0 += 128) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        x[u] = t0 + 16 * u < a.ntiles ? __ldcg(src + (int64_t)(t0 + 16 * u) * KP * KP) : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (t0 + 16 * u < a.ntiles) v += (double)x[u];
    }
    red[tid] = v;
    __syncthreads();
    if (tid < 16) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < 16; ++i) s += red[i * 16 + tid];
      // restarts concatenated along N: only the diagonal kb x kb blocks
      if (a.kb > 0 && e / KP / a.kb != e % KP / a.kb) s = 0.0;
      a.gram64_next[e] = s;
      a.gram32_next[e] = (float)s;
    }
    return;
  }
  if (!a.rec || !a.slots) return;
  // the record: slot s of tiles l, l + 64, ... in thread 4 l + s, xor trees
  // over the threads of a slot in a warp, then the 8 warps in order
  double v = 0.0, g2 = 0.0;
  for (int t = tid >> 2; t < a.ntiles; t += 64) v += a.slots[(int64_t)t * kSlotStride + (tid & 3)];
  if (a.gram64_cur)
    for (int i = tid; i < KP * KP; i += 256) g2 = fma(a.gram64_cur[i], a.gram64_cur[i], g2);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (o >= 4) v += __shfl_xor_sync(0xffffffffu, v, o);
    g2 += __shfl_xor_sync(0xffffffffu, g2, o);
  }
  const int w = tid >> 5, l = tid & 31;
  if (l < 4) red[w * 5 + l] = v;
  if (l == 4) red[w * 5 + 4] = g2;
  __syncthreads();
  if (tid < 5) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += red[i * 5 + tid];
    red[64 + tid] = s;
  }
  __syncthreads();
  if (tid == 0) {
    const double *sc = red + 64;
    DevRecord rc;
    rc.t = a.t;
    rc.tr = sc[0];
    rc.gram2 = sc[4];
    rc.f = a.normS2 - 2.0 * sc[0] + sc[4];
    rc.E = rc.f / a.normS2;
    rc.kkt = sqrt(sc[1]) / ((double)a.n * (double)a.k);
    rc.sumA = sc[2];
    rc.nonfinite = (int)sc[3];
    rc.full = a.full;
    *a.rec = rc;
  }
}

// Gram of the tiles of a list, 16 threads to an entry as in reduce_iter_kernel
// (one thread per entry: 391 tiles at kp = 64 47 us, now 17).  It runs in the
// tail of the products before it, of which it needs nothing, and waits for
// them before it ends, as the epilogue that follows needs both.
template <int KP>
__global__ void __launch_bounds__(256) gram_subset_kernel(const float *gram_part, const int *l1,
                                                          int n1, const int *l2, int n2,
                                                          float *o1, float *o2, int kb) {
  __shared__ double red[256];
  const int tid = threadIdx.x, le = tid & 15, j = tid >> 4;
  const int e = (int)blockIdx.x * 16 + le;
  const int *l = blockIdx.y == 0 ? l1 : l2;
  const int m = blockIdx.y == 0 ? n1 : n2;
  double v = 0.0;
  for (int i0 = j; i0 < m; i0 += 128) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      x[u] = i0 + 16 * u < m ? __ldcg(gram_part + (int64_t)__ldg(l + i0 + 16 * u) * KP * KP + e) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + 16 * u < m) v += (double)x[u];
  }
  red[tid] = v;
  __syncthreads();
  if (tid >= 16) return;
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 16; ++i) s += red[i * 16 + tid];
  if (kb > 0 && e / KP / kb != e % KP / kb) s = 0.0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  (blockIdx.y == 0 ? o1 : o2)[e] = (float)s;
}

// ||S||_F^2: one warp per row, runs of 64 entries in FP32 words (row_sumsq_lane),
// runs and rows in FP64.  FP32 is bound by HBM (n = 12000: 111 us, 5.2 TB/s),
// BF16 and FP8 by the operations per entry (106 and 48 us); a conversion and a
// multiply-add per entry in FP64 bounded all of them by the FP64 pipe (555 to
// 1068 us).
template <int DT>
__global__ void __launch_bounds__(256, 4) norm_s2_kernel(const void *S, int64_t n, int64_t lds,
                                                      const float *scales, int64_t ld_scales,
                                                      bool vec, double *partials) {
  __shared__ double red[40];
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * 8;
  double acc = 0.0;
  for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < n; r += warps)
    acc += row_sumsq_lane<DT>(S, r * lds, n, scales + (r / kTileRows) * ld_scales, vec, lane);
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// fixed-order sum of m values: contiguous runs per thread, then the block's
// order (one thread adding them all took 31 us for 608 values)
__global__ void __launch_bounds__(256) sum_array_kernel(const double *x, int m, int stride, int off,
                                                        double *out) {
  __shared__ double red[40];
  const int per = (m + 255) / 256;
  double s = 0.0;
  for (int i = threadIdx.x * per; i < m && i < (int)(threadIdx.x + 1) * per; ++i)
    s += x[(int64_t)i * stride + off];
  s = block_sum(s, red);
  if (threadIdx.x == 0) *out = s;
}

// caller row-major n x k -> n x kp over all tile rows (pads zeroed)
__global__ void pack_kernel(const float *src, float *dst, int64_t n, int k, int kp) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t tiles = (n + kTileRows - 1) / kTileRows;
  if (e >= tiles * kTileRows * kp) return;
  const int64_t r = e / kp;
  const int c = (int)(e % kp);
  dst[e] = (c < k && r < n) ? src[r * k + c] : 0.f;
}

__global__ void unpack_kernel(const float *src, float *dst, int64_t n, int k, int kp) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * k) return;
  const int64_t r = e / k;
  const int c = (int)(e % k);
  dst[e] = src[r * kp + c];
}

// radix select of the lower median of g^2 over columns c0 .. c0 + kw - 1
// (FP32 bit patterns of non-negative floats order like unsigned integers);
// three passes of 11, 11, 10 bits
__global__ void __launch_bounds__(256) hist_kernel(const float *g, int64_t n, int c0, int kw,
                                                   int kp, int shift, int nbits,
                                                   const unsigned *sel, unsigned *hist) {
  __shared__ unsigned sh[2048];
  const int nb = 1 << nbits;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const unsigned mask = sel[0], val = sel[1];
  const int64_t total = n * kw;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / kw;
    const int c = c0 + (int)(e % kw);
    const float x = g[r * kp + c];
    const float x2 = x * x;
    const unsigned u = __float_as_uint(x2);
    if ((u & mask) == val) atomicAdd(&sh[(u >> shift) & (nb - 1)], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x)
    if (sh[i]) atomicAdd(&hist[i], sh[i]);
}

__global__ void select_kernel(unsigned *hist, int shift, int nbits, unsigned *sel, float *out,
                              int last) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int nb = 1 << nbits;
  unsigned rank = sel[2];
  unsigned cum = 0;
  int b = 0;
  for (; b < nb; ++b) {
    if (cum + hist[b] > rank) break;
    cum += hist[b];
  }
  if (b >= nb) b = nb - 1;
  sel[2] = rank - cum;
  sel[0] |= (unsigned)(nb - 1) << shift;
  sel[1] |= (unsigned)b << shift;
  for (int i = 0; i < nb; ++i) hist[i] = 0u;
  if (last) *out = __uint_as_float(sel[1]);
}

__global__ void init_sel_kernel(unsigned *sel, unsigned rank, unsigned *hist) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sel[0] = 0u;
    sel[1] = 0u;
    sel[2] = rank;
  }
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) hist[i] = 0u;
}

// A = c max(g^2, median) on columns c0 .. c0 + kw - 1; slot 2 of each tile
// gets the tile's sum of the reset entries
template <int KP>
__global__ void __launch_bounds__(256) reset_kernel(float *A, const float *g, const float *med,
                                                    float c, int64_t n, int c0, int kw,
                                                    double *slots) {
  __shared__ double red[40];
  const int tile = blockIdx.x;
  const int64_t r0 = (int64_t)tile * kTileRows;
  const int rows = (int)((n - r0) < kTileRows ? (n - r0) : kTileRows);
  const float m = *med;
  float s = 0.f;
  for (int e = threadIdx.x; e < kTileRows * KP; e += blockDim.x) {
    const int r = e / KP, cc = e % KP;
    if (r < rows && cc >= c0 && cc < c0 + kw) {
      const int64_t gi = (r0 + r) * KP + cc;
      const float x = g[gi];
      const float v = c * fmaxf(x * x, m);
      A[gi] = v;
      s += v;
    }
  }
  const double tot = block_sum((double)s, red);
  if (threadIdx.x == 0) slots[(int64_t)tile * kSlotStride + 2] = tot;
}

// ADMM (appendix, Family 6): the H-update solves H (2 W^T W + rho I) =
// 2 S W + rho (W - U) row by row; every row shares the kp x kp matrix, so
// its inverse is formed once per iteration here and the step's epilogue
// multiplies each right-hand-side row by it.  M = 2 G + rho I is formed in
// FP64 from the FP64 Gram of W = H_t, rounded to FP32 and inverted by
// Gauss-Jordan elimination in place without pivoting (M is symmetric
// positive definite, rho > 0): pivot p maps a_pp -> 1/a_pp,
// a_pj -> a_pj/a_pp, a_ip -> -a_ip/a_pp and a_ij -> a_ij - a_ip a_pj/a_pp.
// Two shared buffers alternate so one barrier per pivot suffices.  Entries
// past k hold the identity, so the padded block of the inverse is the
// identity and the padded columns of H stay zero.
template <int KP>
__global__ void __launch_bounds__(256) admm_minv_kernel(const double *gram64, int k, double rho,
                                                        float *minv) {
  // the next step kernel may start streaming S now; its epilogue warps wait
  // for this grid (griddepcontrol.wait) before they read minv
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // gram64 is written by the preceding reduction kernel
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ float X[2][KP][KP + 1];
  for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) {
    const int i = e / KP, j = e % KP;
    float v = (i == j) ? 1.f : 0.f;
    if (i < k && j < k) v = (float)(2.0 * gram64[e] + (i == j ? rho : 0.0));
    X[0][i][j] = v;
  }
  __syncthreads();
  for (int p = 0; p < KP; ++p) {
    const float(*src)[KP + 1] = X[p & 1];
    float(*dst)[KP + 1] = X[(p + 1) & 1];
    const float d = 1.f / src[p][p];
    for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) {
      const int i = e / KP, j = e % KP;
      float v;
      if (i == p) {
        v = (j == p) ? d : src[p][j] * d;
      } else {
        const float f = src[i][p] * d;
        v = (j == p) ? -f : fmaf(-f, src[p][j], src[i][j]);
      }
      dst[i][j] = v;
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < KP * KP; e += blockDim.x) minv[e] = X[KP & 1][e / KP][e % KP];
}

}  // namespace

#define KP_SWITCH(kp, ...)                              \
  switch (kp) {                                         \
    case 8: { constexpr int KPV = 8; __VA_ARGS__; } break;   \
    case 16: { constexpr int KPV = 16; __VA_ARGS__; } break; \
    case 32: { constexpr int KPV = 32; __VA_ARGS__; } break; \
    case 64: { constexpr int KPV = 64; __VA_ARGS__; } break; \
    default: return cudaErrorInvalidValue;              \
  }

cudaError_t launch_epilogue(const EpiArgs &a, cudaStream_t s) {
  KP_SWITCH(a.kp, {
    constexpr size_t bytes = EpiK<KPV>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(epilogue_kernel<KPV>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    epilogue_kernel<KPV><<<a.ntiles, EpiK<KPV>::T, bytes, s>>>(a);
  });
  return cudaGetLastError();
}

cudaError_t launch_admm_minv(const double *gram64, int k, int kp, double rho, float *minv,
                             cudaStream_t s) {
  KP_SWITCH(kp, return launch_dependent(admm_minv_kernel<KPV>, dim3(1), 256, s, gram64, k, rho, minv));
  return cudaErrorInvalidValue;
}

cudaError_t launch_prepare_tiles(const float *H, int64_t n, int k, int kp, void *Bt, int bt_fmt,
                                 int64_t ldb, float *gram_part, cudaStream_t s) {
  (void)k;
  const int ntiles = (int)((n + kTileRows - 1) / kTileRows);
  KP_SWITCH(kp, prepare_kernel<KPV><<<ntiles, 256, 0, s>>>(H, n, Bt, bt_fmt, ldb, gram_part));
  return cudaGetLastError();
}

cudaError_t launch_reduce_iter(const ReduceArgs &a, int kp, cudaStream_t s) {
  const dim3 grid(1 + (a.gram_part ? kp * kp / 16 : 0));
  KP_SWITCH(kp, return launch_dependent(reduce_iter_kernel<KPV>, grid, 256, s, a));
  return cudaErrorInvalidValue;
}

cudaError_t launch_gram_subset(const float *gram_part, int kp, const int *l1, int n1,
                               const int *l2, int n2, float *o1, float *o2, int kb, cudaStream_t s) {
  KP_SWITCH(kp, return launch_dependent(gram_subset_kernel<KPV>, dim3(kp * kp / 16, 2), 256, s,
                                        gram_part, l1, n1, l2, n2, o1, o2, kb));
  return cudaErrorInvalidValue;
}

cudaError_t launch_norm_s2(const void *S, int64_t n, int64_t lds, int dtype, const float *scales,
                           int64_t ld_scales, double *partials, int nparts, double *out,
                           cudaStream_t s) {
  const bool vec = rows_on_16(S, lds, dtype);
  switch (dtype) {
    case 0: norm_s2_kernel<0><<<nparts, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, partials); break;
    case 1: norm_s2_kernel<1><<<nparts, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, partials); break;
    case 2: norm_s2_kernel<2><<<nparts, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, partials); break;
    default: return cudaErrorInvalidValue;
  }
  sum_array_kernel<<<1, 256, 0, s>>>(partials, nparts, 1, 0, out);
  return cudaGetLastError();
}

cudaError_t launch_pack(const float *src, float *dst, int64_t n, int k, int kp, cudaStream_t s) {
  const int64_t tot = (n + kTileRows - 1) / kTileRows * kTileRows * kp;
  pack_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(src, dst, n, k, kp);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const float *src, float *dst, int64_t n, int k, int kp, cudaStream_t s) {
  const int64_t tot = n * k;
  unpack_kernel<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(src, dst, n, k, kp);
  return cudaGetLastError();
}

cudaError_t launch_median_g2(const float *g, int64_t n, int c0, int kw, int kp, unsigned *hist,
                             unsigned *sel, float *out, cudaStream_t s) {
  const int64_t total = n * kw;
  const unsigned rank = (unsigned)((total - 1) / 2);
  init_sel_kernel<<<1, 256, 0, s>>>(sel, rank, hist);
  const int grid = (int)std::min<int64_t>(1024, (total + 255) / 256);
  const int shifts[3] = {21, 10, 0};
  const int bits[3] = {11, 11, 10};
  for (int p = 0; p < 3; ++p) {
    hist_kernel<<<grid, 256, 0, s>>>(g, n, c0, kw, kp, shifts[p], bits[p], sel, hist);
    select_kernel<<<1, 1, 0, s>>>(hist, shifts[p], bits[p], sel, out, p == 2);
  }
  return cudaGetLastError();
}

cudaError_t launch_reset(float *A, const float *g, const float *med, float c, int64_t n, int c0,
                         int kw, int kp, double *slots, cudaStream_t s) {
  const int ntiles = (int)((n + kTileRows - 1) / kTileRows);
  KP_SWITCH(kp, reset_kernel<KPV><<<ntiles, 256, 0, s>>>(A, g, med, c, n, c0, kw, slots));
  return cudaGetLastError();
}

cudaError_t launch_sum_slot(const double *slots, int ntiles, int which, double *out,
                            cudaStream_t s) {
  sum_array_kernel<<<1, 256, 0, s>>>(slots, ntiles, kSlotStride, which, out);
  return cudaGetLastError();
}

}  // namespace symnmf
