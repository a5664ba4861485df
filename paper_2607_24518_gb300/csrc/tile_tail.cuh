// What a kernel that holds a 128-row tile of a factor in shared memory leaves
// of it for the next product and reduction: the tile's transposed MMA copy and
// its Gram partial.
#pragma once
#include "epi_common.cuh"

namespace symnmf {
namespace {

// The Gram partial of the tile in Hn by the T threads of the block, in the
// row order of every Gram partial: the lanes of a quad hold the four FMA
// chains of a B x B block of the 8 x 8 block grid (T = 512: of half its
// rows), so an entry costs two shared-memory reads per B FMAs, not per FMA.
template <int KP, int T>
__device__ __forceinline__ void tile_gram(const float (*Hn)[KP + 1], float *gp) {
  constexpr int B = KP / 8, PARTS = T / 256, BR = B / PARTS;
  const int part = threadIdx.x >> 8, et = threadIdx.x & 255;
  const int g = et & 3, bl = (et >> 2) & 7, wq = et >> 5;
  const int c0 = (2 * (wq >> 1) + (bl >> 2)) * B + part * BR;
  const int d0 = (4 * (wq & 1) + (bl & 3)) * B;
  float acc[BR][B];
#pragma unroll
  for (int i = 0; i < BR; ++i)
#pragma unroll
    for (int j = 0; j < B; ++j) acc[i][j] = 0.f;
#pragma unroll 4
  for (int i = 0; i < 32; ++i) {
    const float *hr = Hn[4 * i + g];
    float x[BR], y[B];
#pragma unroll
    for (int ii = 0; ii < BR; ++ii) x[ii] = hr[c0 + ii];
#pragma unroll
    for (int jj = 0; jj < B; ++jj) y[jj] = hr[d0 + jj];
#pragma unroll
    for (int ii = 0; ii < BR; ++ii)
#pragma unroll
      for (int jj = 0; jj < B; ++jj) acc[ii][jj] = fmaf(x[ii], y[jj], acc[ii][jj]);
  }
#pragma unroll
  for (int ii = 0; ii < BR; ++ii) {
#pragma unroll
    for (int jj = 0; jj < B; ++jj) acc[ii][jj] = gram_quad_sum(acc[ii][jj]);
    if ((ii * 4) / BR == g) {  // the quad's lanes share the stores
#pragma unroll
      for (int jj = 0; jj < B; ++jj) gp[(c0 + ii) * KP + d0 + jj] = acc[ii][jj];
    }
  }
}

// writes the transposed MMA copy (format bt_fmt) and the Gram partial of
// the tile held in smem Hn[128][KP+1]; every thread of the block calls it
template <int KP, int T>
__device__ void tile_tail(const float (*Hn)[KP + 1], int64_t r0, void *Bt, int bt_fmt, int64_t ldb,
                          float *gram_part, int tile) {
  const int tid = threadIdx.x;
  if (Bt && bt_fmt == 0) {
    uint16_t *B = reinterpret_cast<uint16_t *>(Bt);
    for (int e = tid; e < KP * kTileRows; e += blockDim.x) {
      const int c = e / kTileRows, r = e % kTileRows;
      const float v = Hn[r][c];
      const uint16_t hi = bf16_bits(v);
      const uint16_t lo = bf16_bits(v - bf16_val(hi));
      B[(int64_t)c * ldb + r0 + r] = hi;
      B[(int64_t)(KP + c) * ldb + r0 + r] = lo;
    }
  } else if (Bt && bt_fmt == 2) {
    // tile factor d from the tile's largest entry (H >= 0), then the pieces
    __shared__ float wmax[32];
    float m = 0.f;
    for (int e = tid; e < KP * kTileRows; e += blockDim.x) m = fmaxf(m, Hn[e % kTileRows][e / kTileRows]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) wmax[tid >> 5] = m;
    __syncthreads();
    float amax = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) amax = fmaxf(amax, wmax[w]);
    const float d = e4m3_tile_scale(amax), inv = 1.f / d;
    uint8_t *B = reinterpret_cast<uint8_t *>(Bt);
    for (int e = tid; e < KP * kTileRows; e += blockDim.x) {
      const int c = e / kTileRows, r = e % kTileRows;
      uint8_t hi, lo;
      e4m3_pieces(Hn[r][c], inv, hi, lo);
      B[(int64_t)c * ldb + r0 + r] = hi;
      B[(int64_t)(KP + c) * ldb + r0 + r] = lo;
    }
    if (tid == 0) bt_deq(Bt, KP, ldb)[tile] = d;
    __syncthreads();
  } else if (Bt) {
    float *B = reinterpret_cast<float *>(Bt);
    uint16_t *B16 = bt_b16(Bt, KP, ldb);
    for (int e = tid; e < KP * kTileRows; e += blockDim.x) {
      const int c = e / kTileRows, r = e % kTileRows;
      const float v = Hn[r][c];
      const float hi = tf32_lead<KP>(v);
      B[(int64_t)c * ldb + r0 + r] = hi;
      B[(int64_t)(KP + c) * ldb + r0 + r] = tf32_round(v - hi);
      B16[(int64_t)c * ldb + r0 + r] = bf16_bits(v);
    }
  }
  if (gram_part) tile_gram<KP, T>(Hn, gram_part + (int64_t)tile * KP * KP);
}

}  // namespace
}  // namespace symnmf
