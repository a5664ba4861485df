// Spherical K-means (Lloyd) on the rows of S (Sec. 6, "Clustering
// alternatives"): the rows s_i are normalised, x_i = s_i / ||s_i||, each
// cluster's centroid is the normalised sum of its members, and each row
// joins the cluster of largest cosine.  One Lloyd iteration is two passes
// of the streamed product with n x K operands (S symmetric):
//   C = S (D^-1 B)             columns c_k = sum_{i in C_k} x_i
//   P = S C                    P_ik = <s_i, c_k>
//   cos_ik = P_ik / (||s_i|| ||c_k||),  L'(i) = first argmax_k cos_ik,
//   J = sum_i (1 - max_k cos_ik).
// The kernels here are the small ones around the two product passes: row
// norms (once per matrix), the operand D^-1 B from the labels, the centroid
// gather with per-tile FP64 column sums of squares, the centroid norms, the
// assignment with per-tile FP64 objective partials, and the final
// fixed-order sum.  The two operands are written straight in the product's
// format.  Every cross-tile sum is FP64 in a fixed order, so a run is
// bit-reproducible.  All of them are bound by latency; n = 20000, K = 32
// BF16, per iteration: operand 8.6 + 2 x 3.8 (conversion) -> 3.3, centroids 25
// -> 6.6, norms 10.7 -> 4.5, assignment 16 -> 7 us (scattered reads of the
// partials, FP64 per entry and one thread per column over all tiles before).
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "../../include/symnmf.h"
#include "epi_common.cuh"
#include "tile_tail.cuh"
#include "symnmf_internal.h"

namespace symnmf {
namespace {

// ||s_i|| in FP64: one warp per row, runs of 64 entries in FP32 words (SqSum)
template <int DT>
__global__ void __launch_bounds__(256, 4) row_norms_kernel(const void *S, int64_t n, int64_t lds,
                                                        const float *scales, int64_t ld_scales,
                                                        bool vec, double *rn, float *rinv) {
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  double acc =
      row_sumsq_lane<DT>(S, row * lds, n, scales + (row / kTileRows) * ld_scales, vec, lane);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    const double r = sqrt(acc);
    rn[row] = r;
    rinv[row] = (float)(1.0 / r);
  }
}

// the tile in Cs as the next product's operand
template <int KP>
__device__ __forceinline__ void km_write_operand(const KmArgs &a, const float (*Cs)[KP + 1],
                                                 int tile) {
  const int64_t r0 = (int64_t)tile * kTileRows;
  if (a.C) {
    for (int e = threadIdx.x; e < kTileRows * KP; e += 256) a.C[r0 * KP + e] = Cs[e / KP][e % KP];
  }
  tile_tail<KP, 256>(Cs, r0, a.Bt, a.bt_fmt, a.ldb, nullptr, tile);
}

// operand D^-1 B: row i holds 1 / ||s_i|| in column labels_in[i]
template <int KP>
__global__ void __launch_bounds__(256) km_operand_kernel(KmArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ float Cs[kTileRows][KP + 1];
  const int64_t r0 = (int64_t)blockIdx.x * kTileRows;
  for (int e = threadIdx.x; e < kTileRows * (KP + 1); e += 256) (&Cs[0][0])[e] = 0.f;
  __syncthreads();
  const int r = threadIdx.x;
  if (r < kTileRows && r0 + r < a.n) {
    const int c = a.labels_in[r0 + r];
    if (c >= 0 && c < a.K) Cs[r][c] = a.rinv[r0 + r];
  }
  __syncthreads();
  km_write_operand<KP>(a, Cs, blockIdx.x);
}

// the summed partials of the tile into Cs (rows past n and columns past K 0),
// slots in order, whole rows in 16-byte pieces, four of them in flight
template <int KP>
__device__ __forceinline__ void km_gather(const KmArgs &a, float (*Cs)[KP + 1], int tile) {
  const int64_t r0 = (int64_t)tile * kTileRows;
  int64_t b0, b1;
  part_range(tile, a.skG, a.ncols, a.ntiles, b0, b1);
  const int64_t first = a.skG > 0 ? b0 + tile : tile;
  const int64_t step = (a.skG > 0 ? 1 : (int64_t)a.ntiles) * kTileRows * KP;
  const int count = a.skG > 0 ? (int)(b1 - b0) + 1 : a.nsplit;
  const float *base = a.P + first * kTileRows * KP;
  for (int e = threadIdx.x; e < kTileRows * KP / 4; e += 256) {
    const int r = e / (KP / 4), c = 4 * (e % (KP / 4));
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q0 = 0; q0 < count; q0 += 4) {
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = q0 + u < count ? __ldcg(reinterpret_cast<const float4 *>(base + (q0 + u) * step) + e)
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
    for (int j = 0; j < 4; ++j) Cs[r][c + j] = (r0 + r < a.n && c + j < a.K) ? s[j] : 0.f;
  }
}

// centroid rows C_I = sum of the partials, and per-tile column sums of
// squares: 256 / KP threads per column, each a run (SqSum) of its rows,
// added in order in FP64
template <int KP>
__global__ void __launch_bounds__(256) km_centroid_kernel(KmArgs a) {
  constexpr int G = 256 / KP, RG = kTileRows / G;  // row groups, rows per group
  __shared__ float Cs[kTileRows][KP + 1];
  __shared__ double part[G][KP];
  const int tile = blockIdx.x, tid = threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  km_gather<KP>(a, Cs, tile);
  __syncthreads();
  const int c = tid % KP, g = tid / KP;
  float m = 0.f;
#pragma unroll 8
  for (int r = g * RG; r < (g + 1) * RG; ++r) m = fmaxf(m, fabsf(Cs[r][c]));
  SqSum<> s;
  double d = 0.0;
  if (m == 0.f || s.raise(m)) {
#pragma unroll 8
    for (int r = g * RG; r < (g + 1) * RG; ++r) s.put(Cs[r][c]);
    s.flush();
    d = s.acc;
  } else {
    for (int r = g * RG; r < (g + 1) * RG; ++r) d = fma((double)Cs[r][c], (double)Cs[r][c], d);
  }
  part[g][c] = d;
  __syncthreads();
  if (tid < KP) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < G; ++i) t += part[i][tid];
    a.colsq[(int64_t)tile * KP + tid] = t;
  }
  km_write_operand<KP>(a, Cs, tile);
}

// ||c_k||: 256 / KP threads per column, tiles g, g + G, ... each, the threads
// in order; inv_norm = 0 for an empty cluster.  Runs beside the second product
// (whose launch has seen the centroids complete) and waits for it before it
// ends, as the assignment that follows needs both
template <int KP>
__global__ void __launch_bounds__(256) km_norms_kernel(KmArgs a) {
  constexpr int G = 256 / KP;
  __shared__ double part[G][KP];
  const int c = threadIdx.x % KP, g = threadIdx.x / KP;
  double s = 0.0;
#pragma unroll 4
  for (int t = g; t < a.ntiles; t += G) s += __ldcg(a.colsq + (int64_t)t * KP + c);
  part[g][c] = s;
  __syncthreads();
  if (threadIdx.x >= KP) return;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  s = 0.0;
#pragma unroll
  for (int i = 0; i < G; ++i) s += part[i][c];
  const double nk = sqrt(s);
  a.inv_norm[c] = (c < a.K && nk > 0.0) ? (float)(1.0 / nk) : 0.f;
}

// assignment: first argmax over k < K of P_ik / ||c_k|| (the row's 1 / ||s_i||
// is common to all k); per-tile FP64 sums of 1 - cos and of the changed labels
template <int KP>
__global__ void __launch_bounds__(256) km_assign_kernel(KmArgs a) {
  __shared__ float Cs[kTileRows][KP + 1];
  __shared__ float inv[KP];
  __shared__ double red[8];
  const int tile = blockIdx.x, r = threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (r < KP) inv[r] = a.inv_norm[r];
  km_gather<KP>(a, Cs, tile);
  __syncthreads();
  const int64_t row = (int64_t)tile * kTileRows + r;
  double j = 0.0, ch = 0.0;
  if (r < kTileRows && row < a.n) {
    int best = 0;
    float bs = 0.f;
    for (int c = 0; c < a.K; ++c) {
      const float sc = Cs[r][c] * inv[c];
      if (c == 0 || sc > bs) {
        bs = sc;
        best = c;
      }
    }
    const double cosv = (double)bs / a.rn[row];
    j = 1.0 - cosv;
    a.labels_out[row] = best;
    ch = (best != a.labels_in[row]) ? 1.0 : 0.0;
  }
  // fixed-order block sums: xor tree per warp, warps in order
  double v[2] = {j, ch};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  }
  if (r < kTileRows && (r & 31) == 0) {
    red[(r >> 5) * 2 + 0] = v[0];
    red[(r >> 5) * 2 + 1] = v[1];
  }
  __syncthreads();
  if (r == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int w = 0; w < kTileRows / 32; ++w) {
      s0 += red[2 * w];
      s1 += red[2 * w + 1];
    }
    a.slots[(int64_t)tile * 2 + 0] = s0;
    a.slots[(int64_t)tile * 2 + 1] = s1;
  }
}

// J and the changed count: runs of tiles per thread, runs in order
__global__ void __launch_bounds__(256) km_final_kernel(KmArgs a) {
  __shared__ double red[2][8];
  const int tid = threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int per = (a.ntiles + 255) / 256;
  double s0 = 0.0, s1 = 0.0;
  for (int t = tid * per; t < a.ntiles && t < (tid + 1) * per; ++t) {
    s0 += a.slots[(int64_t)t * 2];
    s1 += a.slots[(int64_t)t * 2 + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = s0;
    red[1][tid >> 5] = s1;
  }
  __syncthreads();
  if (tid == 0) {
    double t0 = 0.0, t1 = 0.0;
    for (int w = 0; w < 8; ++w) {
      t0 += red[0][w];
      t1 += red[1][w];
    }
    a.out[0] = t0;
    a.out[1] = t1;
  }
}

}  // namespace

#define KM_KP_SWITCH(kp, ...)                                \
  switch (kp) {                                              \
    case 8: { constexpr int KPV = 8; __VA_ARGS__; } break;   \
    case 16: { constexpr int KPV = 16; __VA_ARGS__; } break; \
    case 32: { constexpr int KPV = 32; __VA_ARGS__; } break; \
    case 64: { constexpr int KPV = 64; __VA_ARGS__; } break; \
    default: return cudaErrorInvalidValue;                   \
  }

cudaError_t launch_row_norms(const void *S, int64_t n, int64_t lds, int dtype, const float *scales,
                             int64_t ld_scales, double *rn, float *rinv, cudaStream_t s) {
  const unsigned blocks = (unsigned)((n + 7) / 8);
  const bool vec = rows_on_16(S, lds, dtype);
  switch (dtype) {
    case 0: row_norms_kernel<0><<<blocks, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, rn, rinv); break;
    case 1: row_norms_kernel<1><<<blocks, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, rn, rinv); break;
    case 2: row_norms_kernel<2><<<blocks, 256, 0, s>>>(S, n, lds, scales, ld_scales, vec, rn, rinv); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_km_operand(const KmArgs &a, int kp, cudaStream_t s) {
  KM_KP_SWITCH(kp, km_operand_kernel<KPV><<<a.ntiles, 256, 0, s>>>(a));
  return cudaGetLastError();
}

cudaError_t launch_km_centroids(const KmArgs &a, int kp, cudaStream_t s) {
  KM_KP_SWITCH(kp, return launch_dependent(km_centroid_kernel<KPV>, dim3(a.ntiles), 256, s, a));
  return cudaErrorInvalidValue;
}

cudaError_t launch_km_norms(const KmArgs &a, int kp, cudaStream_t s) {
  KM_KP_SWITCH(kp, return launch_dependent(km_norms_kernel<KPV>, dim3(1), 256, s, a));
  return cudaErrorInvalidValue;
}

cudaError_t launch_km_assign(const KmArgs &a, int kp, cudaStream_t s) {
  cudaError_t e = cudaErrorInvalidValue;
  KM_KP_SWITCH(kp, e = launch_dependent(km_assign_kernel<KPV>, dim3(a.ntiles), 256, s, a));
  if (e != cudaSuccess) return e;
  return launch_dependent(km_final_kernel, dim3(1), 256, s, a);
}

}  // namespace symnmf
