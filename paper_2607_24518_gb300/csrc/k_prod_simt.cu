// SIMT product P = S[rows, cols] * H[cols] (Sec. 2.1: the S H term of the
// gradient), FP32 FFMA with FP32 accumulation.  This is the exact-FP32
// path and the fallback for layouts the tensor-core kernel cannot take
// (S row pitch not a multiple of 16 bytes).  One CTA owns one 128-row tile
// and a contiguous share (split) of the column-tile list; partial sums go
// to out[split][row_pos] and are added in split order by the epilogue.
#include <algorithm>

#include "simt_tile.cuh"
#include "symnmf_internal.h"

namespace symnmf {
namespace {

// 128 registers for two CTAs per SM.  BF16 and FP8 above KP = 8 spill 48 to 320
// bytes a thread under that cap, FP32 above KP = 16 24, and are quicker at every
// rank all the same than one 16-value block per thread fed by scalar reads with
// no chunk in flight during the FMAs.  Before -> now in us, KP = 8 / 16 / 32 / 64:
// n = 3001 FP32 23 / 33 / 45 / 61 -> 11 / 15 / 21 / 35, BF16 22 / 33 / 46 / 68 -> 15 /
// 19 / 23 / 41, FP8 34 / 33 / 52 / 69 -> 16 / 19 / 24 / 40; n = 10000 FP32 284 / 339 /
// 442 / 584 -> 80 / 130 / 207 / 367, BF16 216 / 292 / 446 / 761 -> 199 / 209 / 272 /
// 516, FP8 422 / 287 / 584 / 733 -> 190 / 195 / 268 / 466.
template <int DT, int KP>
__global__ void __launch_bounds__(256, 2) prod_simt_kernel(ProdArgs a) {
  extern __shared__ __align__(16) float sm_simt[];
  const int pos = blockIdx.x, split = blockIdx.y;
  const int rt = a.row_list ? a.row_list[pos] : pos;
  const int per = (a.n_cols_list + a.nsplit - 1) / a.nsplit;
  const int cb = min(a.n_cols_list, split * per), ce = min(a.n_cols_list, cb + per);
  simt_tile<DT, KP>(sm_simt, a.S, a.lds, a.n, (int64_t)rt * kTileRows, a.H, KP, KP, a.col_list, cb,
                    ce, DT == 2 ? a.scales + (int64_t)rt * a.ld_scales : nullptr);
  float4 *out = reinterpret_cast<float4 *>(a.out + ((int64_t)split * a.n_rows_list + pos) * kTileRows * KP);
  for (int i = threadIdx.x; i < kTileRows * KP / 4; i += 256)
    out[i] = reinterpret_cast<const float4 *>(sm_simt)[i];
}

template <int DT, int KP>
cudaError_t launch_kp(const ProdArgs &a, cudaStream_t s) {
  constexpr size_t bytes = Simt<DT, KP>::SMEM;
  const cudaError_t e = cudaFuncSetAttribute(
      prod_simt_kernel<DT, KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  prod_simt_kernel<DT, KP><<<dim3(a.n_rows_list, a.nsplit), 256, bytes, s>>>(a);
  return cudaGetLastError();
}

template <int DT>
cudaError_t launch_dt(const ProdArgs &a, cudaStream_t s) {
  switch (a.kp) {
    case 8: return launch_kp<DT, 8>(a, s);
    case 16: return launch_kp<DT, 16>(a, s);
    case 32: return launch_kp<DT, 32>(a, s);
    case 64: return launch_kp<DT, 64>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_prod_simt(const ProdArgs &a, cudaStream_t s) {
  if (a.n_rows_list <= 0 || a.n_cols_list <= 0) return cudaSuccess;
  switch (a.dtype) {
    case 0: return launch_dt<0>(a, s);
    case 1: return launch_dt<1>(a, s);
    case 2: return launch_dt<2>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

int simt_shares(int rows, int cols, int kp, int num_sms, int most) {
  // parts: three CTAs per SM
  const int parts = std::max(1, std::min((3 * num_sms + rows - 1) / std::max(1, rows), most));
  return simt_split(rows, cols, kp, 2 * num_sms, most, parts);
}

}  // namespace symnmf
