// Objective f = ||S||^2 - 2 tr(H^T S H) + ||H^T H||^2 (Eq. 2) for a caller's
// S and H without a handle and without allocating device memory.
//
// Some callers cannot allocate at the moment they need an objective: a
// monitor thread that must not stall a running solve (cudaMalloc / cudaFree
// can synchronise the device), a process whose memory is fully reserved by
// another allocator, or code that has promised its host application a fixed
// device footprint.  This entry point serves them.  Its scratch is one
// fixed array in device memory, created with the library's module, so a
// call only launches kernels.
//
// Three kernels: (1) one CTA per (row tile, column share) multiplies its
// share of S by H (FP32 FMA) and immediately dots the partial product rows
// with H_I, leaving one FP64 partial of tr per CTA, and one more CTA per row
// tile writes the FP32 Gram partial H_I^T H_I; (2) 16 Gram entries per CTA
// are added across tiles in FP64, leaving the sum of their squares; (3) one
// CTA adds the partials in a fixed order in FP64 and writes f.  Every scratch
// slot that is read is written earlier in the same call, so nothing in the
// scratch has to start at zero, and two calls with the same inputs give the
// same bits.
#include <mutex>

#include "../../include/symnmf.h"
#include "simt_tile.cuh"
#include "symnmf_internal.h"

namespace symnmf {
namespace {

constexpr int kSplit = 8;   // at most so many column shares per row tile in kernel (1)
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[SYMNMF_NOALLOC_SCRATCH_BYTES];

struct ObjArgs {
  const void *S;
  int64_t n, lds;
  const float *scales;
  int64_t ld_scales;
  const float *H;   // n x k, row pitch k
  int k;
  int ntiles;
  double normS2;
  int split;        // column shares per row tile, at most kSplit
  double *tr_part;  // ntiles * kSplit; slot [tile * kSplit + split] of a share
  float *gram_part; // ntiles * kp * kp
  // the CTA sums of squares of kernel (2): CTA b's over its own entries 16 b
  // and 16 b + 1 of tile 0's Gram partial, which it alone has read by then
  __device__ double *g2_slot(int b) const { return reinterpret_cast<double *>(gram_part + 16 * b); }
  double *f;
};

// fixed-order sum over the block: xor tree per warp, warps in order
__device__ __forceinline__ double block_sum_fixed(double v, double *sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  __syncthreads();
  return r;  // valid in thread 0
}

// the Gram partial of a row tile: rows r = 4 i + g in four FMA chains, added
// (s0 + s1) + (s2 + s3), the row order of the solver's Gram partials
template <int KP>
__device__ void gram_tile(const ObjArgs &a, int tile, float *sm) {
  float(*Hn)[KP + 1] = reinterpret_cast<float(*)[KP + 1]>(sm);
  const int64_t r0 = (int64_t)tile * kTileRows;
  for (int e = threadIdx.x; e < kTileRows * KP; e += 256) {
    const int r = e / KP, c = e % KP;
    Hn[r][c] = (r0 + r < a.n && c < a.k) ? a.H[(r0 + r) * a.k + c] : 0.f;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < KP * KP; q += 256)
    a.gram_part[(int64_t)tile * KP * KP + q] = gram_entry<KP>(Hn, q / KP, q % KP);
}

// blockIdx.y < split: a column share; == split: the tile's Gram partial.
// n = 10000, KP = 32 FP32: 500 -> 188 us (17 TFMA/s of 37), BF16 695 -> 264, FP8
// 563 -> 243; KP = 64 527 / 854 / 780 -> 337 / 415 / 397 (128 registers: BF16 and FP8
// spill 88 to 240 bytes a thread above KP = 8, FP32 68 above KP = 16).  The tile
// Grams beside the shares and their sum over the chip replace a pass of their
// own and one CTA's 49 us.
template <int DT, int KP>
__global__ void __launch_bounds__(256, 2) tr_share_kernel(ObjArgs a) {
  extern __shared__ __align__(16) float sm_obj[];
  __shared__ double red[8];
  const int tid = threadIdx.x, tile = blockIdx.x, split = blockIdx.y;
  if (split == a.split) {
    gram_tile<KP>(a, tile, sm_obj);
    return;
  }
  const int64_t r0 = (int64_t)tile * kTileRows;
  const int per = (a.ntiles + a.split - 1) / a.split;
  const int cb = min(a.ntiles, split * per), ce = min(a.ntiles, cb + per);
  simt_tile<DT, KP>(sm_obj, a.S, a.lds, a.n, r0, a.H, a.k, a.k, nullptr, cb, ce,
                    DT == 2 ? a.scales + (int64_t)tile * a.ld_scales : nullptr);
  // this share's part of sum_{r, c} H_rc (S H)_rc over the tile's rows
  float t = 0.f;
#pragma unroll 4
  for (int e = tid; e < kTileRows * KP; e += 256) {
    const int r = e / KP, c = e % KP;
    if (r0 + r < a.n && c < a.k) t = fmaf(__ldg(a.H + (r0 + r) * a.k + c), sm_obj[e], t);
  }
  const double s = block_sum_fixed((double)t, red);
  if (tid == 0) a.tr_part[(int64_t)tile * kSplit + split] = s;
}

// 16 Gram entries per CTA, 16 threads to an entry: tiles j, j + 16, ... in
// order, then the 16 sums in order; the sum of the entries' squares goes to
// the CTA's g2_slot
template <int KP>
__global__ void __launch_bounds__(256) gram_sum_kernel(ObjArgs a) {
  __shared__ double red[256];
  const int tid = threadIdx.x, le = tid & 15, j = tid >> 4;
  const float *src = a.gram_part + blockIdx.x * 16 + le;
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
    double g = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) g += red[i * 16 + tid];
    g *= g;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffu, g, o);
    if (tid == 0) *a.g2_slot(blockIdx.x) = g;
  }
}

template <int KP>
__global__ void __launch_bounds__(256) finish_kernel(ObjArgs a) {
  __shared__ double red[8];
  const int tid = threadIdx.x;
  // tr: thread tid adds a contiguous run of tiles, runs added in order
  const int per = (a.ntiles + 255) / 256;
  double tr = 0.0;
  for (int t = tid * per; t < a.ntiles && t < (tid + 1) * per; ++t)
    for (int s = 0; s < a.split; ++s) tr += a.tr_part[(int64_t)t * kSplit + s];
  double g2 = 0.0;
  if (tid < KP * KP / 16) g2 = *a.g2_slot(tid);
  const double trs = block_sum_fixed(tr, red);
  const double g2s = block_sum_fixed(g2, red);
  if (tid == 0) *a.f = a.normS2 - 2.0 * trs + g2s;
}

template <int DT, int KP>
cudaError_t launch_all(const ObjArgs &a, cudaStream_t s) {
  tr_share_kernel<DT, KP><<<dim3(a.ntiles, a.split + 1), 256, Simt<DT, KP>::SMEM, s>>>(a);
  gram_sum_kernel<KP><<<KP * KP / 16, 256, 0, s>>>(a);
  finish_kernel<KP><<<1, 256, 0, s>>>(a);
  return cudaGetLastError();
}

template <int DT>
cudaError_t launch_dt(const ObjArgs &a, int kp, cudaStream_t s) {
  switch (kp) {
    case 8: return launch_all<DT, 8>(a, s);
    case 16: return launch_all<DT, 16>(a, s);
    case 32: return launch_all<DT, 32>(a, s);
    case 64: return launch_all<DT, 64>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

std::mutex g_addr_mu;
void *g_addr[kMaxDevices] = {};
int g_sms[kMaxDevices] = {};

// Load every kernel this entry point launches on the current device.  With
// lazy module loading each kernel would otherwise be loaded at its first
// launch, i.e. inside some later call, which may allocate and synchronise.
// (tr_share also takes more shared memory than a kernel may use by default)
template <int DT, int KP>
cudaError_t preload_tr() {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, tr_share_kernel<DT, KP>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tr_share_kernel<DT, KP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Simt<DT, KP>::SMEM);
  return e;
}
template <int DT>
cudaError_t preload_dt() {
  cudaError_t e = preload_tr<DT, 8>();
  if (e == cudaSuccess) e = preload_tr<DT, 16>();
  if (e == cudaSuccess) e = preload_tr<DT, 32>();
  if (e == cudaSuccess) e = preload_tr<DT, 64>();
  return e;
}
template <int KP>
cudaError_t preload_kp() {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, gram_sum_kernel<KP>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, finish_kernel<KP>);
  return e;
}
cudaError_t preload_kernels() {
  cudaError_t e = preload_dt<0>();
  if (e == cudaSuccess) e = preload_dt<1>();
  if (e == cudaSuccess) e = preload_dt<2>();
  if (e == cudaSuccess) e = preload_kp<8>();
  if (e == cudaSuccess) e = preload_kp<16>();
  if (e == cudaSuccess) e = preload_kp<32>();
  if (e == cudaSuccess) e = preload_kp<64>();
  return e;
}

// Argument and size check of the entry point, host arithmetic only.  On OK
// *need is the scratch the call uses and *kp the padded rank.
int noalloc_validate(bool have_S, int64_t n, int64_t lds, int32_t dtype, bool have_scales,
                     int64_t ld_scales, bool have_H, int32_t k, bool have_f, size_t *need,
                     int *kp_out) {
  if (!have_S || !have_H || !have_f || n < 1 || lds < n || k < 1 || k > 64)
    return SYMNMF_ERR_INVALID;
  if (dtype != SYMNMF_F32 && dtype != SYMNMF_BF16 && dtype != SYMNMF_FP8E4M3)
    return SYMNMF_ERR_INVALID;
  const int64_t ntiles = (n + kTileRows - 1) / kTileRows;
  if (dtype == SYMNMF_FP8E4M3 && (!have_scales || ld_scales < ntiles)) return SYMNMF_ERR_INVALID;
  const int kp = k <= 8 ? 8 : k <= 16 ? 16 : k <= 32 ? 32 : 64;
  // scratch: ntiles * kSplit FP64 tr partials, then (256-byte aligned)
  // ntiles * kp * kp FP32 Gram partials
  const size_t tr_bytes = ((size_t)ntiles * kSplit * sizeof(double) + 255) & ~(size_t)255;
  *need = tr_bytes + (size_t)ntiles * kp * kp * sizeof(float);
  *kp_out = kp;
  if (ntiles > 65535 || *need > (size_t)SYMNMF_NOALLOC_SCRATCH_BYTES) return SYMNMF_ERR_UNSUPPORTED;
  return SYMNMF_OK;
}

}  // namespace
}  // namespace symnmf

using namespace symnmf;

extern "C" int symnmf_objective_noalloc_check(int64_t n, int64_t lds, int32_t dtype,
                                              int32_t have_scales, int64_t ld_scales, int32_t k,
                                              size_t *need) {
  size_t bytes = 0;
  int kp = 0;
  const int st = noalloc_validate(true, n, lds, dtype, have_scales != 0, ld_scales, true, k, true,
                                  &bytes, &kp);
  if (need) *need = bytes;
  return st;
}

extern "C" int symnmf_objective_noalloc(const void *S, int64_t n, int64_t lds, int32_t dtype,
                                        const float *scales, int64_t ld_scales, const float *H,
                                        int32_t k, double normS2, double *f, void *stream) {
  size_t need = 0;
  int kp = 0;
  const int st = noalloc_validate(S != nullptr, n, lds, dtype, scales != nullptr, ld_scales,
                                  H != nullptr, k, f != nullptr, &need, &kp);
  if (st != SYMNMF_OK) return st;
  const int64_t ntiles = (n + kTileRows - 1) / kTileRows;
  const size_t tr_bytes = ((size_t)ntiles * kSplit * sizeof(double) + 255) & ~(size_t)255;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SYMNMF_ERR_CUDA;
  void *base = nullptr;
  int sms = 0;
  {
    // first call on a device: look up that device's copy of the scratch
    // (this loads the library's module there, creating the array) and load
    // every kernel of this entry point, so later calls only launch
    std::lock_guard<std::mutex> lock(g_addr_mu);
    if (!g_addr[dev]) {
      void *p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess ||
          cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          preload_kernels() != cudaSuccess) {
        cudaGetLastError();
        return SYMNMF_ERR_CUDA;
      }
      g_addr[dev] = p;
    }
    base = g_addr[dev];
    sms = g_sms[dev];
  }
  ObjArgs a{};
  a.S = S;
  a.n = n;
  a.lds = lds;
  a.scales = scales;
  a.ld_scales = ld_scales;
  a.H = H;
  a.k = k;
  a.ntiles = (int)ntiles;
  a.split = simt_split(a.ntiles, a.ntiles, kp, 2 * sms, kSplit, kSplit);
  a.normS2 = normS2;
  a.tr_part = reinterpret_cast<double *>(base);
  a.gram_part = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(base) + tr_bytes);
  a.f = f;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e;
  switch (dtype) {
    case SYMNMF_F32: e = launch_dt<0>(a, kp, s); break;
    case SYMNMF_BF16: e = launch_dt<1>(a, kp, s); break;
    default: e = launch_dt<2>(a, kp, s); break;
  }
  return e == cudaSuccess ? SYMNMF_OK : SYMNMF_ERR_CUDA;
}
