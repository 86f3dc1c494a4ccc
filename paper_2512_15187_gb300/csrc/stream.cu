// Host-side dispatch of the streaming pass (kernel in stream_kernel.cuh, instantiated per
// tile class in stream_c*.cu) and two small kernels of the library:
//   * member_coef_kernel — the coefficients of a weighted mean contour (Sec. 4.1).
//   * iso_kernel         — the isovalue map alone (pid_soft_masks, Sec. 3.5).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"

namespace pidk {

// ---------------------------------------------------------------------------------------
// Streaming pass: dispatch to the per-class instantiations (stream_c*.cu)
// ---------------------------------------------------------------------------------------

#define PIDK_CLASS(V, M, G)                                                                  \
  cudaError_t launch_stream_c##V##_##M##_##G(const StreamParams&, int, bool, int, size_t,  \
                                             cudaStream_t);                                \
  cudaError_t init_stream_c##V##_##M##_##G(int);
PIDK_CLASS(4, 8, 1)
PIDK_CLASS(4, 8, 2)
PIDK_CLASS(4, 6, 4)
PIDK_CLASS(4, 8, 4)
PIDK_CLASS(4, 6, 8)
PIDK_CLASS(4, 8, 8)
PIDK_CLASS(4, 6, 16)
PIDK_CLASS(4, 8, 16)
PIDK_CLASS(2, 12, 16)
PIDK_CLASS(2, 13, 16)
PIDK_CLASS(2, 16, 16)
PIDK_CLASS(1, 20, 16)
PIDK_CLASS(1, 24, 16)
PIDK_CLASS(1, 28, 16)
PIDK_CLASS(1, 32, 16)
#undef PIDK_CLASS

cudaError_t launch_stream(const StreamParams& p, int vec, int mpw, int G, int iso_kind, bool coef,
                          int grid, size_t smem, cudaStream_t s) {
#define PIDK_CASE(V, M, GG)                                                                   \
  if (vec == V && mpw == M && G == GG)                                                       \
    return launch_stream_c##V##_##M##_##GG(p, iso_kind, coef, grid, smem, s);
  PIDK_CASE(4, 8, 1)
  PIDK_CASE(4, 8, 2)
  PIDK_CASE(4, 6, 4)
  PIDK_CASE(4, 8, 4)
  PIDK_CASE(4, 6, 8)
  PIDK_CASE(4, 8, 8)
  PIDK_CASE(4, 6, 16)
  PIDK_CASE(4, 8, 16)
  PIDK_CASE(2, 12, 16)
  PIDK_CASE(2, 13, 16)
  PIDK_CASE(2, 16, 16)
  PIDK_CASE(1, 20, 16)
  PIDK_CASE(1, 24, 16)
  PIDK_CASE(1, 28, 16)
  PIDK_CASE(1, 32, 16)
#undef PIDK_CASE
  return cudaErrorInvalidValue;
}

// Opt every streaming instantiation in to the largest dynamic shared memory once per
// device (before any launch, so that launches can be captured into graphs).
cudaError_t stream_kernels_init(int max_smem) {
  cudaError_t e = finalize_kernels_init();
  if (e == cudaSuccess) e = init_stream_c4_8_1(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_8_2(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_6_4(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_8_4(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_6_8(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_8_8(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_6_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c4_8_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c2_12_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c2_13_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c2_16_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c1_20_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c1_24_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c1_28_16(max_smem);
  if (e == cudaSuccess) e = init_stream_c1_32_16(max_smem);
  return e;
}

size_t stream_smem_bytes(int vec, int G, int depth, int stage_floats) {
  const int T = 32 * vec;
  const int n_groups = kStreamWarps / G;
  return static_cast<size_t>(n_groups) * depth * stage_floats * 4 +
         static_cast<size_t>(n_groups) * 2 * (G * T + T) * 4 +
         static_cast<size_t>(n_groups) * depth * 8 + static_cast<size_t>(n_groups) * 8 + 64 +
         static_cast<size_t>(n_groups) * kStreamProducerBytes + 16;
}

constexpr int kCoefThreads = 1024;

// Coefficients of a weighted mean contour (Sec. 4.1): c_j = r_j / sum_k r_k from member
// weights r_j >= 0, summed in FP64 in a fixed order (strided per thread, then a tree).
// Weights that are negative, not finite, or all zero set the domain bit and give c = 0.
__global__ void __launch_bounds__(kCoefThreads, 1) member_coef_kernel(const double* r, int64_t N,
                                                                     float* coef, uint32_t* err) {
  __shared__ double sred[kCoefThreads];
  double acc = 0.0;
  int bad = 0;
  for (int64_t j = threadIdx.x; j < N; j += kCoefThreads) {
    const double v = r[j];
    if (v >= 0.0 && v <= 1.7976931348623157e308) acc += v; else bad = 1;
  }
  sred[threadIdx.x] = acc;
  __syncthreads();
  for (int o = kCoefThreads / 2; o > 0; o >>= 1) {
    if (static_cast<int>(threadIdx.x) < o) sred[threadIdx.x] += sred[threadIdx.x + o];
    __syncthreads();
  }
  const double R = sred[0];
  bad = __syncthreads_or(bad || !(R > 0.0 && R <= 1.7976931348623157e308));
  if (bad && threadIdx.x == 0) atomicOr(err, ERR_DOMAIN);
  for (int64_t j = threadIdx.x; j < N; j += kCoefThreads)
    coef[j] = bad ? 0.0f : static_cast<float>(r[j] / R);
}

cudaError_t launch_member_coef(const double* r, int64_t N, float* coef, uint32_t* err,
                               cudaStream_t s) {
  member_coef_kernel<<<1, kCoefThreads, 0, s>>>(r, N, coef, err);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Isovalue map alone (pid_soft_masks)
// ---------------------------------------------------------------------------------------

// Stores VEC soft masks, as float32 or rounded to nearest-even bfloat16.
template <bool BF16>
__device__ __forceinline__ void iso_store4(void* base, int64_t off, const float4& u) {
  if constexpr (BF16) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(u.x, u.y), b = __floats2bfloat162_rn(u.z, u.w);
    uint2 v;
    v.x = *reinterpret_cast<const uint32_t*>(&a);
    v.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(base) + off) = v;
  } else {
    *reinterpret_cast<float4*>(static_cast<float*>(base) + off) = u;
  }
}

template <bool BF16>
__device__ __forceinline__ void iso_store1(void* base, int64_t off, float u) {
  if constexpr (BF16) static_cast<__nv_bfloat16*>(base)[off] = __float2bfloat16_rn(u);
  else static_cast<float*>(base)[off] = u;
}

template <bool BF16>
__global__ void __launch_bounds__(256) iso_kernel(const __grid_constant__ IsoParams p) {
  // vector path: 16-byte aligned input rows, output rows aligned to 4 elements
  const bool vec = ((p.ld & 3) == 0) && ((p.ld_out & 3) == 0) &&
                   ((reinterpret_cast<uintptr_t>(p.F) & 15) == 0) &&
                   ((reinterpret_cast<uintptr_t>(p.U) & (BF16 ? 7 : 15)) == 0);
  const int64_t per_row = vec ? (p.M + 3) / 4 : p.M;
  const int64_t total = per_row * p.N;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total; t += stride) {
    const int64_t i = t / per_row;
    const int64_t j = t - i * per_row;
    const float* src = p.F + i * p.ld;
    const int64_t row = i * p.ld_out;
    if (vec) {
      const int64_t x = j * 4;
      if (x + 4 <= p.M) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(src + x));
        float4 u;
        u.x = iso_value(f.x, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t);
        u.y = iso_value(f.y, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t);
        u.z = iso_value(f.z, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t);
        u.w = iso_value(f.w, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t);
        iso_store4<BF16>(p.U, row + x, u);
      } else {
        for (int64_t xx = x; xx < p.M; ++xx)
          iso_store1<BF16>(p.U, row + xx,
                           iso_value(__ldg(src + xx), p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t));
      }
    } else {
      iso_store1<BF16>(p.U, row + j,
                       iso_value(__ldg(src + j), p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t));
    }
  }
}

cudaError_t launch_iso(const IsoParams& p, cudaStream_t s) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t work = p.N * ((p.M + 3) / 4);
  int64_t blocks = (work + 255) / 256;
  const int64_t cap = static_cast<int64_t>(sms) * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  if (p.out_bf16)
    iso_kernel<true><<<static_cast<int>(blocks), 256, 0, s>>>(p);
  else
    iso_kernel<false><<<static_cast<int>(blocks), 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace pidk
