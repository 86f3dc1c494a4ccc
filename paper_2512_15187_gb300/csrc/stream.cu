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
    __stcs(reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(base) + off), v);
  } else {
    __stcs(reinterpret_cast<float4*>(static_cast<float*>(base) + off), u);
  }
}

template <bool BF16>
__device__ __forceinline__ void iso_store1(void* base, int64_t off, float u) {
  if constexpr (BF16) static_cast<__nv_bfloat16*>(base)[off] = __float2bfloat16_rn(u);
  else static_cast<float*>(base)[off] = u;
}

constexpr int kIsoThreads = 256;
constexpr int kIsoUnroll = 4;   // 16-byte loads in flight per thread

template <int KIND>
__device__ __forceinline__ float4 iso_map4(const float4& f, const IsoParams& p) {
  if constexpr (KIND == ISO_NORMAL) {   // bitwise four scalar evaluations
    const float2 a = iso_normal2(make_float2(f.x, f.y), p.iso_mu, p.iso_inv);
    const float2 b = iso_normal2(make_float2(f.z, f.w), p.iso_mu, p.iso_inv);
    return make_float4(a.x, a.y, b.x, b.y);
  } else {
    return make_float4(iso_value(f.x, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t),
                       iso_value(f.y, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t),
                       iso_value(f.z, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t),
                       iso_value(f.w, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t));
  }
}

// HBM-bound: 4 B read and 4 (2) B written per element. Rows lie along the grid's y axis, so no
// element divides its index; contiguous ensembles come as one row, whatever M is. VEC: rows
// aligned for 4-element accesses; else element by element. A thread has four accesses in flight:
// along its row, a CTA per row, or (SHORT) one each in four rows, 1 << lg_row threads to a row.
// 64 fields of 2048^2 cells to FP32: 0.453 -> 0.304 ms (7.1 TB/s) against one element group per
// grid-stride step with a 64-bit division; 100 000 rows of 16 cells, 32 apart: 114 -> 16 us against
// a CTA per row.
template <bool BF16, int KIND, bool VEC, bool SHORT>
__global__ void __launch_bounds__(kIsoThreads) iso_kernel(const __grid_constant__ IsoParams p) {
  constexpr int W = VEC ? 4 : 1;
  const int rows = SHORT ? kIsoThreads >> p.lg_row : 1;              // side by side in the CTA
  const int t = SHORT ? static_cast<int>(threadIdx.x) & ((1 << p.lg_row) - 1) : static_cast<int>(threadIdx.x);
  const int64_t x0 = SHORT ? t * W : static_cast<int64_t>(blockIdx.x) * kIsoThreads * kIsoUnroll * W + t * W;
  const int64_t step = SHORT ? int64_t(rows) * kIsoUnroll : 1;       // rows of the CTA at a time
  auto cell = [&](int u) { return SHORT ? x0 : x0 + static_cast<int64_t>(u) * kIsoThreads * W; };
  for (int64_t i0 = blockIdx.y * step + (SHORT ? threadIdx.x >> p.lg_row : 0); i0 < p.N; i0 += gridDim.y * step) {
    auto row = [&](int u) { return SHORT ? i0 + u * rows : i0; };
    if constexpr (VEC) {
      float4 f[kIsoUnroll];
#pragma unroll
      for (int u = 0; u < kIsoUnroll; ++u) {
        const int64_t x = cell(u), i = row(u);
        f[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < p.N && x + 4 <= p.M) f[u] = __ldcs(reinterpret_cast<const float4*>(p.F + i * p.ld + x));
      }
#pragma unroll
      for (int u = 0; u < kIsoUnroll; ++u) {
        const int64_t x = cell(u), i = row(u);
        if (i >= p.N) continue;
        if (x + 4 <= p.M) {
          iso_store4<BF16>(p.U, i * p.ld_out + x, iso_map4<KIND>(f[u], p));
        } else {
          for (int64_t xx = x; xx < p.M; ++xx)
            iso_store1<BF16>(p.U, i * p.ld_out + xx,
                             iso_value(__ldg(p.F + i * p.ld + xx), p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t));
        }
      }
    } else {
      float f[kIsoUnroll];
#pragma unroll
      for (int u = 0; u < kIsoUnroll; ++u) {
        const int64_t x = cell(u), i = row(u);
        f[u] = i < p.N && x < p.M ? __ldcs(p.F + i * p.ld + x) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kIsoUnroll; ++u) {
        const int64_t x = cell(u), i = row(u);
        if (i < p.N && x < p.M)
          iso_store1<BF16>(p.U, i * p.ld_out + x, iso_value(f[u], p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t));
      }
    }
  }
}

template <bool BF16, bool VEC, bool SHORT>
static void iso_launch_kind(const IsoParams& p, dim3 grid, cudaStream_t s) {
  if (p.iso_mode == ISO_NORMAL) iso_kernel<BF16, ISO_NORMAL, VEC, SHORT><<<grid, kIsoThreads, 0, s>>>(p);
  else iso_kernel<BF16, ISO_NONE, VEC, SHORT><<<grid, kIsoThreads, 0, s>>>(p);
}

template <bool BF16>
static void iso_launch(const IsoParams& q, cudaStream_t s) {
  IsoParams p = q;
  if (p.ld == p.M && p.ld_out == p.M) {   // contiguous: one row of N M elements
    p.M *= p.N;
    p.N = 1;
  }
  // rows that start on 16 bytes in the input and on 4 elements in the output
  const bool vec = (p.N == 1 || ((p.ld & 3) == 0 && (p.ld_out & 3) == 0)) &&
                   (reinterpret_cast<uintptr_t>(p.F) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(p.U) & (BF16 ? 7 : 15)) == 0;
  // rows of up to one access per thread share a CTA
  const int64_t accesses = vec ? (p.M + 3) / 4 : p.M;
  const bool is_short = p.N > 1 && accesses <= kIsoThreads;
  p.lg_row = 0;
  while (is_short && (int64_t(1) << p.lg_row) < accesses) ++p.lg_row;
  const int64_t gx = is_short ? 1 : (accesses + kIsoThreads * kIsoUnroll - 1) / (kIsoThreads * kIsoUnroll);
  const int64_t per_y = is_short ? int64_t(kIsoThreads >> p.lg_row) * kIsoUnroll : 1;
  const int64_t gy = (p.N + per_y - 1) / per_y;
  const dim3 grid(static_cast<unsigned>(gx), static_cast<unsigned>(gy < 65535 ? gy : 65535));
  if (vec && is_short) iso_launch_kind<BF16, true, true>(p, grid, s);
  else if (vec) iso_launch_kind<BF16, true, false>(p, grid, s);
  else if (is_short) iso_launch_kind<BF16, false, true>(p, grid, s);
  else iso_launch_kind<BF16, false, false>(p, grid, s);
}

cudaError_t launch_iso(const IsoParams& p, cudaStream_t s) {
  if (p.out_bf16) iso_launch<true>(p, s);
  else iso_launch<false>(p, s);
  return cudaGetLastError();
}

}  // namespace pidk
