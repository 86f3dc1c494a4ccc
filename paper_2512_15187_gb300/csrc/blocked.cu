// PID-mean and exact full PID for ensembles beyond one CTA's tile (N > 512 members).
//
// The fused streaming kernel holds every member of a cell tile on chip, which bounds N by
// the rows one CTA group can own. Larger ensembles go through three simpler passes per
// streaming pass, all over the member-major data [N][ld]:
//   1. colsum_kernel  per block of kBlockRows members, the column sum
//                     s_b(x) = sum_{j in b} c_j u_j(x) (compensated FP32), one row per block;
//   2. combine_kernel s(x) = sum_b s_b(x) in block order, in FP64, stored as FP32;
//   3. accum_kernel   per member i and chunk of cells, m_i = sum_x w u_i and
//                     A_i = sum_x w u_i s (FP32 per lane, one warp per (member, chunk)),
//                     written as the same per-chunk partials the fused kernel writes.
// With c_j = 1 this is PID-mean's pass (A_i = N x the sum against u_bar, Eq. 15-16); with
// c_j = 1/(N m_j) it is the second pass of the exact full PID (IN_out of Eq. 10 with the
// sums of Eq. 14). The isovalue map of Sec. 3.5 is applied to each element as it is read.
// rank_kernel ranks the members.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "capi_internal.h"
#include "device.cuh"
#include "internal.h"

namespace pidk {

constexpr int kBlockRows = 512;      // members per column-sum block
constexpr int kAccChunk = 8192;      // cells per accumulation chunk (one partial per member)

struct BlockedParams {
  const float* data;     // [N][ld]
  const float* w;        // [M] or nullptr
  const float* coef;     // [N] column-sum coefficients, or nullptr (every c_j = 1)
  float* S;              // [n_blocks][ldS] per-block column sums
  float* s;              // [ldS] combined column sum
  float* part;           // [n_chunks][2N]
  int64_t N, M, ld, ldS;
  int32_t n_blocks, n_chunks;
  int32_t iso_mode;
  float iso_mu, iso_inv, iso_t;
};

__device__ __forceinline__ float blocked_u(const BlockedParams& p, float f) {
  return p.iso_mode == ISO_NONE ? f : iso_value(f, p.iso_mode, p.iso_mu, p.iso_inv, p.iso_t);
}

// Grid: x over 4-cell groups, y over member blocks. Kahan-compensated FP32 sums.
__global__ void __launch_bounds__(256) colsum_kernel(const __grid_constant__ BlockedParams p) {
  const int64_t x = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) * 4;
  if (x >= p.M) return;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * kBlockRows;
  const int64_t r1 = min(r0 + kBlockRows, p.N);
  const bool vec = (p.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(p.data) & 15) == 0 &&
                   x + 4 <= p.M;
  float sum[4] = {0.f, 0.f, 0.f, 0.f}, comp[4] = {0.f, 0.f, 0.f, 0.f};
  for (int64_t i = r0; i < r1; ++i) {
    const float* row = p.data + i * p.ld + x;
    float v[4];
    if (vec) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(row));
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = x + k < p.M ? __ldg(row + k) : 0.f;
    }
    const float c = p.coef ? __ldg(p.coef + i) : 1.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float term = c * blocked_u(p, v[k]) - comp[k];
      const float t = sum[k] + term;
      comp[k] = (t - sum[k]) - term;
      sum[k] = t;
    }
  }
  float* out = p.S + static_cast<int64_t>(blockIdx.y) * p.ldS + x;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (x + k < p.M) out[k] = sum[k];
}

__global__ void __launch_bounds__(256) combine_kernel(const __grid_constant__ BlockedParams p) {
  const int64_t x = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (x >= p.M) return;
  double acc = 0.0;
  for (int b = 0; b < p.n_blocks; ++b) acc += static_cast<double>(p.S[b * p.ldS + x]);
  p.s[x] = static_cast<float>(acc);
}

// One warp per (member, chunk): lanes stride the chunk's cells 4 at a time.
__global__ void __launch_bounds__(256) accum_kernel(const __grid_constant__ BlockedParams p) {
  const int64_t wid = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= p.N * p.n_chunks) return;
  const int64_t i = wid % p.N;
  const int64_t c = wid / p.N;
  const int64_t x0 = c * kAccChunk;
  const int64_t x1 = min(x0 + kAccChunk, p.M);
  const bool vec = (p.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(p.data) & 15) == 0 &&
                   (p.w == nullptr || (reinterpret_cast<uintptr_t>(p.w) & 15) == 0);
  const float* row = p.data + i * p.ld;
  float m = 0.f, a = 0.f;
  for (int64_t x = x0 + lane * 4; x < x1; x += 32 * 4) {
    float v[4], sv[4], wv[4] = {1.f, 1.f, 1.f, 1.f};
    if (vec && x + 4 <= x1) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(row + x));
      const float4 qs = __ldg(reinterpret_cast<const float4*>(p.s + x));
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
      sv[0] = qs.x; sv[1] = qs.y; sv[2] = qs.z; sv[3] = qs.w;
      if (p.w) {
        const float4 qw = __ldg(reinterpret_cast<const float4*>(p.w + x));
        wv[0] = qw.x; wv[1] = qw.y; wv[2] = qw.z; wv[3] = qw.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool in = x + k < x1;
        v[k] = in ? __ldg(row + x + k) : 0.f;
        sv[k] = in ? __ldg(p.s + x + k) : 0.f;
        if (p.w) wv[k] = in ? __ldg(p.w + x + k) : 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (x + k < x1) {
        const float t = wv[k] * blocked_u(p, v[k]);
        m += t;
        a = fmaf(t, sv[k], a);
      }
    }
  }
  m = warp_sum(m);
  a = warp_sum(a);
  if (lane == 0) {
    p.part[c * 2 * p.N + i] = m;
    p.part[c * 2 * p.N + p.N + i] = a;
  }
}

// ---- finalisation: the outputs of Eq. 10 / Eq. 16 from the chunk partials ----

constexpr int kLargeThreads = 256;
constexpr int kLargeMembers = 32;                          // members per CTA of the reduction
constexpr int kLargeRows = kLargeThreads / kLargeMembers;  // row groups that share a column

struct LargeFin {
  const float* part;       // [n_chunks][2N]
  int64_t N;
  int32_t n_chunks, kind;  // FinKind (no Gram)
  double* sums;            // [2N] m, N A of the first pass; [N] B of the second
  double* block_mass;      // [ceil(N / 32)] mass sums, then their total
  unsigned int* ticket;    // zero before the launch; the last CTA resets it
  float* coef;             // FIN_LIN1 writes the coefficients; FIN_WMEAN reads them
  double *depth, *in_in, *in_out, *mass, *mean_depth;
};

// Column i of the partials summed over this thread's rows.
__device__ __forceinline__ Sum3 large_column(const float* src, int64_t stride, int rows, int r0) {
  Sum3 s;
  int r = r0;
  for (; r + 3 * kLargeRows < rows; r += 4 * kLargeRows) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldcg(src + (r + k * kLargeRows) * stride);
#pragma unroll
    for (int k = 0; k < 4; ++k) sum3_add(s, v[k]);
  }
  for (; r < rows; r += kLargeRows) sum3_add(s, __ldcg(src + r * stride));
  return s;
}

// The sum of a column's row groups in FP64; sums that leave the finite FP32 range again in FP64.
__device__ __forceinline__ double large_total(const Sum3 (*acc)[kLargeMembers], int lane,
                                              const float* src, int64_t stride, int rows) {
  Sum3 s = acc[0][lane];
#pragma unroll
  for (int g = 1; g < kLargeRows; ++g) sum3_add(s, acc[g][lane]);
  if (fabsf(s.x) <= kMaxFloat) return sum3_value(s);
  double v = 0.0;
  for (int r = 0; r < rows; ++r) v += static_cast<double>(__ldcg(src + r * stride));
  return v;
}

// Member sums over the chunks, and the masses' total: 32 members per CTA, the CTAs' mass sums
// added by the last CTA in order. (One CTA used to form every member's outputs as well, with
// FP64 divisions at two operations per clock: 107 us for 10 000 members.)
__global__ void __launch_bounds__(kLargeThreads) large_sum_kernel(const __grid_constant__ LargeFin p) {
  __shared__ Sum3 acc[2][kLargeRows][kLargeMembers];
  __shared__ double red[kLargeThreads];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, rg = threadIdx.x >> 5;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * kLargeMembers + lane;
  const int64_t stride = 2 * p.N;
  const bool second = p.kind == FIN_LIN2, in = i < p.N;
  const Sum3 zero{};
  acc[0][rg][lane] = in && !second ? large_column(p.part + i, stride, p.n_chunks, rg) : zero;
  acc[1][rg][lane] = in ? large_column(p.part + p.N + i, stride, p.n_chunks, rg) : zero;
  __syncthreads();
  if (second) {
    if (rg == 0 && in) p.sums[2 * p.N + i] = large_total(acc[1], lane, p.part + p.N + i, stride, p.n_chunks);
    return;
  }
  if (rg == 1 && in) p.sums[p.N + i] = large_total(acc[1], lane, p.part + p.N + i, stride, p.n_chunks);
  if (rg == 0) {
    double m = 0.0;
    if (in) {
      m = large_total(acc[0], lane, p.part + i, stride, p.n_chunks);
      p.sums[i] = m;
      if (p.kind == FIN_WMEAN) m *= static_cast<double>(p.coef[i]);
    }
    m = warp_sum(m);
    if (lane == 0) {
      p.block_mass[blockIdx.x] = m;
      __threadfence();
      last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (unsigned k = threadIdx.x; k < gridDim.x; k += kLargeThreads) t += __ldcg(p.block_mass + k);
  red[threadIdx.x] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    t = red[threadIdx.x];
    for (int k = 32; k < kLargeThreads; k += 32) t += red[threadIdx.x + k];
    t = warp_sum(t);
    if (threadIdx.x == 0) {
      p.block_mass[gridDim.x] = t;
      *p.ticket = 0u;
    }
  }
}

__global__ void __launch_bounds__(kLargeThreads) large_out_kernel(const __grid_constant__ LargeFin p, unsigned blocks) {
  grid_dependency_wait();
  const int64_t i = static_cast<int64_t>(blockIdx.x) * kLargeThreads + threadIdx.x;
  if (i >= p.N) return;
  const bool second = p.kind == FIN_LIN2;
  const double m = __ldcg(p.sums + i), A = __ldcg(p.sums + p.N + i);
  if (p.kind == FIN_LIN1)
    p.coef[i] = m > 0.0 ? static_cast<float>(1.0 / (static_cast<double>(p.N) * m)) : 0.0f;
  if (p.mass && !second) p.mass[i] = m;
  if (p.kind == FIN_LIN1 && !p.mean_depth) return;
  const double in_in = m > 0.0 ? A / (p.kind == FIN_WMEAN ? m : m * static_cast<double>(p.N)) : 0.0;
  double in_out = 0.0;
  if (second) {
    in_out = __ldcg(p.sums + 2 * p.N + i);
  } else {
    const double total = __ldcg(p.block_mass + blocks);
    in_out = total > 0.0 ? A / total : 0.0;
    if (p.mean_depth) p.mean_depth[i] = fmin(in_in, in_out);
  }
  if (p.kind == FIN_LIN1) return;
  if (p.depth) p.depth[i] = fmin(in_in, in_out);
  if (p.in_in) p.in_in[i] = in_in;
  if (p.in_out) p.in_out[i] = in_out;
}

// rank[i] += number of members j in this block's slice that are deeper than i, or as deep with a
// lower index. A thread ranks four members against each key it reads from shared memory, and
// slices that lie wholly below or above the members need no index comparison: about 14
// instructions per four pairs, and enough slices to fill the GPU (10 000 members: one member
// per thread and two slices took 141 us; with the finalisation above, 1910 -> 1713 us a call). The counts are integers, so adding them with atomics
// gives the same ranks in any order. rank must be zero before the launch.
constexpr int kRankThreads = 256;
constexpr int kRankPer = 4;
constexpr int kRankMembers = kRankThreads * kRankPer;
constexpr int kRankSlice = 256;                        // largest slice: one key per thread

__global__ void __launch_bounds__(kRankThreads) rank_kernel(const double* depth, int64_t N, int32_t slice,
                                                            int32_t* rank) {
  __shared__ unsigned long long tile[kRankSlice];   // order keys of the slice's depths
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kRankMembers;
  const int64_t j0 = static_cast<int64_t>(blockIdx.y) * slice;
  const int n = static_cast<int>(min(static_cast<int64_t>(slice), N - j0));
  if (threadIdx.x < n) tile[threadIdx.x] = order_key(depth[j0 + threadIdx.x]);
  unsigned long long ki[kRankPer];
  int cnt[kRankPer];
#pragma unroll
  for (int k = 0; k < kRankPer; ++k) {
    const int64_t i = i0 + k * kRankThreads + threadIdx.x;
    ki[k] = order_key(i < N ? depth[i] : 0.0);
    cnt[k] = 0;
  }
  __syncthreads();
  if (j0 + n <= i0) {                       // every j below every i: ties count
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const unsigned long long kj = tile[j];
#pragma unroll
      for (int k = 0; k < kRankPer; ++k) cnt[k] += kj >= ki[k];
    }
  } else if (j0 >= i0 + kRankMembers) {     // every j above every i: ties do not
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const unsigned long long kj = tile[j];
#pragma unroll
      for (int k = 0; k < kRankPer; ++k) cnt[k] += kj > ki[k];
    }
  } else {
    for (int j = 0; j < n; ++j) {
      const unsigned long long kj = tile[j];
#pragma unroll
      for (int k = 0; k < kRankPer; ++k) {
        const int64_t i = i0 + k * kRankThreads + threadIdx.x;
        cnt[k] += (kj > ki[k]) || (kj == ki[k] && j0 + j < i);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kRankPer; ++k) {
    const int64_t i = i0 + k * kRankThreads + threadIdx.x;
    if (i < N && cnt[k] > 0) atomicAdd(rank + i, cnt[k]);
  }
}

}  // namespace pidk

namespace pidh {

using namespace pidk;

static int64_t rup(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

static pid_status blocked_pass(pid_handle h, const BlockedParams& p, double bytes, cudaStream_t s) {
  ProfScope ps(h, PID_KERNEL_STREAM, bytes, 0.0, s);
  const dim3 gc(static_cast<unsigned>((p.M + 4 * 256 - 1) / (4 * 256)), static_cast<unsigned>(p.n_blocks));
  colsum_kernel<<<gc, 256, 0, s>>>(p);
  combine_kernel<<<static_cast<unsigned>((p.M + 255) / 256), 256, 0, s>>>(p);
  const int64_t warps = p.N * p.n_chunks;
  accum_kernel<<<static_cast<unsigned>((warps * 32 + 255) / 256), 256, 0, s>>>(p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(h, e, "member-blocked pass launch");
  return PID_OK;
}

static pid_status large_fin(pid_handle h, const LargeFin& p, cudaStream_t s) {
  ProfScope ps(h, PID_KERNEL_FINALIZE, 0.0, 0.0, s);
  const unsigned blocks = static_cast<unsigned>((p.N + kLargeMembers - 1) / kLargeMembers);
  large_sum_kernel<<<blocks, kLargeThreads, 0, s>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((p.N + kLargeThreads - 1) / kLargeThreads));
    cfg.blockDim = dim3(kLargeThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, large_out_kernel, p, blocks);
  }
  if (e != cudaSuccess) return cuda_fail(h, e, "finalize launch");
  return PID_OK;
}

pid_status run_blocked(pid_handle h, const EnsInput& in, const EnsOutputs& out, cudaStream_t s) {
  if (in.mode == PID_MODE_FULL && in.precision != PID_FP32)
    return fail(h, PID_ERR_UNSUPPORTED,
                "the tensor-core Gram takes N <= 512; use PID_MODE_FULL_LINEAR");
  if (in.validate)
    return fail(h, PID_ERR_UNSUPPORTED, "validation is not available for N > 512");
  const bool linear = in.mode != PID_MODE_MEAN;
  const int64_t N = in.N, M = in.M;
  const int64_t ldS = rup(M, 4);
  const int n_blocks = static_cast<int>((N + kBlockRows - 1) / kBlockRows);
  const int n_chunks = static_cast<int>((M + kAccChunk - 1) / kAccChunk);
  const size_t S_bytes = rup(static_cast<int64_t>(n_blocks) * ldS * 4, 256);
  const size_t s_bytes = rup(ldS * 4, 256);
  const size_t part_bytes = rup(static_cast<int64_t>(n_chunks) * 2 * N * 4, 256);
  const int64_t fin_blocks = (N + kLargeMembers - 1) / kLargeMembers;
  const size_t sums_bytes = rup((3 * N + fin_blocks + 1) * 8, 256);
  const size_t coef_bytes = rup(N * 4, 256);
  const size_t dtmp_bytes = (out.rank && !out.depth) ? rup(N * 8, 256) : 0;
  pid_status st = ensure_workspace(h, S_bytes + s_bytes + part_bytes + sums_bytes + coef_bytes +
                                          dtmp_bytes, s);
  if (st != PID_OK) return st;
  char* ws = static_cast<char*>(h->ws);
  BlockedParams p;
  std::memset(&p, 0, sizeof(p));
  p.S = reinterpret_cast<float*>(ws);
  p.s = reinterpret_cast<float*>(ws + S_bytes);
  p.part = reinterpret_cast<float*>(ws + S_bytes + s_bytes);
  double* sums = reinterpret_cast<double*>(ws + S_bytes + s_bytes + part_bytes);
  float* coef = reinterpret_cast<float*>(ws + S_bytes + s_bytes + part_bytes + sums_bytes);
  double* dtmp = dtmp_bytes ? reinterpret_cast<double*>(ws + S_bytes + s_bytes + part_bytes +
                                                        sums_bytes + coef_bytes)
                            : nullptr;
  p.data = in.data; p.w = in.w; p.N = N; p.M = M; p.ld = in.ld; p.ldS = ldS;
  p.n_blocks = n_blocks; p.n_chunks = n_chunks;
  iso_fill(in.is_field ? &in.iso : nullptr, &p.iso_mode, &p.iso_mu, &p.iso_inv, &p.iso_t);
  const double bytes = 4.0 * N * M + (in.w ? 4.0 * M : 0.0);

  LargeFin fd;
  std::memset(&fd, 0, sizeof(fd));
  fd.part = p.part;
  fd.N = N;
  fd.n_chunks = n_chunks;
  fd.sums = sums;
  fd.block_mass = sums + 3 * N;
  fd.coef = coef;
  fd.ticket = h->ticket;
  fd.depth = out.depth ? out.depth : dtmp;
  fd.in_in = out.in_in;
  fd.in_out = out.in_out;
  fd.mass = out.mass;
  fd.mean_depth = out.mean_depth;

  if (in.member_weights) {   // PID-mean against the weighted mean contour: one pass
    if ((st = launch_member_coef_one(h, in.member_weights, N, coef, s)) != PID_OK) return st;
    p.coef = coef;
    if ((st = blocked_pass(h, p, bytes, s)) != PID_OK) return st;
    fd.kind = FIN_WMEAN;
    if ((st = large_fin(h, fd, s)) != PID_OK) return st;
  } else if ((st = blocked_pass(h, p, bytes, s)) != PID_OK) {
    return st;
  } else if (!linear) {
    fd.kind = FIN_MEAN;
    if ((st = large_fin(h, fd, s)) != PID_OK) return st;
  } else {
    LargeFin f1 = fd;
    f1.kind = FIN_LIN1;
    if ((st = large_fin(h, f1, s)) != PID_OK) return st;
    p.coef = coef;
    if ((st = blocked_pass(h, p, bytes, s)) != PID_OK) return st;
    LargeFin f2 = fd;
    f2.kind = FIN_LIN2;
    if ((st = large_fin(h, f2, s)) != PID_OK) return st;
  }
  if (out.rank) {
    // slices of at most 256 keys, shorter ones where the members alone do not give every SM
    // a few blocks
    const int64_t groups = (N + kRankMembers - 1) / kRankMembers;
    int64_t slice = rup((N * groups + 4 * h->sms - 1) / (4 * h->sms), 32);
    slice = std::max<int64_t>(32, std::min<int64_t>(slice, kRankSlice));
    cudaError_t e = cudaMemsetAsync(out.rank, 0, static_cast<size_t>(N) * sizeof(int32_t), s);
    if (e != cudaSuccess) return cuda_fail(h, e, "rank reset");
    rank_kernel<<<dim3(static_cast<unsigned>(groups), static_cast<unsigned>((N + slice - 1) / slice)),
                  kRankThreads, 0, s>>>(fd.depth, N, static_cast<int32_t>(slice), out.rank);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(h, e, "rank kernel launch");
  }
  return PID_OK;
}

}  // namespace pidh
