// Contour boxplot bands (Sec. 6): binarise every member at a probability threshold and
// collect, per cell, the unions and intersections over the deepest members and over all
// members, and the median member. One HBM-bound pass over the ensemble: 4 B read per
// member-cell, 1 B written per cell.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "capi_internal.h"
#include "internal.h"

namespace pidk {

struct BandParams {
  const float* data;     // [N][ld]
  const int32_t* rank;   // [N], 0 = deepest
  uint8_t* out;          // [M]
  int64_t N, M, ld;
  int32_t n_inner;       // members with rank < n_inner form the inner population
  int32_t cmp;           // 0: value > thr, 1: value < thr, 2: value > thr (field, super-level),
                         // 3: thr < value < thr2 (field, level map)
  float thr, thr2;
};

constexpr int kBandThreads = 256;
constexpr int kBandChunk = 1024;     // members whose flags are staged in shared memory at a time

// Whether a value's soft mask is above the threshold.
template <int CMP>
__device__ __forceinline__ bool band_in(float v, float t, float t2) {
  if constexpr (CMP == 1) return v < t;
  else if constexpr (CMP == 3) return v > t && v < t2;
  else return v > t;
}

// HBM-bound: 4 B read per member-cell. The kernel waits on memory alone, so what counts is the
// loads in flight: a thread issues U rows' loads before it looks at the first, and the grid is
// not capped, so no wave is left nearly empty. 64 fields of 2048^2 cells: 0.250 -> 0.152 ms,
// 7.1 TB/s, against one load at a time in a grid-stride loop. A member's part is
// one word of flags in shared memory: bits to set where its mask is in (unions, median), and
// bits that mark an intersection as broken where it is not, so a value costs a compare, a
// select and an OR whatever its rank.
//   VEC: 4 consecutive cells per thread, 16-byte loads (aligned rows); else one cell per
//   thread, neighbouring threads on neighbouring cells.
template <int CMP, bool VEC>
__global__ void __launch_bounds__(kBandThreads) bands_kernel(const __grid_constant__ BandParams p) {
  constexpr int C = VEC ? 4 : 1;
  constexpr int U = VEC ? 8 : 16;
  __shared__ uint8_t flag[kBandChunk];
  __shared__ long long s_median;
  __shared__ int s_inner;
  const int64_t x = (static_cast<int64_t>(blockIdx.x) * kBandThreads + threadIdx.x) * C;
  // The median member: the last one of rank 0 (ranks within groups repeat).
  if (threadIdx.x == 0) { s_median = -1; s_inner = 0; }
  __syncthreads();
  long long med = -1;
  for (int64_t i = threadIdx.x; i < p.N; i += kBandThreads)
    if (__ldg(p.rank + i) == 0) med = i;
  if (med >= 0) atomicMax(&s_median, med);
  const bool in = x < p.M;
  const float* src = p.data + (in ? x : 0);
  uint32_t acc[C];
#pragma unroll
  for (int c = 0; c < C; ++c) acc[c] = 0;
  for (int64_t i0 = 0; i0 < p.N; i0 += kBandChunk) {
    const int n = static_cast<int>(min(static_cast<int64_t>(kBandChunk), p.N - i0));
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += kBandThreads) {
      const bool inner = __ldg(p.rank + i0 + k) < p.n_inner;
      // in: all-union 4, inner union 1, median 16; not in: all broken 8, inner broken 2
      flag[k] = static_cast<uint8_t>(12 | (inner ? 3 : 0) | (i0 + k == s_median ? 16 : 0));
      if (inner) s_inner = 1;
    }
    __syncthreads();
    if (!in) continue;
    int k = 0;
    for (; k + U <= n; k += U) {
      float v[U][C];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float* row = src + (i0 + k + u) * p.ld;
        if constexpr (VEC) {
          const float4 q = __ldcs(reinterpret_cast<const float4*>(row));
          v[u][0] = q.x; v[u][1] = q.y; v[u][2] = q.z; v[u][3] = q.w;
        } else {
          v[u][0] = __ldcs(row);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t f = flag[k + u], set = f & 0x15u, broken = f & 0x0au;
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] |= band_in<CMP>(v[u][c], p.thr, p.thr2) ? set : broken;
      }
    }
    for (; k < n; ++k) {
      const float* row = src + (i0 + k) * p.ld;
      const uint32_t f = flag[k], set = f & 0x15u, broken = f & 0x0au;
      float v[C];
      if constexpr (VEC) {
        const float4 q = __ldcs(reinterpret_cast<const float4*>(row));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
      } else {
        v[0] = __ldcs(row);
      }
#pragma unroll
      for (int c = 0; c < C; ++c) acc[c] |= band_in<CMP>(v[c], p.thr, p.thr2) ? set : broken;
    }
  }
  if (!in) return;
  // an empty inner population intersects to nothing
  const uint32_t keep = s_inner ? 0x1fu : 0x1du;
#pragma unroll
  for (int c = 0; c < C; ++c) acc[c] = (acc[c] ^ 0x0au) & keep;
  if constexpr (VEC) {
    *reinterpret_cast<uint32_t*>(p.out + x) = acc[0] | (acc[1] << 8) | (acc[2] << 16) | (acc[3] << 24);
  } else {
    p.out[x] = static_cast<uint8_t>(acc[0]);
  }
}

template <int CMP>
static void bands_launch(const BandParams& p, int sms, cudaStream_t s) {
  // 16-byte loads where every row and the output allow them and the cells are enough to fill
  // the GPU with a quarter of the threads; small grids spread one cell per thread.
  const bool vec = (p.ld & 3) == 0 && (p.M & 3) == 0 && (reinterpret_cast<uintptr_t>(p.data) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(p.out) & 3) == 0 &&
                   p.M >= int64_t(sms) * 4 * kBandThreads * 2;
  const int64_t cells = kBandThreads * (vec ? 4 : 1);
  const unsigned grid = static_cast<unsigned>((p.M + cells - 1) / cells);
  if (vec) bands_kernel<CMP, true><<<grid, kBandThreads, 0, s>>>(p);
  else bands_kernel<CMP, false><<<grid, kBandThreads, 0, s>>>(p);
}

cudaError_t launch_bands(const BandParams& p, int sms, cudaStream_t s) {
  if (p.cmp == 1) bands_launch<1>(p, sms, s);
  else if (p.cmp == 3) bands_launch<3>(p, sms, s);
  else bands_launch<0>(p, sms, s);
  return cudaGetLastError();
}

}  // namespace pidk

using namespace pidk;
using namespace pidh;

namespace {

// z with Phi(z) = p (0 < p < 1), by bisection on the FP64 complementary error function.
double normal_quantile(double pr) {
  double lo = -40.0, hi = 40.0;
  for (int it = 0; it < 200 && hi - lo > 0.0; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid == lo || mid == hi) break;
    if (0.5 * std::erfc(-mid / std::sqrt(2.0)) < pr) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}

float float_at_or_above(double v) {
  float f = static_cast<float>(v);
  if (static_cast<double>(f) < v) f = std::nextafter(f, INFINITY);
  return f;
}

float float_at_or_below(double v) {
  float f = static_cast<float>(v);
  if (static_cast<double>(f) > v) f = std::nextafter(f, -INFINITY);
  return f;
}

}  // namespace

extern "C" pid_status pid_contour_bands(pid_handle h, const float* data, int64_t N, int64_t M,
                                        int64_t ld, const pid_iso* iso, const int32_t* rank,
                                        double tau, double inner_fraction, uint8_t* bands,
                                        void* stream) {
  pid_status st = check_shape(h, data, N, M, ld);
  if (st == PID_ERR_UNSUPPORTED && N > kMaxMembers) st = PID_OK;  // elementwise: any N
  if (st != PID_OK) return st;
  if (iso && (st = check_iso(h, iso)) != PID_OK) return st;
  if (!rank || !bands) return fail(h, PID_ERR_INVALID_ARG, "rank and bands must be non-NULL");
  if (!(tau > 0.0 && tau < 1.0)) return fail(h, PID_ERR_INVALID_ARG, "tau must be in (0, 1)");
  if (!(inner_fraction > 0.0 && inner_fraction <= 1.0))
    return fail(h, PID_ERR_INVALID_ARG, "inner_fraction must be in (0, 1]");
  BandParams p;
  std::memset(&p, 0, sizeof(p));
  p.data = data; p.rank = rank; p.out = bands; p.N = N; p.M = M; p.ld = ld;
  p.n_inner = static_cast<int32_t>(std::ceil(inner_fraction * static_cast<double>(N)));
  // The binarisation u > tau, decided exactly: for soft masks u > tau <=> u > (largest float
  // <= tau); for fields u is monotone in F, so u(F) > tau <=> F beyond F_tau with
  // u(F_tau) = tau, i.e. F compared with the float nearest F_tau on the correct side.
  if (!iso) {
    p.cmp = 0;
    p.thr = float_at_or_below(tau);
  } else if (iso->kind == PID_ISO_UNIFORM) {
    const double h = iso->sigma;
    if (!iso->superlevel) {            // u = (mu + h - F) / 2h > tau <=> F < mu + h (1 - 2 tau)
      p.cmp = 1;
      p.thr = float_at_or_above(iso->mu + h * (1.0 - 2.0 * tau));
    } else {                           // u = (F - mu + h) / 2h > tau <=> F > mu + h (2 tau - 1)
      p.cmp = 2;
      p.thr = float_at_or_below(iso->mu + h * (2.0 * tau - 1.0));
    }
  } else if (iso->kind == PID_ISO_LEVEL) {  // 1 - |F - mu| / h > tau <=> |F - mu| < h (1 - tau)
    const double r = iso->sigma * (1.0 - tau);
    p.cmp = 3;
    p.thr = float_at_or_below(iso->mu - r);
    p.thr2 = float_at_or_above(iso->mu + r);
  } else if (iso->sigma > 0.0) {
    const double z = normal_quantile(tau);
    if (!iso->superlevel) {            // u = Phi((mu - F) / sigma) > tau <=> F < mu - sigma z
      p.cmp = 1;
      p.thr = float_at_or_above(iso->mu - iso->sigma * z);
    } else {                           // u = Phi((F - mu) / sigma) > tau <=> F > mu + sigma z
      p.cmp = 2;
      p.thr = float_at_or_below(iso->mu + iso->sigma * z);
    }
  } else {                             // u in {0, 1}: u > tau <=> u = 1
    p.cmp = iso->superlevel ? 2 : 1;
    p.thr = iso->superlevel ? float_at_or_below(iso->mu) : float_at_or_above(iso->mu);
  }
  DeviceGuard g(h->device);
  ProfScope ps(h, PID_KERNEL_BANDS, 4.0 * N * M + M, 0.0, static_cast<cudaStream_t>(stream));
  cudaError_t e = launch_bands(p, h->sms, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(h, e, "bands kernel launch");
  return PID_OK;
}
