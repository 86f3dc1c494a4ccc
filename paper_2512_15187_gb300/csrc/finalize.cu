// Finalisation: fixed-order reduction of the per-chunk partials, then the inclusion
// fractions, depths and ranks of Eq. 10 / Eq. 16, and the calibration of the tensor-core
// Gram.
//
// The members of an ensemble (up to 512) lie in kFinBlocks contiguous blocks. A cluster of C CTAs
// takes an ensemble, CTA r the blocks r kFinBlocks / C onwards, from the partials to their ranks.
// What one member needs from all the others (the mean contour's mass, the calibration scales, the
// order keys of the depths) is pushed into every CTA's shared memory and separated by cluster
// barriers, so a finalisation is one launch without tickets or round trips through L2.
//
// Every sum is ordered by the blocks, never by C: an ensemble's results are the same bits alone
// and in any batch, whatever C its launch takes.
//
// What bounds it is latency: a chain of an L2 read, a few FP64 operations and barriers. GB300
// issues two FP64 operations per clock and SM, so
//   * the partials, which are FP32 values, are summed as unevaluated sums of three FP32 numbers
//     (Sum3: what is lost lies below FP64's last bit) and become FP64 once per column; a sum that
//     leaves the finite FP32 range is formed again in FP64;
//   * the FP64 divisions and the N^2 rank comparisons are spread over the cluster's SMs.
#include <cuda.h>
#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"

namespace pidk {

namespace {

constexpr int kFinBlocks = 8;      // member blocks, and most CTAs per ensemble: the portable cluster size
constexpr int kFinThreads = 512;
constexpr int kFinWarps = kFinThreads / 32;
constexpr int kFinMaxN = 512;
constexpr int kFinMaxRows = kFinMaxN / kFinBlocks;     // members per block
constexpr int kFinRowsPerWarp = kFinMaxRows / kFinWarps;   // rows that a warp takes at a time

__device__ __forceinline__ const FinDesc& fin_desc(const FinParams& p, int e) {
  return p.descs ? p.descs[e] : p.one;
}

// The barrier of an ensemble's C CTAs.
template <int C>
__device__ __forceinline__ void fin_sync() {
  if constexpr (C == 1) __syncthreads();
  else cluster_sync_all();
}

// Writes v to the shared-memory object at p in each of the ensemble's C CTAs.
template <int C, typename T>
__device__ __forceinline__ void fin_push(T* p, T v) {
  if constexpr (C == 1) {
    *p = v;
  } else {
#pragma unroll
    for (int r = 0; r < C; ++r) st_cluster(cluster_addr(p, r), v);
  }
}

// State shared by the members of one CTA.
template <int C>
struct FinShared {
  double tot[2][kFinMaxN / C];          // m of this CTA's members; N A (or B)
  double csum[kFinBlocks];              // every block's share of the mean contour's mass
  unsigned long long key[kFinMaxN];     // order keys of all depths
};
// Partial column sums of a CTA's blocks (dynamic shared memory): [columns][row groups + 1]. The pad
// keeps both the lanes that write a row group's columns and those that read a column's groups on
// banks of their own.
template <int C>
constexpr size_t fin_acc_bytes(int N = kFinMaxN) {
  int cp = 1;
  while (cp * kFinBlocks < N) cp *= 2;
  return sizeof(Sum3) * (kFinBlocks / C) * (kFinThreads + 2 * cp);
}

// The power of two that holds n >= 1: its exponent.
__device__ __forceinline__ int ceil_log2(int n) { return 32 - __clz(n - 1); }

// Members of one CTA: [m0, m0 + nm) in V blocks of `per` members, the first of them block b0; cp =
// 1 << lg_cp is the power of two that holds a block.
struct FinSpan {
  int N, b0, per, m0, nm, lg_cp, cp;
};
template <int C>
__device__ __forceinline__ FinSpan fin_span(int N, int rank) {
  constexpr int V = kFinBlocks / C;
  FinSpan s;
  s.N = N;
  s.b0 = rank * V;
  s.per = (N + kFinBlocks - 1) / kFinBlocks;
  s.m0 = min(N, s.b0 * s.per);
  s.nm = min(N, s.m0 + V * s.per) - s.m0;
  s.lg_cp = ceil_log2(s.per);
  s.cp = 1 << s.lg_cp;
  return s;
}

// Columns of the [rows][2N] partials that belong to this CTA's members into sh.tot: m and
// N A, or (second) the second half alone. RG row groups take the rows g, g + RG, ... of a column,
// then the groups of a column are summed. RG, and so the order, depends on N and rows alone: as
// many groups as give a thread the 8 loads that it keeps in flight, up to one CTA's threads per
// block.
template <int C>
__device__ void fin_reduce(FinShared<C>& sh, Sum3* acc, const float* part, int rows, const FinSpan& sp,
                           bool second) {
  constexpr int V = kFinBlocks / C;
  const int lg_ncol = sp.lg_cp + (second ? 0 : 1);      // columns of a block, of the CTA
  const int ncol = 1 << lg_ncol, columns = V * ncol;
  const int lg_RG = min(ceil_log2((rows + 7) / 8), ceil_log2(kFinThreads) - lg_ncol);
  const int RG = 1 << lg_RG;
  const int t = threadIdx.x, pitch = RG + 1;
  const int64_t stride = 2 * static_cast<int64_t>(sp.N);
  // the partials of column c, or nullptr for a slot past the CTA's members
  auto column = [&](int c, int* lm, int* half) -> const float* {
    const int col = c & (ncol - 1), slot = col & (sp.cp - 1), v = c >> lg_ncol;
    *half = (second || col >= sp.cp) ? 1 : 0;
    *lm = v * sp.per + slot;
    return slot < sp.per && *lm < sp.nm ? part + *half * sp.N + sp.m0 + *lm : nullptr;
  };
  for (int e = t; e < columns * RG; e += kFinThreads) {
    int lm, half;
    const float* src = column(e & (columns - 1), &lm, &half);
    Sum3 s;
    if (src != nullptr) {
      // the next 8 rows are in flight while these are added (an addition costs 13 instructions)
      float v[8], w[8];
      auto load = [&](float (&x)[8], int r) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = r + k * RG < rows ? __ldcg(src + (r + k * RG) * stride) : 0.f;
      };
      int r = (e >> lg_ncol) / V;
      load(v, r);
      while (r < rows) {
        load(w, r + 8 * RG);
#pragma unroll
        for (int k = 0; k < 8; ++k) sum3_add(s, v[k]);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = w[k];
        r += 8 * RG;
      }
    }
    acc[(e & (columns - 1)) * pitch + ((e >> lg_ncol) / V)] = s;
  }
  __syncthreads();
  const int lg_L = min(5, lg_RG), L = 1 << lg_L;        // lanes that share one column
  const int l = t & (L - 1);
  for (int c0 = 0; L > 1 && c0 < columns; c0 += kFinThreads >> lg_L) {
    const int c = c0 + (t >> lg_L);
    Sum3 s;
    if (c < columns)
      for (int k = l; k < RG; k += L) sum3_add(s, acc[c * pitch + k]);
    for (int o = L / 2; o > 0; o >>= 1) {     // tree: lane 0 ends with the column's sum
      Sum3 other;
      other.x = __shfl_xor_sync(0xffffffffu, s.x, o);
      other.y = __shfl_xor_sync(0xffffffffu, s.y, o);
      other.z = __shfl_xor_sync(0xffffffffu, s.z, o);
      sum3_add(s, other);
    }
    if (c < columns && l == 0) acc[c * pitch] = s;   // in place of the group 0 that this lane alone read
  }
  if (L > 1) __syncthreads();
  // to FP64 with a thread per column (few warps: the FP64 pipe takes 16 clocks an instruction)
  for (int c = t; c < columns; c += kFinThreads) {
    int lm, half;
    const float* src = column(c, &lm, &half);
    if (src == nullptr) continue;
    const Sum3 total = acc[c * pitch];
    double v = sum3_value(total);
    if (!(fabsf(total.x) <= kMaxFloat)) {      // infinities, NaN, or beyond the FP32 range: in FP64
      v = 0.0;
      for (int r = 0; r < rows; ++r) v += static_cast<double>(__ldcg(src + r * stride));
    }
    sh.tot[half][lm] = v;
  }
  __syncthreads();
}

// The blocks' sums of the masses (times the coefficients c, if any), an xor tree over the power of
// two that holds a block, pushed to all CTAs; the barrier that must follow makes csum readable.
template <int C>
__device__ __forceinline__ void fin_push_mass(FinShared<C>& sh, const FinSpan& sp, const float* coef) {
  constexpr int V = kFinBlocks / C;
  const int lg = min(sp.lg_cp, 5);                       // 1 << lg lanes of a block, 32 >> lg blocks of a warp
  const int lane = threadIdx.x & 31, slot = lane & ((1 << lg) - 1);
  const int v = static_cast<int>(threadIdx.x) >> lg;
  if ((v & ~((32 >> lg) - 1)) >= V) return;              // the warp's first block
  auto mass = [&](int x) {
    const int lm = v * sp.per + x;
    if (v >= V || x >= sp.per || lm >= sp.nm) return 0.0;
    return coef ? sh.tot[0][lm] * static_cast<double>(__ldcg(coef + sp.m0 + lm)) : sh.tot[0][lm];
  };
  double s = mass(slot);
  if (sp.lg_cp > 5) s += mass(slot + 32);
  for (int o = (1 << lg) >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if constexpr (V == 1) {                                // one block: a lane per CTA
    s = __shfl_sync(0xffffffffu, s, 0);
    if (lane < C) st_cluster(cluster_addr(&sh.csum[sp.b0], lane), s);
  } else {
    if (slot == 0 && v < V) fin_push<C>(&sh.csum[sp.b0 + v], s);
  }
}
template <int C>
__device__ __forceinline__ double fin_total(const FinShared<C>& sh) {
  static_assert(kFinBlocks == 8, "pairwise sum of eight");
  return ((sh.csum[0] + sh.csum[1]) + (sh.csum[2] + sh.csum[3])) +
         ((sh.csum[4] + sh.csum[5]) + (sh.csum[6] + sh.csum[7]));
}

// Ranks of this CTA's members: one warp per member counts the members that are deeper, or as
// deep with a lower index.
template <int C>
__device__ __forceinline__ void fin_ranks(const FinShared<C>& sh, const FinSpan& sp, int32_t* rank) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = warp; r < sp.nm; r += kFinWarps) {
    const int i = sp.m0 + r;
    const unsigned long long ki = sh.key[i];
    int n = 0;
    for (int j = lane; j < sp.N; j += 32) {
      const unsigned long long kj = sh.key[j];
      n += (kj > ki) || (kj == ki && j < i);
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) rank[i] = n;
  }
}

}  // namespace

// PID-mean, exact full PID and the weighted mean contour. Whole calls against a last CTA that
// formed the outputs in FP64: 64 x 512^2 fields PID-mean 45.5 -> 33.0 us, 128 x 2^20 exact full
// PID 215 -> 188 us, of which the finalisation was 15 to 18 us each time.
template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(kFinThreads, 2)
finalize_kernel(const __grid_constant__ FinParams p) {
  extern __shared__ float fin_dyn[];
  __shared__ FinShared<C> sh;
  if constexpr (C > 1) cluster_arrive(); // every CTA has started before its memory is written
  grid_dependency_wait();
  grid_launch_dependents();              // a second pass may start loading (it waits for this grid's end)
  const FinDesc& d = fin_desc(p, blockIdx.y);
  const int rank = static_cast<int>(blockIdx.x);
  const FinSpan sp = fin_span<C>(d.N, rank);
  const int N = sp.N, t = threadIdx.x;
  const int kind = d.kind;
  const bool wm = kind == FIN_WMEAN, second = kind == FIN_LIN2;
  fin_reduce<C>(sh, reinterpret_cast<Sum3*>(fin_dyn), d.part, d.n_chunks, sp, second);
  const int i = sp.m0 + t;
  const bool mine = t < sp.nm;
  double m = 0.0, A = 0.0;               // m_i, N A_i (against a weighted mean contour: A_i)
  if (mine) {
    m = second ? __ldcg(d.sums + i) : sh.tot[0][t];
    A = second ? __ldcg(d.sums + N + i) : sh.tot[1][t];
  }
  if constexpr (C > 1) cluster_wait();
  const bool need_mean = !second && (kind != FIN_LIN1 || d.mean_depth != nullptr);
  double msum = 0.0;
  if (need_mean) {
    fin_push_mass<C>(sh, sp, wm ? d.coef : nullptr);
    fin_sync<C>();
    if (mine) msum = fin_total<C>(sh);
  }
  double depth = 0.0;
  if (mine) {
    // The kernels sum A_i against the column sum N u_bar, so in_in = N A_i / (N m_i) (Eq. 17)
    // and, the mean contour's mass being (1/N) sum_j m_j, mean_out = N A_i / sum_j m_j (Eq. 16).
    const double in_in = m > 0.0 ? A / (wm ? m : m * N) : 0.0;
    double mean_out = 0.0;
    if (need_mean) {
      mean_out = msum > 0.0 ? A / msum : 0.0;
      if (d.mean_depth) d.mean_depth[i] = fmin(in_in, mean_out);
    }
    if (d.mass) d.mass[i] = m;
    if (kind == FIN_LIN1) {
      d.sums[i] = m;                     // the second pass's finalisation reads both
      d.sums[N + i] = A;
      d.coef[i] = m > 0.0 ? static_cast<float>(1.0 / (static_cast<double>(N) * m)) : 0.0f;
    } else {
      const double in_out = second ? sh.tot[1][t] : mean_out;
      depth = fmin(in_in, in_out);
      if (d.depth) d.depth[i] = depth;
      if (d.in_in) d.in_in[i] = in_in;
      if (d.in_out) d.in_out[i] = in_out;
    }
  }
  if (kind != FIN_LIN1 && d.rank != nullptr) {
    if (mine) fin_push<C>(&sh.key[i], order_key(depth));
    fin_sync<C>();
    fin_ranks<C>(sh, sp, d.rank);
  }
}

// ---------------------------------------------------------------------------------------
// Finalisation of the tensor-core Gram
// ---------------------------------------------------------------------------------------

namespace {

// acc + comp carries the running sum; comp holds the low-order part lost by acc (Kahan).
__device__ __forceinline__ void kahan_add(float& acc, float& comp, float v) {
  const float y = v - comp;
  const float t = acc + y;
  comp = (t - acc) - y;
  acc = t;
}

// Element `col` of the [n][NN] Gram partials summed over the chunks in order: compensated
// FP32, close to an FP64 sum at the FP32 rate. 16 values are loaded before they are added.
__device__ __forceinline__ float gram_chunk_sum(const float* src, int n, int64_t NN) {
  float acc = 0.f, comp = 0.f;
  int r = 0;
  for (; r + 16 <= n; r += 16) {
    float v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __ldcs(src + (r + k) * NN);
#pragma unroll
    for (int k = 0; k < 16; ++k) kahan_add(acc, comp, v[k]);
  }
  for (; r + 4 <= n; r += 4) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldcs(src + (r + k) * NN);
#pragma unroll
    for (int k = 0; k < 4; ++k) kahan_add(acc, comp, v[k]);
  }
  for (; r < n; ++r) kahan_add(acc, comp, __ldcs(src + r * NN));
  return acc;
}

constexpr int kGramSumThreads = 256;

__device__ __forceinline__ float* fin_gram(const FinDesc& d) { return reinterpret_cast<float*>(d.sums + 4 * d.N); }

// Dot products of this warp's rows r0, r0 + 16, ... (kFinRowsPerWarp of them) of the CTA's
// [nm][stride] block with the shared vector v: lane l takes the columns l, l + 32, ... in order,
// then a fixed xor tree.
__device__ __forceinline__ void rows_dot(const float* C, int stride, int r0, int nm, const float* v, int N,
                                         float (&acc)[kFinRowsPerWarp]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kFinRowsPerWarp; ++k) acc[k] = 0.f;
#pragma unroll 4
  for (int j = lane; j < N; j += 32) {
    const float vj = v[j];
#pragma unroll
    for (int k = 0; k < kFinRowsPerWarp; ++k) {
      const int r = r0 + k * kFinWarps;
      if (r < nm) acc[k] = fmaf(C[r * stride + j], vj, acc[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < kFinRowsPerWarp; ++k) acc[k] = warp_sum(acc[k]);
}

}  // namespace

// The sums of the Gram partials over the chunks, one thread per element (large ensembles).
// HBM / L2-bound: n_gchunks N^2 floats read once.
__global__ void __launch_bounds__(kGramSumThreads) gram_sum_kernel(const __grid_constant__ FinParams p) {
  grid_dependency_wait();
  grid_launch_dependents();
  const FinDesc& d = fin_desc(p, blockIdx.y);
  if (d.gram_inline) return;
  const int64_t NN = static_cast<int64_t>(d.N) * d.N;
  const int64_t col = static_cast<int64_t>(blockIdx.x) * kGramSumThreads + threadIdx.x;
  if (col < NN) fin_gram(d)[col] = gram_chunk_sum(d.gpart + col, d.n_gchunks, NN);
}

// The calibration of the tensor-core Gram, its depths and ranks.
//
// The Gram G' (stored G'[i + j N] ~ G_ij = sum_x w u_i u_j) carries each member's rounding
// bias in its row and column. Its row sums are known exactly from the same pass:
// sum_j G_ij = N A_i (the recall identity, Eq. 17). Calibrate by a symmetric diagonal scaling
// C_ij = d_i d_j (G'_ij + G'_ji) / 2 with d_i sum_j C... = N A_i (symmetric Sinkhorn
// iteration), then P_ij = C_ij / m_i, IN_in = mean_j P_ij (= A_i / m_i), IN_out = mean_j
// P_ji. err_est reports the uncalibrated |mean_j G'_ij / m_i - A_i / m_i|. The O(N^2) work runs
// in FP32 (the scales converge to FP32 precision, ~1e-7, far inside the Gram bound); the
// per-member scalars are FP64.
//
// Each CTA keeps its members' rows of the symmetrised Gram in shared memory (64 x 512 floats at
// N = 512; rows padded to an odd stride so that the transposed half writes without bank
// conflicts) and its warps dot them with the scales, which every sweep pushes to all CTAs.
// Small ensembles with few chunks take one CTA (fin_gram_single): a sweep then costs a CTA barrier
// instead of a cluster's (20 x 128^2 BF16 with P: 35.0 -> 30.9 us a call).
// 512 x 2^20 split BF16 with P: the whole call 2806 -> 2411 us against one CTA that did all of
// this (437 us); the plume step's three items 1076 -> 996 us (131 us).
template <int C, int PER_SM>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(kFinThreads, PER_SM)
finalize_gram_kernel(const __grid_constant__ FinParams p) {
  extern __shared__ float fin_dyn[];
  float* const fin_c0 = fin_dyn;                        // [nm][N | 1], where the column sums were before
  __shared__ FinShared<C> sh;
  __shared__ float sd[2][kFinMaxN], sdm[kFinMaxN];      // calibration scales; d_j / m_j
  __shared__ float starget[kFinMaxN / C], sraw[kFinMaxN / C];
  __shared__ int smoved[2][C];
  __shared__ double serr[C], swarp[kFinWarps];
  if constexpr (C > 1) cluster_arrive();
  grid_dependency_wait();
  grid_launch_dependents();
  const FinDesc& d = fin_desc(p, blockIdx.y);
  const int rank = static_cast<int>(blockIdx.x);
  const FinSpan sp = fin_span<C>(d.N, rank);
  const int N = sp.N, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int stride = N | 1;
  float* const G = fin_gram(d);
  if (d.gram_inline) {   // sum this CTA's rows of the stored array
    const int64_t NN = static_cast<int64_t>(N) * N;
    for (int e = t; e < sp.nm * N; e += kFinThreads) {
      const int64_t col = static_cast<int64_t>(sp.m0) * N + e;
      G[col] = gram_chunk_sum(d.gpart + col, d.n_gchunks, NN);
    }
  }
  fin_reduce<C>(sh, reinterpret_cast<Sum3*>(fin_dyn), d.part, d.n_chunks, sp, false);
  const int i = sp.m0 + t;
  const bool mine = t < sp.nm;
  const double m = mine ? sh.tot[0][t] : 0.0, A = mine ? sh.tot[1][t] : 0.0;   // m_i, N A_i
  if constexpr (C > 1) cluster_wait();
  fin_push_mass<C>(sh, sp, nullptr);
  fin_sync<C>();       // the other CTAs' shares of the mass; their rows of G (inline sums)

  // Row r of the stored array is G'_{., r}, which equals row r of G' up to the rounding of the
  // tensor-core sums: its raw sum, and one half of C0.
  for (int r = warp; r < sp.nm; r += kFinWarps) {
    const float* row = G + static_cast<int64_t>(sp.m0 + r) * N;
    float acc = 0.f;
    for (int b = 0; b < N; b += 256) {
      float x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int j = b + lane + 32 * k;
        x[k] = j < N ? __ldcg(row + j) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int j = b + lane + 32 * k;
        if (j < N) {
          acc += x[k];
          fin_c0[r * stride + j] = x[k];
        }
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) sraw[r] = acc;
  }
  __syncthreads();
  {   // ... plus the other half, read across the rows of the other members
    const int lg = sp.nm > 0 ? ceil_log2(sp.nm) : 0;   // threads across this CTA's members
    const int rr = t & ((1 << lg) - 1), c0 = t >> lg, step = kFinThreads >> lg;
    if (rr < sp.nm) {
      const float* src = G + sp.m0 + rr;
      for (int c = c0; c < N; c += 8 * step) {
        float x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int cc = c + k * step;
          x[k] = cc < N ? __ldcg(src + static_cast<int64_t>(cc) * N) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int cc = c + k * step;
          if (cc < N) fin_c0[rr * stride + cc] = 0.5f * (x[k] + fin_c0[rr * stride + cc]);
        }
      }
    }
  }
  double in_in = 0.0, err = 0.0;
  if (mine) {
    const double msum = fin_total<C>(sh);
    const double nm_i = m * N;
    in_in = m > 0.0 ? A / nm_i : 0.0;
    if (d.mean_depth) d.mean_depth[i] = fmin(in_in, msum > 0.0 ? A / msum : 0.0);
    if (d.mass) d.mass[i] = m;
    const double raw = sraw[t];
    if (d.err_est) err = m > 0.0 ? fabs(raw / nm_i - in_in) : 0.0;
    starget[t] = static_cast<float>(A);                 // row-sum target N A_i
    const float s0 = (A > 0.0 && raw > 0.0) ? 1.0f : 0.0f;
    fin_push<C>(&sd[0][i], s0);
  }
  fin_sync<C>();
  const int groups = C == kFinBlocks ? 1 : (sp.nm + kFinMaxRows - 1) / kFinMaxRows;   // of rows_dot
  // Symmetric Sinkhorn: d_r <- sqrt(d_r N A_r / sum_j C0_rj d_j), until no scale moves by more
  // than 2^-22 relative (at most 24 sweeps).
  int cur = 0;
  for (int it = 0; it < 24; ++it) {
    bool moved = false;
    for (int g = 0, r0 = warp; g < groups; ++g, r0 += kFinMaxRows) {
      float acc[kFinRowsPerWarp];
      rows_dot(fin_c0, stride, r0, sp.nm, sd[cur], N, acc);
#pragma unroll
      for (int k = 0; k < kFinRowsPerWarp; ++k) {
        const int r = r0 + k * kFinWarps;
        if (r < sp.nm) {
          const float so = sd[cur][sp.m0 + r];
          const float sn = (so > 0.f && acc[k] > 0.f) ? sqrtf(so * starget[r] / acc[k]) : 0.f;
          moved = moved || fabsf(sn - so) > 2.4e-7f * so;
          if constexpr (C == 1) {
            if (lane == 0) sd[cur ^ 1][sp.m0 + r] = sn;
          } else {
            if (lane < C) st_cluster(cluster_addr(&sd[cur ^ 1][sp.m0 + r], lane), sn);
          }
        }
      }
    }
    int more = __syncthreads_or(moved);
    if constexpr (C > 1) {
      if (t < C) st_cluster(cluster_addr(&smoved[cur][rank], t), more);
      cluster_sync_all();
      more = 0;
#pragma unroll
      for (int r = 0; r < C; ++r) more |= smoved[cur][r];
    }
    cur ^= 1;
    if (!more) break;
  }
  // IN_out(i) = (1/N) sum_j C_ji / m_j = (d_i / N) sum_j (d_j / m_j) C0_ij (C0 symmetric).
  double inv_m = 0.0;
  if (mine) {
    const float dm = m > 0.0 ? static_cast<float>(static_cast<double>(sd[cur][i]) / m) : 0.f;
    fin_push<C>(&sdm[i], dm);
    if (d.P) inv_m = m > 0.0 ? 1.0 / m : 0.0;
  }
  fin_sync<C>();
  for (int g = 0, r0 = warp; g < groups; ++g, r0 += kFinMaxRows) {
    float acc[kFinRowsPerWarp];
    rows_dot(fin_c0, stride, r0, sp.nm, sdm, N, acc);
#pragma unroll
    for (int k = 0; k < kFinRowsPerWarp; ++k) {
      const int r = r0 + k * kFinWarps;
      if (r < sp.nm && lane == 0) sraw[r] = sd[cur][sp.m0 + r] * acc[k];
    }
  }
  __syncthreads();
  double depth = 0.0;
  if (mine) {
    const double in_out = static_cast<double>(sraw[t]) / N;
    depth = fmin(in_in, in_out);
    if (d.depth) d.depth[i] = depth;
    if (d.in_in) d.in_in[i] = in_in;
    if (d.in_out) d.in_out[i] = in_out;
    if (d.rank) fin_push<C>(&sh.key[i], order_key(depth));
    if (d.P) sh.tot[0][t] = inv_m;       // 1 / m_i: m is in the owner's registers by now
  }
  if (d.err_est) {
    constexpr int W = kFinMaxN / C / 32;   // warps that can hold members
    if (warp < W) {
      if (warp * 32 < sp.nm) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) err = fmax(err, __shfl_xor_sync(0xffffffffu, err, o));
      }
      if (lane == 0) swarp[warp] = err;
    }
    __syncthreads();
    if (warp == 0) {
      double e = swarp[lane & (W - 1)];
#pragma unroll
      for (int o = W / 2; o > 0; o >>= 1) e = fmax(e, __shfl_xor_sync(0xffffffffu, e, o));
      if (lane == 0) {
        if constexpr (C == 1) serr[0] = e;
        else st_cluster(cluster_addr(&serr[rank], 0), e);
      }
    }
  }
  fin_sync<C>();
  if (d.err_est && rank == 0 && t == 0) {
    double e = serr[0];
#pragma unroll
    for (int r = 1; r < C; ++r) e = fmax(e, serr[r]);
    d.err_est[0] = e;
  }
  if (d.rank) fin_ranks<C>(sh, sp, d.rank);
  if (d.P) {
    // P[r][c] = C_rc / m_r. Small ensembles: written here; else C (FP32) and 1 / m_r are
    // stored for gram_matrix_kernel.
    const bool here = N <= kFinInlineMatrixN;
    float* const C0 = G + static_cast<int64_t>(N) * N;
    for (int r = warp; r < sp.nm; r += kFinWarps) {
      const float sr = sd[cur][sp.m0 + r];
      const double inv = sh.tot[0][r];
      const int64_t row = static_cast<int64_t>(sp.m0 + r) * N;
      for (int c = lane; c < N; c += 32) {
        const float v = sr * sd[cur][c] * fin_c0[r * stride + c];
        if (here) d.P[row + c] = static_cast<double>(v) * inv;
        else C0[row + c] = v;
      }
    }
    if (!here && mine) d.sums[i] = inv_m;
  }
}

// P = C / m per row, over the whole GPU: its N^2 FP64 conversions and products take 17 us on one
// cluster at N = 512.
__global__ void __launch_bounds__(256) gram_matrix_kernel(const __grid_constant__ FinParams p) {
  grid_dependency_wait();
  const FinDesc& d = fin_desc(p, blockIdx.y);
  const int N = d.N;
  if (d.P == nullptr || N <= kFinInlineMatrixN) return;
  const float* C = fin_gram(d) + static_cast<int64_t>(N) * N;
  const int NN = N * N;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < NN; e += gridDim.x * 256)
    d.P[e] = static_cast<double>(__ldcg(C + e)) * __ldcg(d.sums + e / N);
}

namespace {

constexpr int kFinMaxDynamic = 200 * 1024;   // besides at most 23 KB of static shared memory
constexpr int kFinAlone = 112 * 1024;        // so that no second CTA fits it
constexpr int kFinTwoDynamic = 88 * 1024;    // so that two CTAs fit an SM

// Dynamic shared memory of the Gram's finalisation: its rows, or the column sums before them.
template <int C>
constexpr size_t fin_gram_smem(int N) {
  const size_t rows = static_cast<size_t>((N + kFinBlocks - 1) / kFinBlocks) * (kFinBlocks / C);
  const size_t bytes = rows * (N | 1) * sizeof(float);
  return bytes > fin_acc_bytes<C>(N) ? bytes : fin_acc_bytes<C>(N);
}

template <int C>
cudaError_t fin_init() {
  cudaError_t e = cudaFuncSetAttribute(finalize_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinAlone);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(finalize_gram_kernel<C, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinMaxDynamic);
  if constexpr (C < kFinBlocks) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(finalize_gram_kernel<C, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinTwoDynamic);
  }
  return e;
}

}  // namespace

cudaError_t finalize_kernels_init() {
  cudaError_t e = fin_init<1>();
  if (e == cudaSuccess) e = fin_init<2>();
  if (e == cudaSuccess) e = fin_init<4>();
  if (e == cudaSuccess) e = fin_init<8>();
  return e;
}

namespace {

template <typename K>
cudaError_t fin_launch(K kernel, dim3 grid, int threads, size_t smem, bool pdl, const FinParams& p,
                       cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

// The launch with C CTAs per ensemble if `force`, or if all of them are on the GPU at once; sets `done`
// if it was made. Ensembles that fill less than the SMs get one each: two on an SM are slower than
// one (the Gram is compiled for either, with 80 and 64 registers: 50 x (32 x 4096) 53.6 and 49.5 us).
template <int C>
cudaError_t fin_try(const FinParams& p, const FinLaunch& l, int sms, bool pdl, bool force, bool* done, cudaStream_t s) {
  if (*done) return cudaSuccess;
  const int64_t ctas = static_cast<int64_t>(l.count) * C;
  const dim3 grid(C, static_cast<unsigned>(l.count));
  if (!l.gram) {
    if (!force && ctas > 2 * sms) return cudaSuccess;
    *done = true;
    // Few ensembles: shared memory for one CTA per SM, or the scheduler packs a cluster's CTAs two to
    // an SM (10 x (300 x 5000) exact full PID 106.5 -> 102 us). Clusters of eight fill three quarters of
    // the SMs before the rest lie scattered over the GPCs.
    const size_t acc = 4 * ctas <= 3 * sms ? size_t(kFinAlone) : fin_acc_bytes<C>(l.max_n);
    return fin_launch(finalize_kernel<C>, grid, kFinThreads, acc, pdl, p, s);
  }
  const size_t smem = fin_gram_smem<C>(l.max_n);
  if (smem > kFinMaxDynamic) return cudaSuccess;
  if constexpr (C < kFinBlocks) {
    const bool two = smem <= kFinTwoDynamic;
    if (ctas > sms && two && (force || ctas <= 2 * sms)) {
      *done = true;
      return fin_launch(finalize_gram_kernel<C, 2>, grid, kFinThreads, smem, pdl, p, s);
    }
  }
  if (!force && ctas > sms) return cudaSuccess;
  *done = true;
  return fin_launch(finalize_gram_kernel<C, 1>, grid, kFinThreads, smem, pdl, p, s);
}

// CTAs per ensemble: the most that let every ensemble start at once. An ensemble's chain of barriers
// and round trips gets shorter with more CTAs, but a second wave of ensembles waits for all of the
// first one's. More ensembles than that take one CTA each; two or four if some have more than 128 or 256
// members, for which all the others would wait (200 x (20 x 4096) with 3 x (512 x 20 000) PID-mean, 203
// ensembles: 145 us with one CTA each, 124 with four), or the fewest that hold the Gram's rows.
// Batches, eight CTAs each -> this rule: PID-mean of 1000 x (8 x 1024) 198 -> 51 us, of 200 x
// (20 x 16 384) 149 -> 123; BF16 Gram of 200 x (64 x 4096) 369 -> 123, of 50 x (200 x 8192) 321 -> 264.
cudaError_t fin_launch_ctas(const FinParams& p, const FinLaunch& l, int sms, bool pdl, cudaStream_t s) {
  bool done = false;
  cudaError_t e = cudaSuccess;
  if (!(l.gram && l.single)) {
    e = fin_try<8>(p, l, sms, pdl, false, &done, s);
    if (e == cudaSuccess) e = fin_try<4>(p, l, sms, pdl, false, &done, s);
    if (e == cudaSuccess) e = fin_try<2>(p, l, sms, pdl, false, &done, s);
  }
  if (e == cudaSuccess && (l.gram || l.max_n <= 128)) e = fin_try<1>(p, l, sms, pdl, true, &done, s);
  if (e == cudaSuccess && (l.gram || l.max_n <= 256)) e = fin_try<2>(p, l, sms, pdl, true, &done, s);
  if (e == cudaSuccess) e = fin_try<4>(p, l, sms, pdl, true, &done, s);
  if (e == cudaSuccess) e = fin_try<8>(p, l, sms, pdl, true, &done, s);
  return e;
}

}  // namespace

cudaError_t launch_finalize(const FinParams& p, const FinLaunch& l, int sms, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  bool pdl = l.pdl;
  const unsigned count = static_cast<unsigned>(l.count);
  const unsigned NN = static_cast<unsigned>(l.max_n) * static_cast<unsigned>(l.max_n);
  if (l.sum_gram) {
    e = fin_launch(gram_sum_kernel, dim3((NN + kGramSumThreads - 1) / kGramSumThreads, count),
                   kGramSumThreads, 0, pdl, p, s);
    if (e != cudaSuccess) return e;
    pdl = true;
  }
  e = fin_launch_ctas(p, l, sms, pdl, s);
  if (e != cudaSuccess || !l.matrix) return e;
  return fin_launch(gram_matrix_kernel, dim3((NN + 1023) / 1024, count), 256, 0, true, p, s);
}

}  // namespace pidk
