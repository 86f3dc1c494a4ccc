// Full PID on the tensor cores for 256 < N <= 512 members, in one pass over the data: the Gram
// G = U' U'^T of the weighted soft masks U' = U diag(sqrt w) (Eq. 9, sums of Eq. 14).
//
// One CTA's tensor memory holds 128 x 512 FP32 sums, a quarter of this Gram, so a cluster of one
// CTA per 128-member row block (3 or 4) takes a chunk of cells together:
//   * 16 warps of CTA r read the FP32 values of row block r from HBM (prefetched into registers one
//     stage ahead), map and weight them, and write them as tensor-core operands into the CTA's
//     shared memory (K-major, 128-byte swizzle; BF16, a BF16 hi + lo pair, or E4M3);
//   * the courier thread copies the finished block into the shared memory of the CTAs that multiply
//     by it (shared memory to shared memory, counted on the receiver's mbarrier), so no operand
//     ever goes to HBM and each value is converted once;
//   * the issuer thread multiplies row block r by the column blocks r, r + 1 (and r + 2 for the
//     first half of four), modulo the block count: every pair of blocks once. Its commit frees the
//     stage in this CTA and in the CTAs whose blocks it used.
// The finalisation symmetrises, so each off-diagonal block is written with its mirror image.
//
// Chunks and the order of their products are those of the tiled kernel (gram_tiled.cu), and so are
// the results' bits. The clusters share the chunks' stages evenly all the same: a chunk that falls
// into two clusters' shares is begun by the one at its start, which leaves the accumulators in the
// chunk's partial Gram and raises a flag, and completed by the other at its end.
//
// What bounds it: at 512 members the chain from a stage's conversion over the copy and the products
// to its release (4.3 us; the ring holds two split stages), not HBM (2.0 TB/s) or the tensor pipe
// (1.2 us of a stage's 2.1); BF16 and E4M3 the row segments of 256 and 512 bytes that are in flight
// (3.4 TB/s). Per call against a pass that staged the operands in HBM and a tiled product over them,
// with the same bits: 512 x 1 048 576 split BF16 2335 -> 1545 us (staging 676 and product 1084 before,
// 1006 now), E4M3 1842 -> 1474, BF16 1462 -> 1115; 384 members split BF16 1435 -> 1033.
//
// A stage is one 128-byte K-block (64 cells, or 128 of E4M3). Every wait is bounded; after a wait
// that ran out a thread stops, the others run out in turn, and all meet at the closing cluster
// barrier before shared or tensor memory is given up.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"
#include "stream_kernel.cuh"

namespace pidk {

namespace {

constexpr int kClConv = 16;                          // converter warps: 8 rows each
constexpr int kClRows = 128 / kClConv;
constexpr int kClThreads = (kClConv + 2) * 32;       // and the issuer's and the courier's warp
constexpr uint32_t kClBlock = 128 * 128;             // one K-block of one row block and plane
constexpr int kClRing = 192 * 1024;                  // bytes of operand stages
constexpr int kClMaxStages = 6;

struct ClBars {
  uint64_t opW[kClMaxStages];      // own block written (one arrival per converter warp)
  uint64_t opE[kClMaxStages];      // stage consumed: here and by the CTAs that use this block
  uint64_t rx[kClMaxStages];       // the other CTAs' blocks have landed
  uint64_t accF, accE, fin;        // accumulator ready, drained; all tensor-core work done
  uint32_t tmem;
};

// shared::cta -> shared::cluster copy (16-byte aligned), counted on the receiver's mbarrier.
__device__ __forceinline__ void bulk_to_cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// A whole warp's bounded wait: the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, kWaitTimeoutNs)) != 0;
}
// The stages of cell chunk c that a cluster works through at one go.
struct ClSegment {
  int c, st0, st1;
  bool resumed, final;             // continues another cluster's accumulators; completes the chunk
};
// What cluster g of G does, in order. Shares [W g / G, W (g + 1) / G) of the W stages when there
// are more chunks than clusters (so a share is no shorter than a chunk): its last chunk's
// beginning, its whole chunks, then the rest of its first chunk. Else chunk g.
struct ClShare {
  int nst, n_chunks, last_st, lo, hi;
  bool split;
  __device__ ClShare(const ClusterGramParams& p, int kb, int g, int G) {
    nst = p.chunk_cells / kb;
    n_chunks = p.n_chunks;
    last_st = (p.M - (n_chunks - 1) * p.chunk_cells + kb - 1) / kb;
    const int64_t W = static_cast<int64_t>(n_chunks - 1) * nst + last_st;
    split = n_chunks > G;
    lo = split ? static_cast<int>(W * g / G) : g * nst;
    hi = split ? static_cast<int>(W * (g + 1) / G) : (g + 1 < n_chunks ? (g + 1) * nst : static_cast<int>(W));
  }
  __device__ int stages(int c) const { return c + 1 < n_chunks ? nst : last_st; }
  __device__ bool at(int s, ClSegment* seg) const {
    const bool end = hi == (n_chunks - 1) * nst + last_st;      // the share ends with the last chunk
    const int c_lo = lo / nst, o_lo = lo - c_lo * nst;
    const int c_hi = end ? n_chunks : hi / nst, o_hi = end ? 0 : hi - c_hi * nst;
    if (o_hi > 0) {
      if (s == 0) { *seg = ClSegment{c_hi, 0, o_hi, false, false}; return true; }
      --s;
    }
    const int first = c_lo + (o_lo > 0 ? 1 : 0);
    if (s < c_hi - first) { *seg = ClSegment{first + s, 0, stages(first + s), false, true}; return true; }
    if (s > c_hi - first || o_lo == 0) return false;
    *seg = ClSegment{c_lo, o_lo, stages(c_lo), true, true};
    return true;
  }
};

// Before the Gram: the flags cleared, and sqrt(w) once per cell instead of once per cell and
// converter warp (zero up to a whole stage past the last cell).
__global__ void __launch_bounds__(256) gram_cluster_prep_kernel(const float* w, int M, float* sqrt_w, unsigned int* flags,
                                                                int n_flags) {
  const int x = blockIdx.x * 256 + threadIdx.x;
  if (x < n_flags) flags[x] = 0u;
  if (w != nullptr && x < ((M + 127) & ~127)) sqrt_w[x] = x < M ? sqrtf(__ldg(w + x)) : 0.f;
}

// 32 consecutive FP32 columns of this warp's 32 TMEM lanes, stored (see tmem_ld32).
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]),
      "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]),
      "f"(v[16]), "f"(v[17]), "f"(v[18]), "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]),
      "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]), "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// Wait (bounded) until the counter has reached n.
__device__ __forceinline__ bool flag_wait(const unsigned int* flag, unsigned int n) {
  const uint64_t t0 = global_timer_ns();
  while (true) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= n) return true;
    if (global_timer_ns() - t0 > kWaitTimeoutNs) return false;
    __nanosleep(100);
  }
}
// tc_commit whose arrival goes to the barrier at this offset in every CTA of the mask.
__device__ __forceinline__ void tc_commit_mask(uint64_t* bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"(mask) : "memory");
}

}  // namespace

template <int PREC, int ISO>
__global__ void __launch_bounds__(kClThreads, 1) gram_cluster_kernel(const __grid_constant__ ClusterGramParams p) {
  constexpr int PLANES = PREC == 2 ? 2 : 1;
  constexpr uint32_t FMT = PREC == 3 ? 0u : 1u;      // E4M3 : BF16
  constexpr int KB = PREC == 3 ? 128 : 64;           // cells per stage
  constexpr int RPL = PREC == 3 ? 1 : 2;             // rows per load: KB / 4 lanes each
  constexpr int LOADS = kClRows / RPL;
  constexpr int DEPTH = PREC == 3 ? 1 : 2;           // stages whose loads are in flight
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ ClBars bars;
  unsigned char* const ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int R = p.R;                                 // row blocks = CTAs of the cluster
  const int r = static_cast<int>(blockIdx.x) % R;
  const int cluster = static_cast<int>(blockIdx.x) / R, n_clusters = static_cast<int>(gridDim.x) / R;
  const uint32_t PLANE = static_cast<uint32_t>(R == 4 ? 3 : 2) * kClBlock;
  const uint32_t STAGE = PLANES * PLANE;
  const int S = p.stages;
  const int N = p.N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // This CTA multiplies by the blocks of r (slot 0), r + 1 (slot 1) and, r < 2 of 4, r + 2 (slot 2).
  const bool two = R == 4 && r < 2;                  // receives two blocks
  const int next1 = (r + 1) % R, next2 = (r + 2) % R;
  // Bytes of a block's plane that are sent: rows past N stay what they were in the receiver (they
  // reach accumulator columns that are never read).
  auto block_bytes = [&](int b) { return static_cast<uint32_t>(min(128, (N - 128 * b + 7) & ~7)) * 128u; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&bars.opW[s], kClConv);
      mbar_init(&bars.opE[s], 1u + (R == 4 && r >= 2 ? 2u : 1u));
      mbar_init(&bars.rx[s], 1);
    }
    mbar_init(&bars.accF, 1);
    mbar_init(&bars.accE, kClConv);
    mbar_init(&bars.fin, 1);
    fence_mbar_init();
  }
  // rows past N of a received block are multiplied too: finite from the start
  for (uint32_t o = threadIdx.x * 16; o < static_cast<uint32_t>(S) * STAGE; o += kClThreads * 16)
    *reinterpret_cast<uint4*>(ring + o) = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  if (warp == 0) {
    tmem_alloc(&bars.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  cluster_sync_all();                                // every CTA's barriers are ready
  tc_fence_after();
  grid_launch_dependents();
  const uint32_t tmem = bars.tmem;
  bool ok = true;
  int k = 0, slot = 0;                               // stages so far; ring slot (k mod S) and
  uint32_t par = 0;                                  // parity (k / S) of the next one
  auto advance = [&]() {
    ++k;
    if (++slot == S) { slot = 0; par ^= 1u; }
  };
  const ClShare share(p, KB, cluster, n_clusters);

  if (warp < kClConv) {
    // ---- converters: warp q owns rows 8 q .. 8 q + 7 of the block; a load takes 16 bytes per lane
    // of RPL rows ----
    const int q = warp;
    const int sub = lane / (32 / RPL);               // row of a load
    const int xl = (lane % (32 / RPL)) * 4;          // first of this lane's four cells
    const int row0 = 128 * r + 8 * q + sub;
    float sc[PREC == 3 ? LOADS : 1];
    if constexpr (PREC == 3) {
#pragma unroll
      for (int m = 0; m < LOADS; ++m)
        sc[m] = p.op_scale == nullptr ? 256.f : (row0 + m < N ? p.op_scale[row0 + m] : 1.f);
    }
    const float* const base = p.F + static_cast<int64_t>(row0) * p.ld + xl;
    const int64_t hop = RPL * p.ld;
    const int rows_in = N - row0;                    // load m is this lane's if m RPL < rows_in
    // The values of a stage, in flight until it is their turn (DEPTH stages ahead: with one the
    // loads' latency shows).
    struct Values { float x[LOADS][4]; float4 w; };
    auto load = [&](Values& s, int x0) {             // the stage that starts at cell x0
      const float* src = base + x0;
      if (p.vec_ok && x0 + KB <= p.M) {
#pragma unroll
        for (int m = 0; m < LOADS; ++m) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
          if (m * RPL < rows_in) t = __ldcs(reinterpret_cast<const float4*>(src + m * hop));
          s.x[m][0] = t.x; s.x[m][1] = t.y; s.x[m][2] = t.z; s.x[m][3] = t.w;
        }
      } else {
#pragma unroll
        for (int m = 0; m < LOADS; ++m)
#pragma unroll
          for (int v = 0; v < 4; ++v)
            s.x[m][v] = m * RPL < rows_in && x0 + xl + v < p.M ? __ldg(src + m * hop + v) : 0.f;
      }
      if (p.sqrt_w != nullptr) s.w = __ldg(reinterpret_cast<const float4*>(p.sqrt_w + x0 + xl));
    };
    // byte offset of this lane's operands of load m in the block: row 8 q + m RPL + sub, 16-byte
    // chunk c of it at c ^ (row mod 8)
    const int byte = PREC == 3 ? xl : 2 * xl;
    auto off = [&](int m) {
      const int row = m * RPL + sub;
      return static_cast<uint32_t>(q * 1024 + row * 128 + (((byte >> 4) ^ row) << 4) + (byte & 15));
    };
    // this warp's part of the accumulator: rows 32 (q & 3) .. + 31, columns 32 (q >> 2) .. + 31 of
    // every block; block b's first column there is member cols(b)
    const int i = 128 * r + 32 * (q & 3) + lane;
    const int nb = two ? 3 : 2;
    auto cols = [&](int b) { return 128 * (b == 0 ? r : (b == 1 ? next1 : next2)) + 32 * (q >> 2); };
    const uint32_t tpart = tmem + (static_cast<uint32_t>(32 * (q & 3)) << 16) + static_cast<uint32_t>(32 * (q >> 2));
    const bool vec_row = (N & 3) == 0 && (reinterpret_cast<uintptr_t>(p.gpart) & 15) == 0;
    ClSegment sg;
    for (int t = 0; ok && share.at(t, &sg); ++t) {
      const int cell0 = sg.c * p.chunk_cells;
      float* const gp = p.gpart + static_cast<size_t>(sg.c) * N * N;
      Values values[DEPTH];
#pragma unroll
      for (int d = 0; d < DEPTH; ++d) load(values[d], cell0 + min(sg.st0 + d, sg.st1 - 1) * KB);
      // ---- the accumulator is free; another cluster's sums go back into it ----
      if (sg.resumed) {
        if (!__all_sync(0xffffffffu, flag_wait(p.flags + (cluster - 1) * R + r, kClConv))) { ok = false; break; }
        for (int b = 0; b < nb; ++b) {
          const int jb = cols(b);
          float v[32];
#pragma unroll
          for (int jj = 0; jj < 32; ++jj)
            v[jj] = i < N && jb + jj < N ? __ldcg(gp + static_cast<size_t>(jb + jj) * N + i) : 0.f;
          tmem_st32(tpart + static_cast<uint32_t>(128 * b), v);
        }
        tc_fence_before();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.accE);
      // One stage: its values to operands, the loads of the stage DEPTH further on, and the operands
      // into their slot once that is free.
      auto step = [&](Values& s, int st) {
        const int x0 = cell0 + st * KB;
        if constexpr (ISO != ISOK_NONE) {
          iso_map_tile<ISO>(s.x, p.iso_mu, p.iso_inv, p.iso_t, iso_pad_sign(p.iso_mode), p.iso_mode);
#pragma unroll
          for (int m = 0; m < LOADS; ++m)            // rows past N and cells past M map to anything
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (m * RPL >= rows_in || x0 + xl + v >= p.M) s.x[m][v] = 0.f;
        }
        uint32_t h[LOADS][2], l[PREC == 2 ? LOADS : 1][2];   // operands: pairs of cells (E4M3: all four)
#pragma unroll
        for (int m = 0; m < LOADS; ++m) {
          float2 t = make_float2(s.x[m][0], s.x[m][1]), u = make_float2(s.x[m][2], s.x[m][3]);
          if (p.sqrt_w != nullptr) {
            t = f2_mul(t, make_float2(s.w.x, s.w.y));
            u = f2_mul(u, make_float2(s.w.z, s.w.w));
          }
          if constexpr (PREC == 3) {
            const uint32_t a = __nv_cvt_float2_to_fp8x2(f2_mul(t, f2(sc[m])), __NV_SATFINITE, __NV_E4M3);
            const uint32_t b = __nv_cvt_float2_to_fp8x2(f2_mul(u, f2(sc[m])), __NV_SATFINITE, __NV_E4M3);
            h[m][0] = (a & 0xffffu) | (b << 16);
          } else {
            const __nv_bfloat162 ha = __floats2bfloat162_rn(t.x, t.y), hb = __floats2bfloat162_rn(u.x, u.y);
            h[m][0] = *reinterpret_cast<const uint32_t*>(&ha);
            h[m][1] = *reinterpret_cast<const uint32_t*>(&hb);
            if constexpr (PREC == 2) {
              const float2 fa = __bfloat1622float2(ha), fb = __bfloat1622float2(hb);
              const __nv_bfloat162 la = __floats2bfloat162_rn(t.x - fa.x, t.y - fa.y);
              const __nv_bfloat162 lb = __floats2bfloat162_rn(u.x - fb.x, u.y - fb.y);
              l[m][0] = *reinterpret_cast<const uint32_t*>(&la);
              l[m][1] = *reinterpret_cast<const uint32_t*>(&lb);
            }
          }
        }
        if (st + DEPTH < sg.st1) load(s, x0 + DEPTH * KB);
        if (k >= S && !warp_wait(&bars.opE[slot], par ^ 1u)) {
          ok = false;
          return;
        }
        unsigned char* dst = ring + static_cast<uint32_t>(slot) * STAGE;
#pragma unroll
        for (int m = 0; m < LOADS; ++m) {
          if constexpr (PREC == 3) {
            *reinterpret_cast<uint32_t*>(dst + off(m)) = h[m][0];
          } else {
            *reinterpret_cast<uint2*>(dst + off(m)) = make_uint2(h[m][0], h[m][1]);
            if constexpr (PREC == 2) *reinterpret_cast<uint2*>(dst + PLANE + off(m)) = make_uint2(l[m][0], l[m][1]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars.opW[slot]);
        advance();
      };
      for (int st = sg.st0; ok && st < sg.st1; st += DEPTH) {
#pragma unroll
        for (int d = 0; d < DEPTH; ++d)
          if (ok && st + d < sg.st1) step(values[d], st + d);
      }
      // ---- drain: the chunk's partial Gram, or the sums so far in its place ----
      if (!ok || !warp_wait(&bars.accF, static_cast<uint32_t>(t & 1))) { ok = false; break; }
      tc_fence_after();
      const float* inv = PREC == 3 && p.op_scale ? p.op_scale + N : nullptr;
      const float ir = PREC != 3 ? 1.f : (inv ? inv[min(i, N - 1)] : 1.f / 65536.f);
      for (int b = 0; b < nb; ++b) {
        const int jb = cols(b);
        if (jb >= N) continue;                       // the same for the whole warp
        float v[32];
        tmem_ld32(tpart + static_cast<uint32_t>(128 * b), v);
        if (i < N) {
          if (PREC == 3 && sg.final) {
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) v[jj] *= inv ? ir * inv[min(jb + jj, N - 1)] : ir;
          }
#pragma unroll
          for (int jj = 0; jj < 32; ++jj)
            if (jb + jj < N) gp[static_cast<size_t>(jb + jj) * N + i] = v[jj];
          if (sg.final && b > 0) {                   // the mirror image
            float* row = gp + static_cast<size_t>(i) * N + jb;
#pragma unroll
            for (int jj = 0; jj < 32; jj += 4) {
              if (vec_row && jb + jj + 3 < N) {
                *reinterpret_cast<float4*>(row + jj) = make_float4(v[jj], v[jj + 1], v[jj + 2], v[jj + 3]);
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (jb + jj + e < N) row[jj + e] = v[jj + e];
              }
            }
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      if (!sg.final) {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(p.flags + cluster * R + r, 1u);
      }
    }
  } else if (warp == kClConv && lane == 0) {
    // ---- issuer ----
    const uint32_t id256 = umma_idesc(FMT, 128, 256), id128 = umma_idesc(FMT, 128, 128);
    const uint32_t rx_bytes = PLANES * (block_bytes(next1) + (two ? block_bytes(next2) : 0u));
    const uint16_t mask = static_cast<uint16_t>((1u << r) | (1u << next1) | (two ? 1u << next2 : 0u));
    ClSegment sg;
    for (int t = 0; ok && share.at(t, &sg); ++t) {
      for (int st = sg.st0; st < sg.st1; ++st, advance()) {
        mbar_arrive_expect_tx(&bars.rx[slot], rx_bytes);
        if (!mbar_wait_bounded(&bars.opW[slot], par, kWaitTimeoutNs) ||
            (st == sg.st0 && !mbar_wait_bounded(&bars.accE, static_cast<uint32_t>(t & 1), kWaitTimeoutNs))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t a0 = umma_desc_sw128(smem_u32(ring) + static_cast<uint32_t>(slot) * STAGE);
        const uint64_t lo = PLANE >> 4;              // hi plane -> lo plane (descriptor units)
        // columns from n0 on; below: a block below the diagonal, whose two cross terms are added in
        // the order of its transpose
        auto product = [&](int n0, uint32_t id, bool below) {
          const uint32_t d = tmem + static_cast<uint32_t>(n0);
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {           // 4 x 32 bytes along K in the 128-byte row
            const uint64_t a = a0 + static_cast<uint64_t>((ks * 32) >> 4);
            const uint64_t b = a + static_cast<uint64_t>((n0 * 128) >> 4);
            const uint32_t acc = (st == sg.st0 && ks == 0 && !sg.resumed) ? 0u : 1u;
            if constexpr (PREC == 3) {
              umma_f8(d, a, b, id, acc);
            } else {
              umma_f16(d, a, b, id, acc);
              if constexpr (PREC == 2) {
                umma_f16(d, below ? a + lo : a, below ? b : b + lo, id, 1u);
                umma_f16(d, below ? a : a + lo, below ? b + lo : b, id, 1u);
              }
            }
          }
        };
        product(0, id128, false);                    // its own block, while the others arrive
        if (!mbar_wait_bounded(&bars.rx[slot], par, kWaitTimeoutNs)) {
          ok = false;
          break;
        }
        tc_fence_after();
        product(128, two ? id256 : id128, next1 < r);
        tc_commit_mask(&bars.opE[slot], mask);
        if (st == sg.st1 - 1) tc_commit(&bars.accF);
      }
    }
    tc_commit(&bars.fin);
    if (!mbar_wait_bounded(&bars.fin, 0u, kWaitTimeoutNs)) ok = false;
  } else if (warp == kClConv + 1 && lane == 0) {
    // ---- courier: block r to CTA r - 1 (its slot 1) and, r >= 2 of 4, to CTA r - 2 (slot 2) ----
    const uint32_t bytes = block_bytes(r);
    const uint32_t d1 = static_cast<uint32_t>((r + R - 1) % R), d2 = static_cast<uint32_t>((r + R - 2) % R);
    ClSegment sg;
    for (int t = 0; ok && share.at(t, &sg); ++t) {
      for (int st = sg.st0; st < sg.st1; ++st, advance()) {
        if (!mbar_wait_bounded(&bars.opW[slot], par, kWaitTimeoutNs)) {
          ok = false;
          break;
        }
        const unsigned char* src = ring + static_cast<uint32_t>(slot) * STAGE;
#pragma unroll
        for (int pl = 0; pl < PLANES; ++pl) {
          bulk_to_cluster(cluster_addr(src + pl * PLANE + kClBlock, d1), smem_u32(src + pl * PLANE), bytes,
                          cluster_addr(&bars.rx[slot], d1));
          if (R == 4 && r >= 2)
            bulk_to_cluster(cluster_addr(src + pl * PLANE + 2 * kClBlock, d2), smem_u32(src + pl * PLANE), bytes,
                            cluster_addr(&bars.rx[slot], d2));
        }
      }
    }
    // the other CTAs' last commits have arrived here before this CTA may go
    for (int j = max(0, k - S); j < k && ok; ++j)
      if (!mbar_wait_bounded(&bars.opE[j % S], static_cast<uint32_t>((j / S) & 1), kWaitTimeoutNs)) ok = false;
  }
  if (!ok) {
    atomicOr(p.err, ERR_TIMEOUT);
    const uint64_t t0 = global_timer_ns();           // copies in flight land well within this
    while (global_timer_ns() - t0 < 2000000ull) __nanosleep(1000);
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();                                // no copy and no commit arrives after this
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

namespace {

template <int PREC, int ISO>
cudaError_t cluster_launch_t(const ClusterGramParams& p, int clusters, cudaStream_t s, int* max_clusters) {
  auto kernel = gram_cluster_kernel<PREC, ISO>;
  const int smem = kClRing + 1024;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(p.R * clusters));
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(p.R);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (max_clusters != nullptr) return cudaOccupancyMaxActiveClusters(max_clusters, kernel, &cfg);
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int PREC>
cudaError_t cluster_launch(const ClusterGramParams& p, int clusters, cudaStream_t s) {
  const int kind = iso_kind(p.iso_mode);
  if (kind == ISOK_NONE) return cluster_launch_t<PREC, ISOK_NONE>(p, clusters, s, nullptr);
  if (kind == ISOK_NORMAL) return cluster_launch_t<PREC, ISOK_NORMAL>(p, clusters, s, nullptr);
  return cluster_launch_t<PREC, ISOK_STEP>(p, clusters, s, nullptr);
}

}  // namespace

int gram_cluster_stages(int R, int prec) {
  return std::min<int>(kClMaxStages, kClRing / (static_cast<int>(kClBlock) * (prec == 2 ? 2 : 1) * (R == 4 ? 3 : 2)));
}

cudaError_t launch_gram_cluster(const ClusterGramParams& p, const float* w, float* sqrt_w, int prec, int clusters,
                                cudaStream_t s) {
  const int n_flags = p.n_chunks > clusters ? clusters * p.R : 0;
  const int n = std::max(n_flags, w != nullptr ? (p.M + 127) / 128 * 128 : 0);
  if (n > 0) {
    gram_cluster_prep_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(w, p.M, sqrt_w, p.flags, n_flags);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (prec == 1) return cluster_launch<1>(p, clusters, s);
  if (prec == 2) return cluster_launch<2>(p, clusters, s);
  if (prec == 3) return cluster_launch<3>(p, clusters, s);
  return cudaErrorInvalidValue;
}

// Clusters of R CTAs that run at once (the same for every instantiation: the ring bounds it).
cudaError_t gram_max_clusters(int R, int* clusters) {
  ClusterGramParams p = {};
  p.R = R;
  return cluster_launch_t<1, ISOK_NONE>(p, 64, nullptr, clusters);
}

}  // namespace pidk
