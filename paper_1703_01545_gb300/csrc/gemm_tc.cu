// Split-BF16 ("BF16x3") tensor-core GEMM for the Cholesky contractions on sm_103a.
//
//   C[n*ldc + m] = alpha * sum_k (Ahi + Alo)[m][k] (Bhi + Blo)[n][k]     (lo*lo dropped)
//
// A float64 operand x is carried as x ~ hi + lo with hi = bf16(x), lo = bf16(x - hi), so
// each product needs three BF16 MMAs (hi*hi, hi*lo, lo*hi) accumulated in FP32 in tensor
// memory; the product error is about 2^-17 relative instead of BF16's 2^-9.
//
// Structure (one 128 x BN output tile per CTA, 4 warps):
//   warp 0 / lane 0  TMA producer: 128B-swizzled boxes of Ahi, Alo, Bhi, Blo per 64-wide
//                    k slice into a STAGES-deep ring, completion on a "full" mbarrier.
//   warp 1 / lane 0  MMA issuer: per k slice 4 x 3 tcgen05.mma (K = 16 each) into one TMEM
//                    accumulator, then tcgen05.commit frees the stage ("empty" mbarrier);
//                    a final commit signals "done".
//   all 4 warps      epilogue: tcgen05.ld of their 32 TMEM lanes (= 32 output rows m),
//                    scaled by alpha, stored so that a warp writes 32 consecutive m.
// Every mbarrier wait is bounded; on expiry the kernel sets *err, drains what it issued,
// frees its TMEM and returns.  Operand rows are K-major with K padded to a multiple of 64
// (zero-filled), so every TMA box starts on a 128-byte boundary.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "device_util.cuh"
#include "internal.h"
#include "tc_device.cuh"

namespace afq {
namespace {

using namespace tc;

constexpr int BM = 128, BK = 64, NTHREADS = 128;
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // 2 s: far beyond any legitimate wait here

template <int BN, int STAGES>
struct TcLayout {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
  static constexpr int BAR_OFFSET = STAGES * STAGE_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFFSET + 256 + 1024;  // barriers + TMEM slot + alignment
};

// Split output of 32 accumulator columns of output row m = i M + j: hi = bf16(x), lo =
// bf16(x - hi) at n * ld + i * Mp + j for columns n = n0 .. n0 + 31 below Nd.
__device__ __forceinline__ void store_split(const SplitOut& so, int m, int n0, int Nd, float alpha,
                                            const uint32_t (&v)[32]) {
  const int i = m / so.M, j = m - i * so.M;
  const int64_t off = (int64_t)i * so.Mp + j;
#pragma unroll
  for (int q = 0; q < 32; ++q) {
    const int n = n0 + q;
    if (n < Nd) {
      const float x = alpha * __uint_as_float(v[q]);
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      so.hi[(int64_t)n * so.ld + off] = h;
      so.lo[(int64_t)n * so.ld + off] = __float2bfloat16_rn(x - __bfloat162float(h));
    }
  }
}

// Lower-triangle block layout of the V_HS rows: tile tm is half h of block q = tm / 2 in the
// order (0,0), (1,0), (1,1), (2,0), ...; block (a, b), a >= b, holds the index pairs
// i in 16 a + [0, 16), j in 16 b + [0, 16), and half h the rows i in 16 a + 8 h + [0, 8).
// Row r of a tile is (i, j) = (16 a + 8 h + r / 16, 16 b + r % 16).
__device__ __forceinline__ void tri_tile(int tm, int& a, int& b, int& h) {
  const int q = tm >> 1;
  h = tm & 1;
  a = (int)((sqrtf(8.f * (float)q + 1.f) - 1.f) * 0.5f);
  while ((a + 1) * (a + 2) / 2 <= q) ++a;
  while (a * (a + 1) / 2 > q) --a;
  b = q - a * (a + 1) / 2;
}

// Split output of 16 accumulator columns of a half block of the lower triangle, by the 128 threads of an
// epilogue group (thread r holds the index pair (i, j) = (i0 + r / 16, j0 + r % 16)).  A pair of lanes
// (j even, j + 1) exchanges columns, so that each writes both of its j for half of them, 4 bytes at a time
// (rows of V are whole 16-byte units: what an odd M's last pair writes beyond j < M is the padding's zero).
// With `stg` ([16 columns][16 j][8 i] packed hi | lo words, the 16-byte halves of a j's 32 bytes swapped by
// bit 2 of j, so that neither side meets a bank conflict beyond two lanes) the values are also staged for
// the mirror block.
__device__ __forceinline__ void store_tri16(const SplitOut& so, int i, int j, int n0, int Nd, float alpha,
                                            const uint32_t (&v)[16], uint32_t* stg, int r) {
  const bool in = i < so.M && (j & ~1) < so.M;
  const int odd = j & 1, jj = r & 15, ii = r >> 4;
  const int64_t off = (int64_t)i * so.Mp + (j & ~1);
  uint32_t* sw = stg ? stg + jj * 8 + ((((ii >> 2) ^ (jj >> 2)) & 1) << 2) + (ii & 3) : nullptr;
#pragma unroll
  for (int q = 0; q < 16; q += 2) {
    uint32_t w[2];   // columns q, q + 1: hi in the low half
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float x = alpha * __uint_as_float(v[q + u]);
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
      w[u] = (uint32_t)__bfloat16_as_ushort(h) | ((uint32_t)__bfloat16_as_ushort(l) << 16);
      if (sw) sw[(q + u) * 128] = w[u];
    }
    // even lanes write column q, odd ones q + 1
    const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? w[0] : w[1], 1);
    const uint32_t lo_j = odd ? got : w[0], hi_j = odd ? w[1] : got;
    const int n = n0 + q + odd;
    if (in && n < Nd) {
      *reinterpret_cast<uint32_t*>(so.hi + (int64_t)n * so.ld + off) = __byte_perm(lo_j, hi_j, 0x5410);
      *reinterpret_cast<uint32_t*>(so.lo + (int64_t)n * so.ld + off) = __byte_perm(lo_j, hi_j, 0x7632);
    }
  }
}

// The staged half block written transposed: V[j][i0 .. i0 + 7] for the 16 j, 16 bytes per (column, j, hi /
// lo); two (column, j) tasks for each of the group's 128 threads.
__device__ __forceinline__ void store_mirror16(const SplitOut& so, const uint32_t* stg, int i0, int j0, int n0,
                                               int Nd, int tid) {
#pragma unroll
  for (int task = tid; task < 16 * 16; task += 128) {
    const int q = task >> 4, jj = task & 15, n = n0 + q, j = j0 + jj;
    const uint32_t* src = stg + q * 128 + jj * 8;
    const int f = (jj >> 2) & 1;
    const uint4 a = *reinterpret_cast<const uint4*>(src + 4 * f), b = *reinterpret_cast<const uint4*>(src + 4 * (f ^ 1));
    if (n >= Nd || j >= so.M) continue;
    const uint4 hi = make_uint4(__byte_perm(a.x, a.y, 0x5410), __byte_perm(a.z, a.w, 0x5410),
                                __byte_perm(b.x, b.y, 0x5410), __byte_perm(b.z, b.w, 0x5410));
    const uint4 lo = make_uint4(__byte_perm(a.x, a.y, 0x7632), __byte_perm(a.z, a.w, 0x7632),
                                __byte_perm(b.x, b.y, 0x7632), __byte_perm(b.z, b.w, 0x7632));
    const int64_t off = (int64_t)n * so.ld + (int64_t)j * so.Mp + i0;
    if (i0 < so.M) {   // a row's 8 elements lie within its pitch; beyond i < M they are zero
      *reinterpret_cast<uint4*>(so.hi + off) = hi;
      *reinterpret_cast<uint4*>(so.lo + off) = lo;
    }
  }
}

// AND of `ok` over the epilogue threads (named barrier 5): they leave the tile loop together, so none is
// left waiting at a staging barrier.
template <int THREADS>
__device__ __forceinline__ bool epilogue_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 5, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)ok), "n"(THREADS)
      : "memory");
  return r != 0;
}

// The four warps of epilogue group g (named barrier 1 + g, 128 threads).
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }

template <int BN, int STAGES, class TC>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_gemm_bf16x3_tc(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                     const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                     int Md, int Nd, int nkb, float alpha, TC* __restrict__ C, int64_t ldc,
                     SplitOut so, int* err, uint64_t wait_ns, int skip_producer) {
  after_previous();
  using Lay = TcLayout<BN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::BAR_OFFSET);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
  volatile int* s_fail = reinterpret_cast<volatile int*>(tmem_slot + 1);   // a wait for operands expired
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES),
                 done = smem_u32(bars + 2 * STAGES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- TMA producer (skip_producer: self-test of the bounded waits, nothing is issued) ----
    int issued = 0;
    for (int kb = 0; kb < (skip_producer ? 0 : nkb); ++kb) {
      const int s = kb % STAGES, use = kb / STAGES;
      if (kb >= STAGES && !mbar_wait(empty0 + 8 * s, (use - 1) & 1, err, wait_ns)) break;
      const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
      const uint32_t fb = full0 + 8 * s;
      mbar_expect_tx(fb, Lay::STAGE_BYTES);
      tma_load_2d(st, &tmAh, fb, kb * BK, m0);
      tma_load_2d(st + Lay::A_BYTES, &tmAl, fb, kb * BK, m0);
      tma_load_2d(st + 2 * Lay::A_BYTES, &tmBh, fb, kb * BK, n0);
      tma_load_2d(st + 2 * Lay::A_BYTES + Lay::B_BYTES, &tmBl, fb, kb * BK, n0);
      issued = kb + 1;
    }
    // drain: every issued stage must have landed before the CTA may exit
    for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb)
      mbar_wait(full0 + 8 * (kb % STAGES), (kb / STAGES) & 1, err, wait_ns);
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer ----
    const uint32_t idesc = idesc_bf16<BN>();
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % STAGES, use = kb / STAGES;
      if (!mbar_wait(full0 + 8 * s, use & 1, err, wait_ns)) {
        *s_fail = 1;
        __threadfence_block();
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
      const uint64_t ah = sw128_desc(st), al = sw128_desc(st + Lay::A_BYTES);
      const uint64_t bh = sw128_desc(st + 2 * Lay::A_BYTES);
      const uint64_t bl = sw128_desc(st + 2 * Lay::A_BYTES + Lay::B_BYTES);
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk) {
        const uint64_t dk = (uint64_t)((kk * 32) >> 4);  // advance 16 bf16 inside the swizzle atom
        mma_bf16(tmem, ah + dk, bh + dk, idesc, (kb | kk) != 0);
        mma_bf16(tmem, ah + dk, bl + dk, idesc, 1u);
        mma_bf16(tmem, al + dk, bh + dk, idesc, 1u);
      }
      mma_commit(empty0 + 8 * s);
    }
    mma_commit(done);  // also on an early exit: arrives once the issued MMAs are complete
  }
  __syncwarp();

  // ---- epilogue: TMEM lanes 32*warp .. 32*warp+31 hold output rows m ----
  const bool ok = mbar_wait(done, 0, err, 2 * wait_ns);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncwarp();
  const int m = m0 + warp * 32 + lane;
  if (__all_sync(0xffffffffu, ok && *s_fail == 0)) {
    for (int c0 = 0; c0 < BN; c0 += 32) {
      uint32_t v[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
      if (m < Md) {
        if (so.hi) {
          store_split(so, m, n0 + c0, Nd, alpha, v);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int n = n0 + c0 + j;
            if (n < Nd) C[(int64_t)n * ldc + m] = (TC)(alpha * __uint_as_float(v[j]));
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN)
                 : "memory");
}

// Persistent variant for one row tile and many columns (where a pair would leave a CTA without rows):
// 128 x 256 tiles, grid = one CTA
// per SM looping over tiles, 10 warps.
//   warp 8 / lane 0  TMA producer over all of the CTA's tiles (2-stage ring of 96 KB stages)
//   warp 9 / lane 0  MMA issuer: tile i accumulates into TMEM buffer i & 1 (2 x 256 columns),
//                    commits "tile full" for the epilogue and waits for "tile empty" before it
//                    reuses a buffer
//   warps 0..7       epilogue, two groups of four: group g drains columns 128 g .. 128 g + 127
//                    of buffer i & 1 (warp w reads TMEM lanes 32 (w % 4) ..) while the MMAs of
//                    tile i + 1 run, then arrives on "tile empty"
// Tiles run m-fastest, so consecutive CTAs share B tiles.  Every wait is bounded as above.
constexpr int PBN = 256, PSTAGES = 2, PTHREADS = 320, PEPI = 256;   // PEPI: epilogue threads
struct PLayoutG {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_BYTES = PBN * BK * 2;
  static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
  static constexpr int BAR_OFFSET = PSTAGES * STAGE_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFFSET + 256 + 1024;
};

// Accumulator columns cbeg .. cbeg + cnt - 1 of the lanes at TMEM address `acc`: output row m of the thread.
__device__ __forceinline__ void store_columns(const SplitOut& so, float* __restrict__ C, int64_t ldc, uint32_t acc,
                                              int m, int n0, int cbeg, int cnt, int Md, int Nd, float alpha) {
  for (int c0 = cbeg; c0 < cbeg + cnt; c0 += 32) {
    uint32_t v[32];
    tmem_ld32(acc + (uint32_t)c0, v);
    if (m < Md) {
      if (so.hi) {
        store_split(so, m, n0 + c0, Nd, alpha, v);
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int n = n0 + c0 + j;
          if (n < Nd) C[(int64_t)n * ldc + m] = alpha * __uint_as_float(v[j]);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(PTHREADS, 1)
    k_gemm_bf16x3_tc_persist(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                             const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                             int Md, int Nd, int nkb, float alpha, float* __restrict__ C, int64_t ldc,
                             SplitOut so, int* err, uint64_t wait_ns) {
  after_previous();
  using Lay = PLayoutG;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::BAR_OFFSET);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * PSTAGES + 5);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + PSTAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * PSTAGES), tempty0 = smem_u32(bars + 2 * PSTAGES + 2);
  const uint32_t done = smem_u32(bars + 2 * PSTAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = (Md + BM - 1) / BM, ntiles = mt * ((Nd + PBN - 1) / PBN);

  if (threadIdx.x == 0) {
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, PEPI);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 8) {
    if (lane == 0) {
      // ---- TMA producer ----
      int g = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int m0 = (t % mt) * BM, n0 = (t / mt) * PBN;
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          const int s = g % PSTAGES, use = g / PSTAGES;
          if (g >= PSTAGES && !mbar_wait(empty0 + 8 * s, (use - 1) & 1, err, wait_ns)) { ok = false; break; }
          const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
          const uint32_t fb = full0 + 8 * s;
          mbar_expect_tx(fb, Lay::STAGE_BYTES);
          tma_load_2d(st, &tmAh, fb, kb * BK, m0);
          tma_load_2d(st + Lay::A_BYTES, &tmAl, fb, kb * BK, m0);
          const uint32_t bh = st + 2 * Lay::A_BYTES, bl = bh + Lay::B_BYTES;
          tma_load_2d(bh, &tmBh, fb, kb * BK, n0);
          tma_load_2d(bh + Lay::B_BYTES / 2, &tmBh, fb, kb * BK, n0 + PBN / 2);
          tma_load_2d(bl, &tmBl, fb, kb * BK, n0);
          tma_load_2d(bl + Lay::B_BYTES / 2, &tmBl, fb, kb * BK, n0 + PBN / 2);
        }
      }
      // every issued stage must have landed before the CTA may exit
      for (int q = (g > PSTAGES ? g - PSTAGES : 0); q < g; ++q)
        mbar_wait(full0 + 8 * (q % PSTAGES), (q / PSTAGES) & 1, err, wait_ns);
    }
  } else if (warp == 9) {
    if (lane == 0) {
      // ---- MMA issuer ----
      const uint32_t idesc = idesc_bf16<PBN>();
      int g = 0, i = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
        const int b = i & 1;
        if (i >= 2 && !mbar_wait(tempty0 + 8 * b, ((i >> 1) - 1) & 1, err, wait_ns)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + (uint32_t)(b * PBN);
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          const int s = g % PSTAGES, use = g / PSTAGES;
          if (!mbar_wait(full0 + 8 * s, use & 1, err, wait_ns)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
          const uint64_t ah = sw128_desc(st), al = sw128_desc(st + Lay::A_BYTES);
          const uint64_t bh = sw128_desc(st + 2 * Lay::A_BYTES);
          const uint64_t bl = sw128_desc(st + 2 * Lay::A_BYTES + Lay::B_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t dk = (uint64_t)((kk * 32) >> 4);
            mma_bf16(d, ah + dk, bh + dk, idesc, (kb | kk) != 0);
            mma_bf16(d, ah + dk, bl + dk, idesc, 1u);
            mma_bf16(d, al + dk, bh + dk, idesc, 1u);
          }
          mma_commit(empty0 + 8 * s);
        }
        if (ok) mma_commit(tfull0 + 8 * b);
      }
      mma_commit(done);   // arrives once every issued MMA has completed
    }
  } else {
    // ---- epilogue: warp w drains TMEM lanes 32 (w % 4) .. + 31 (output rows m) of its
    // group's columns 128 g .. 128 g + 127 ----
    int i = 0;
    const int grp = warp >> 2, wq = warp & 3;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
      const int b = i & 1, m0 = (t % mt) * BM, n0 = (t / mt) * PBN;
      const bool ok = mbar_wait(tfull0 + 8 * b, (i >> 1) & 1, err, wait_ns);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!__all_sync(0xffffffffu, ok)) break;
      store_columns(so, C, ldc, tmem + (uint32_t)(b * PBN) + ((uint32_t)(wq * 32) << 16), m0 + wq * 32 + lane, n0,
                    grp * (PBN / 2), PBN / 2, Md, Nd, alpha);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(tempty0 + 8 * b);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(done, 0, err, wait_ns);   // no MMA may still write TMEM
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// The persistent kernel by pairs of SMs (cta_group::2): a cluster of two CTAs computes a 256 x 256 tile,
// each with 128 of its rows (A and the accumulator) and half of its columns' B operand in its own shared
// memory; the first CTA issues the MMAs for both.  A 64-wide k slice of hi and lo operands is 64 KB a CTA
// instead of the 96 KB of a 128 x 256 tile: with 12 MMAs of some 131 cycles a slice, one CTA per tile
// asked L2 for 61 bytes a cycle and SM, 7.7 TB/s over the chip, which bounded it.  Ring of 3 stages.
//   warp 16 / lane 0  TMA producer of its CTA's operands; every byte of both CTAs counts on the first
//                     CTA's "full" barrier
//   warp 17 / lane 0  (first CTA) MMA issuer; its commits arrive on the barriers of both CTAs
//   warps 0..15       epilogue of the CTA's own 128 rows, four groups of four warps with 64 columns each;
//                     "tile empty" counts the warps of both
// The V_HS epilogue (split, transposed for the mirror block) was the longer side of a tile with 8 warps
// and 2-byte accesses (36 k cycles beside 19 k of MMAs at K = 768), hence 16 warps, 4-byte stores of lane
// pairs and 16-byte staging reads.  V_HS at M = 128, X = 768, 4096 walkers, beside the other system's
// kernels: 344 us with one CTA per tile, 313 us by pairs with the old epilogue, 273 us so (tensor pipe 54 %
// active, L2 45 %, the last of the tiles' waves half empty at smaller sizes); M = 64, 2048 walkers:
// 32.4 -> 28.8 us; M = 200: 495 -> 436 us.
constexpr int QSTAGES = 3, QEPI = 512, QTHREADS = QEPI + 64;
struct QLayout {
  static constexpr int T_BYTES = 128 * BK * 2;
  static constexpr int STAGE_BYTES = 4 * T_BYTES;   // A hi, lo, B hi, lo
  static constexpr int STG_OFFSET = QSTAGES * STAGE_BYTES;
  static constexpr int STG_BYTES = 16 * 16 * 8 * 4;   // mirror staging of an epilogue group
  static constexpr int BAR_OFFSET = STG_OFFSET + 4 * STG_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFFSET + 256 + 1024;
};

// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// TMA load into this CTA whose bytes count on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far have completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(1000000u)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, int* err, uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  do {
    if (try_wait_cluster(bar, parity)) return true;
  } while (global_ns() - t0 <= limit_ns);
  atomicOr(err, 1);
  return false;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(QTHREADS, 1)
    k_gemm_bf16x3_tc_pair(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                          const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl,
                          int Md, int Nd, int nkb, float alpha, float* __restrict__ C, int64_t ldc,
                          SplitOut so, int* err, uint64_t wait_ns) {
  after_previous();
  using Lay = QLayout;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::BAR_OFFSET);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * QSTAGES + 5);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + QSTAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * QSTAGES), tempty0 = smem_u32(bars + 2 * QSTAGES + 2);
  const uint32_t done = smem_u32(bars + 2 * QSTAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
  const int mt = (Md + 2 * BM - 1) / (2 * BM), ntiles = mt * ((Nd + PBN - 1) / PBN);

  if (threadIdx.x == 0) {
    for (int s = 0; s < QSTAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, 2 * (QEPI / 32));
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  cluster_sync();   // both CTAs' barriers are initialised
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 16) {
    if (lane == 0) {
      // ---- TMA producer ----
      int s = 0, g = 0;
      uint32_t ph = 0;   // parity of the stage's current use
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += npairs) {
        const int m0 = (2 * (t % mt) + rank) * BM, n0 = (t / mt) * PBN + rank * (PBN / 2);
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          if (g >= QSTAGES && !mbar_wait(empty0 + 8 * s, ph ^ 1u, err, wait_ns)) { ok = false; break; }
          const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
          const uint32_t fb = map_rank(full0 + 8 * s, 0);
          if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2 * Lay::STAGE_BYTES);
          tma_load_2d_pair(st, &tmAh, fb, kb * BK, m0);
          tma_load_2d_pair(st + Lay::T_BYTES, &tmAl, fb, kb * BK, m0);
          tma_load_2d_pair(st + 2 * Lay::T_BYTES, &tmBh, fb, kb * BK, n0);
          tma_load_2d_pair(st + 3 * Lay::T_BYTES, &tmBl, fb, kb * BK, n0);
          if (++s == QSTAGES) { s = 0; ph ^= 1u; }
        }
      }
      // every issued stage of both CTAs must have landed before either may exit (the other one's bytes
      // and this one's count here)
      if (rank == 0) {
        const int left = g < QSTAGES ? g : QSTAGES;
        for (int q = g - left; q < g; ++q)
          mbar_wait(full0 + 8 * (q % QSTAGES), (q / QSTAGES) & 1, err, wait_ns);
      }
    }
  } else if (warp == 17) {
    if (lane == 0 && rank == 0) {
      // ---- MMA issuer ----
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(PBN >> 3) << 17) |
                             ((uint32_t)(2 * BM >> 4) << 24);
      int s = 0, i = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += npairs, ++i) {
        const int b = i & 1;
        if (i >= 2 && !wait_cluster(tempty0 + 8 * b, ((i >> 1) - 1) & 1, err, wait_ns)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + (uint32_t)(b * PBN);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(full0 + 8 * s, ph, err, wait_ns)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = smem_u32(smem + s * Lay::STAGE_BYTES);
          const uint64_t ah = sw128_desc(st), al = sw128_desc(st + Lay::T_BYTES);
          const uint64_t bh = sw128_desc(st + 2 * Lay::T_BYTES), bl = sw128_desc(st + 3 * Lay::T_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t dk = (uint64_t)((kk * 32) >> 4);
            mma_bf16_pair(d, ah + dk, bh + dk, idesc, (kb | kk) != 0);
            mma_bf16_pair(d, ah + dk, bl + dk, idesc, 1u);
            mma_bf16_pair(d, al + dk, bh + dk, idesc, 1u);
          }
          mma_commit_pair(empty0 + 8 * s);
          if (++s == QSTAGES) { s = 0; ph ^= 1u; }
        }
        if (ok) mma_commit_pair(tfull0 + 8 * b);
      }
      mma_commit_pair(done);   // arrives once every issued MMA has completed
    }
  } else {
    // ---- epilogue ----
    int i = 0;
    const int grp = warp >> 2, wq = warp & 3, r = wq * 32 + lane;
    uint32_t* stg = reinterpret_cast<uint32_t*>(smem + Lay::STG_OFFSET + grp * Lay::STG_BYTES);
    for (int t = pair; t < ntiles; t += npairs, ++i) {
      const int b = i & 1, tm = 2 * (t % mt) + rank, n0 = (t / mt) * PBN;
      const bool ok = mbar_wait(tfull0 + 8 * b, (i >> 1) & 1, err, wait_ns);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!epilogue_all<QEPI>(ok)) break;
      const uint32_t acc = tmem + (uint32_t)(b * PBN) + ((uint32_t)(wq * 32) << 16);
      if (so.tri) {
        // lower-triangle block rows: V[i][j] directly and, off the diagonal, V[j][i] through the staging
        int ba, bb, bh;
        tri_tile(tm, ba, bb, bh);
        const int i0 = 16 * ba + 8 * bh, j0 = 16 * bb;
        const bool mirror = ba != bb;
        for (int c0 = 64 * grp; c0 < 64 * grp + 64; c0 += 16) {
          uint32_t v[16];
          tmem_ld16(acc + (uint32_t)c0, v);
          store_tri16(so, i0 + (r >> 4), j0 + (r & 15), n0 + c0, Nd, alpha, v, mirror ? stg : nullptr, r);
          if (mirror) {
            group_sync(grp);   // the half block's 16 columns are staged
            store_mirror16(so, stg, i0, j0, n0 + c0, Nd, r);
            group_sync(grp);   // and written: the group's staging array is free again
          }
        }
      } else {
        store_columns(so, C, ldc, acc, tm * BM + r, n0, 64 * grp, 64, Md, Nd, alpha);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) arrive_remote(map_rank(tempty0 + 8 * b, 0));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(done, 0, err, wait_ns);   // no MMA may still write TMEM
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncthreads();
  // neither CTA's shared or tensor memory, nor its barriers, are used by the other any more
  cluster_sync();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// Clusters of the pair kernel that the device holds at once (its grid: a cluster that waited for an SM
// would run its tiles after the others').
int find_pair_clusters() {
  static int have[64] = {};
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (!have[dev]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(152);
    cfg.blockDim = dim3(QTHREADS);
    cfg.dynamicSmemBytes = QLayout::SMEM_BYTES;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_gemm_bf16x3_tc_pair, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    have[dev] = n > 0 ? n : -1;
  }
  return std::max(have[dev], 0);
}

// ---- operand preparation ----

// split rows of a float64 matrix into bf16 hi/lo, K padded with zeros:
// out_{hi,lo}[r][k] for k < Kp; in[r*ld_in + k] for k < K.
__global__ void k_split_bf16(const double* __restrict__ in, int64_t ld_in, int rows, int K, int Kp,
                             __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo) {
  const int64_t total = (int64_t)rows * Kp;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / Kp;
    const int k = (int)(e % Kp);
    const double x = k < K ? in[r * ld_in + k] : 0.0;
    const __nv_bfloat16 h = __float2bfloat16_rn((float)x);
    hi[e] = h;
    lo[e] = __float2bfloat16_rn((float)(x - (double)__bfloat162float(h)));
  }
}

// The lower-triangle block rows (tri_tile) of the V_HS operand: row r of tile r / 128 is the
// index pair (i, j) of row i M + j of `in` ([M^2][ld_in]), zero outside the M x M matrix.
__global__ void k_split_bf16_tri(const double* __restrict__ in, int64_t ld_in, int M, int rows,
                                 int K, int Kp, __nv_bfloat16* __restrict__ hi,
                                 __nv_bfloat16* __restrict__ lo) {
  const int64_t total = (int64_t)rows * Kp;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / Kp), k = (int)(e % Kp);
    int a, b, h;
    tri_tile(r >> 7, a, b, h);
    const int i = 16 * a + 8 * h + ((r & 127) >> 4), j = 16 * b + (r & 15);
    const double x = (k < K && i < M && j < M) ? in[((int64_t)i * M + j) * ld_in + k] : 0.0;
    const __nv_bfloat16 hh = __float2bfloat16_rn((float)x);
    hi[e] = hh;
    lo[e] = __float2bfloat16_rn((float)(x - (double)__bfloat162float(hh)));
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

template <int BN, int STAGES, class TC>
cudaError_t launch_tc(const TcOperand& A, const TcOperand& B, int Md, int Nd, float alpha, TC* C,
                      int64_t ldc, int* err, cudaStream_t s, uint64_t wait_ns = kWaitLimitNs,
                      int skip_producer = 0, SplitOut so = SplitOut()) {
  using Lay = TcLayout<BN, STAGES>;
  dim3 grid((Md + BM - 1) / BM, (Nd + BN - 1) / BN);
  if (grid.y > 65535u) return cudaErrorInvalidConfiguration;
  return launch_after(k_gemm_bf16x3_tc<BN, STAGES, TC>, grid, NTHREADS, Lay::SMEM_BYTES, s, A.map_hi, A.map_lo,
                      B.map_hi, B.map_lo, Md, Nd, A.Kp / BK, alpha, C, ldc, so, err, wait_ns, skip_producer);
}

}  // namespace

cudaError_t tc_make_operand(TcOperand& op, __nv_bfloat16* hi, __nv_bfloat16* lo, int rows, int Kp,
                            int box_rows) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  // rows must be whole boxes (buffers are padded), so no box ever reaches outside the tensor
  if (Kp % BK != 0 || rows < 1 || rows % box_rows != 0) return cudaErrorInvalidValue;
  op.hi = hi;
  op.lo = lo;
  op.rows = rows;
  op.Kp = Kp;
  cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  for (int q = 0; q < 2; ++q) {
    CUresult r = fn(q == 0 ? &op.map_hi : &op.map_lo, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                    q == 0 ? (void*)hi : (void*)lo, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

cudaError_t split_bf16(const double* in, int64_t ld_in, int rows, int K, int Kp, __nv_bfloat16* hi,
                       __nv_bfloat16* lo, cudaStream_t s) {
  const int64_t total = (int64_t)rows * Kp;
  int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 64);
  if (grid < 1) grid = 1;
  k_split_bf16<<<grid, 256, 0, s>>>(in, ld_in, rows, K, Kp, hi, lo);
  return cudaGetLastError();
}

int vhs_tri_rows(int M) {
  const int nb = (M + 15) / 16;
  return nb * (nb + 1) / 2 * 2 * BM;
}

cudaError_t split_bf16_tri(const double* in, int64_t ld_in, int M, int K, int Kp, __nv_bfloat16* hi,
                           __nv_bfloat16* lo, cudaStream_t s) {
  const int rows = vhs_tri_rows(M);
  const int64_t total = (int64_t)rows * Kp;
  int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 64);
  if (grid < 1) grid = 1;
  k_split_bf16_tri<<<grid, 256, 0, s>>>(in, ld_in, M, rows, K, Kp, hi, lo);
  return cudaGetLastError();
}

static bool tc_persistent_ok(int Md, int Nd, int b_rows) {
  const int64_t tiles = (int64_t)((Md + BM - 1) / BM) * ((Nd + PBN - 1) / PBN);
  return tiles >= 2 * 152 && b_rows % PBN == 0;
}

// Whether 256 x 256 tiles by pairs of SMs beat 128 x 128 tiles by single ones (of Md1 rows: all M^2 for a
// lower triangle), in whole waves: a 64-wide k slice takes a pair's tile about 1.6 k cycles (its MMAs) and a
// single's 1.3 k (its 64 KB from L2).  Steps with the old line (two 128 x 256 tiles an SM, whole 256-column
// tiles) and this one: M = 200, 300 walkers 484 -> 370 us, M = 150, 800 walkers 691 -> 605, M = 128, 300
// walkers 231 -> 204, 100 walkers 168 -> 149, M = 101, 777 walkers 315 -> 291; the force bias at M = 128 and
// 4096 walkers (6 x 64 single tiles, three waves; 96 pairs, two) 133 -> 124 us.  M = 90, 200 walkers and
// M = 64, 2048 walkers' force bias (three row tiles, one wave either way) stay with single tiles.
static bool pair_pays(int64_t Md, int64_t Nd, int64_t Md1) {
  const int np = find_pair_clusters();
  const int64_t pt = (Md + 2 * BM - 1) / (2 * BM) * ((Nd + PBN - 1) / PBN);
  const int64_t t1 = (Md1 + BM - 1) / BM * ((Nd + 127) / 128);
  return np > 0 && (pt + np - 1) / np * 6 < (t1 + 151) / 152 * 5;
}

// The lower-triangle output is the pair kernel's.
bool vhs_tri_ok(int M, int Nd) { return pair_pays(vhs_tri_rows(M), Nd, (int64_t)M * M); }

// A operand boxes are BM = 128 rows; B operand boxes are tc_bn() rows.  Operand buffers
// hold pad_rows(rows) rows (zero-filled beyond `rows`).
int tc_bn() { return 128; }
int tc_pad_rows(int rows) { return (rows + 127) / 128 * 128; }

namespace {
cudaError_t gemm_f32_or_split(const TcOperand& A, const TcOperand& B, int Md, int Nd, float alpha,
                              float* C, int64_t ldc, const SplitOut& so, int* err, cudaStream_t s) {
  if (A.Kp != B.Kp || Md > A.rows || Nd > B.rows) return cudaErrorInvalidValue;
  if (Md <= 0 || Nd <= 0) return cudaSuccess;
  if (so.tri && !vhs_tri_ok(so.M, Nd)) return cudaErrorInvalidValue;
  if (so.tri || (A.pairs && pair_pays(Md, Nd, Md))) {
    const int64_t pt = (int64_t)((Md + 2 * BM - 1) / (2 * BM)) * ((Nd + PBN - 1) / PBN);
    return launch_after(k_gemm_bf16x3_tc_pair, 2 * (int)std::min<int64_t>(pt, find_pair_clusters()), QTHREADS,
                        QLayout::SMEM_BYTES, s, A.map_hi, A.map_lo, B.map_hi, B.map_lo, Md, Nd, A.Kp / BK, alpha, C,
                        ldc, so, err, kWaitLimitNs);
  }
  // at least two 128 x 256 tiles per SM (here: a single row tile, X <= 128 or M <= 11): the persistent kernel,
  // whose epilogue overlaps the next tile's MMAs; B tiles of 256 rows stay inside the operand's padded rows (a
  // multiple of 256 here).  Force bias, us: this kernel / pairs of SMs / 128 x 128 tiles: X = 128, K = 192,
  // 39000 walkers 23.7 / 30.4 / 34.5, 60000 34.8 / 44.4 / 51.9, 77000 37.9 / 50.6 / 63.2; X = 90, K = 128, 50000
  // walkers 21.0 / 31.9 / 35.5; X = 120, K = 512, 60000 walkers 63.0 / 63.6 / 74.6
  if (tc_persistent_ok(Md, Nd, B.rows)) {
    const int64_t tiles = (int64_t)((Md + BM - 1) / BM) * ((Nd + PBN - 1) / PBN);
    const int grid = (int)std::min<int64_t>(tiles, 152);
    return launch_after(k_gemm_bf16x3_tc_persist, grid, PTHREADS, PLayoutG::SMEM_BYTES, s, A.map_hi, A.map_lo,
                        B.map_hi, B.map_lo, Md, Nd, A.Kp / BK, alpha, C, ldc, so, err, kWaitLimitNs);
  }
  return launch_tc<128, 3, float>(A, B, Md, Nd, alpha, C, ldc, err, s, kWaitLimitNs, 0, so);
}
}  // namespace

cudaError_t gemm_bf16x3(const TcOperand& A, const TcOperand& B, int Md, int Nd, float alpha,
                        float* C, int64_t ldc, int* err, cudaStream_t s) {
  return gemm_f32_or_split(A, B, Md, Nd, alpha, C, ldc, SplitOut(), err, s);
}

cudaError_t gemm_bf16x3_split_out(const TcOperand& A, const TcOperand& B, int Md, int Nd,
                                  float alpha, const SplitOut& so, int* err, cudaStream_t s) {
  if (!so.hi || !so.lo || so.M < 1 || so.Mp < so.M || so.ld < (int64_t)so.M * so.Mp ||
      (so.tri ? vhs_tri_rows(so.M) != Md || so.Mp % 8 != 0 || so.ld % 8 != 0
              : (int64_t)so.M * so.M != Md))
    return cudaErrorInvalidValue;
  return gemm_f32_or_split(A, B, Md, Nd, alpha, nullptr, 0, so, err, s);
}

cudaError_t gemm_bf16x3(const TcOperand& A, const TcOperand& B, int Md, int Nd, float alpha,
                        double* C, int64_t ldc, int* err, cudaStream_t s) {
  if (A.Kp != B.Kp || Md > A.rows || Nd > B.rows) return cudaErrorInvalidValue;
  if (Md <= 0 || Nd <= 0) return cudaSuccess;
  return launch_tc<128, 3, double>(A, B, Md, Nd, alpha, C, ldc, err, s);
}

// Self-test of the bounded waits: the producer issues nothing, so the MMA issuer's wait on
// the first stage expires after `wait_ns`; the kernel must set *err and exit cleanly.
cudaError_t gemm_bf16x3_wait_selftest(const TcOperand& A, const TcOperand& B, int Md, int Nd,
                                      float* C, int64_t ldc, int* err, uint64_t wait_ns,
                                      cudaStream_t s) {
  if (A.Kp != B.Kp || Md > A.rows || Nd > B.rows || Md <= 0 || Nd <= 0) return cudaErrorInvalidValue;
  return launch_tc<128, 3, float>(A, B, Md, Nd, 1.0f, C, ldc, err, s, wait_ns, 1);
}

// Once per device, before any launch or capture: the rings need up to ~217 KB of shared memory.
cudaError_t prepare_tc_kernels() {
  static SmemLimits limits;
  auto raise = [&](int slot, auto k, int bytes) {
    return limits.raise(slot, (size_t)bytes, [&] {
      return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    });
  };
  using Lay = TcLayout<128, 3>;
  cudaError_t e = raise(0, k_gemm_bf16x3_tc<128, 3, float>, Lay::SMEM_BYTES);
  if (e == cudaSuccess) e = raise(1, k_gemm_bf16x3_tc<128, 3, double>, Lay::SMEM_BYTES);
  if (e == cudaSuccess) e = raise(2, k_gemm_bf16x3_tc_persist, PLayoutG::SMEM_BYTES);
  if (e == cudaSuccess) e = raise(3, k_gemm_bf16x3_tc_pair, QLayout::SMEM_BYTES);
  if (e == cudaSuccess) find_pair_clusters();   // asked for here, after the limit and not under a capture
  return e;
}

}  // namespace afq
