// FP64 contraction on the BF16 tensor cores, exact to the last bits of float64.
//
//   C[n*ldc + m] = alpha * sum_k A[m*lda + k] * B[n*ldb + k]  (+ beta * C)
//
// GB300's FP64 pipe issues two multiply-adds per clock and SM, the tensor cores 4096 in BF16,
// so a float64 product formed from 36 BF16 products has about 55 times the pipe's rate.  The
// digits follow Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012): the products are
// error-free, so nothing is lost but what lies below the 62 bits kept of every element.
//
//   Digits.  Row r of an operand is scaled by 2^-E, E the exponent of its largest element, and
//   rounded to the 62-bit integer Y = round(x 2^(62-E)) = sum_j d_j 2^(56-8j), j = 0..7, with
//   balanced digits: |d_0| <= 64, -128 <= d_j <= 127.  A BF16 number holds every integer up to
//   256 exactly, and a product of two digits every bit in FP32.
//   Levels.  S_l = sum_k sum_{i+j=l} d^A_i d^B_j, l = 0..7: 36 digit pairs; the pairs beyond
//   l = 7 are below 2^-64 of (row maximum of A) (row maximum of B) each.  The FP32 sums of a
//   chunk of 256 k are exact integers where they must be: |S_l| <= 2^24 for l <= 4 by the
//   digit bounds, and a rounding of the levels 5..7 (weights 2^-40 and below) is beyond the
//   53 bits of the result.
//   Sum.  V = sum_l S_l 2^(56-8l) is accumulated over the chunks as a 96-bit integer and
//   rounded once to float64: no operation touches the FP64 pipe.
// The result carries the rounding of the operands to 62 bits of their row maximum and one final
// rounding, where the multiply-add chain of the SIMT kernel rounds K times.
//
// A_i meets B_0 .. B_(7-i), whose products belong to the levels i .. 7: with the digits of B as
// consecutive 64-row blocks of one shared-memory tile and the levels as consecutive 64-column
// blocks of tensor memory, that is one contiguous window, so a K step of 16 takes 12 MMAs (N up
// to 256) for the 36 products.
//
// One CTA per SM, persistent over (128 x 64 tile, K range) items; all 512 TMEM columns hold the
// 8 levels of one tile.
//   warp 8   TMA producer: the 8 digits of a 64-row, 64-wide B block in one 64 KB box
//            (2 stages), the digits of A as 16 KB boxes (6 slots)
//   warp 9   MMA issuer
//   warps 0..7  epilogue: a thread holds one row and 32 columns; per chunk it reads the 8 levels
//            and adds them to its 96-bit sums, after the item's last chunk it rounds and stores
//            while the next item's MMAs run
// Bounds of a 128 x 64 tile and 16 k: 1184 cycles of MMA (of which 32 for windows whose operand
// reads outlast their products), and 49 KB of digits from L2, 42 bytes per clock and SM.
// Measured (GB300, relative 2-norm error against exact rational arithmetic in brackets): the
// contractions of the reverse-mode run at M = 96, X = 480, 128 walkers, 10 steps, 223 ms on the
// FP64 pipe [2.6e-16 .. 1.1e-15 for a float64 multiply-add chain], 17.5 ms here with the digits
// and partial sums [4.3e-17 .. 1.2e-16].
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "internal.h"
#include "tc_device.cuh"

namespace afq {
namespace {

using namespace tc;

constexpr int kDig = 8;                        // digits per element
constexpr int kBR = 128, kBC = 64, kBK = 64;   // tile rows, columns, K block
constexpr int kChunk = 4;                      // K blocks per exact chunk (256 k)
constexpr int kASlots = 6, kBStages = 2;
constexpr int kABytes = kBR * kBK * 2, kBBytes = kDig * kBC * kBK * 2;
constexpr int kThreadsE = 320, kEpi = 256;
constexpr int kBarOff = kBStages * kBBytes + kASlots * kABytes;
constexpr int kSmemE = kBarOff + 256 + 1024;
constexpr uint64_t kWaitE = 2000000000ull;
constexpr int kExpNaN = 4095, kExpInf = 4094;  // exponent marks of rows with NaN / infinities

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x,
                                            int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}

__device__ __forceinline__ uint32_t elect_lane() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}"
               : "=r"(p));
  return p;
}

__device__ __forceinline__ uint32_t idesc_cols(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// V 2^(ea + eb - 25 - 32 ...) as float64: V = hi 2^32 + lo (96-bit two's complement) scaled so
// that a = b = 1 with one k gives V = 2^66 and ea = eb = 1023 (biased exponents of the row
// maxima).  One rounding, to nearest.
__device__ __forceinline__ double level_sum_to_f64(long long hi, uint32_t lo, int ea, int eb) {
  const uint32_t neg = hi < 0;
  uint64_t h = (uint64_t)hi;
  if (neg) {
    lo = 0u - lo;
    h = ~h + (lo == 0u ? 1ull : 0ull);
  }
  uint64_t top;
  int n;
  if (h) {
    n = __clzll((long long)h);
    top = n ? (h << n) | (((uint64_t)lo << 32) >> (64 - n)) : h;
  } else {
    if (lo == 0u) return 0.0;
    const int c = __clz((int)lo);
    n = 64 + c;
    top = (uint64_t)lo << (32 + c);
  }
  const uint64_t m = (top >> 11) + ((top >> 10) & 1ull);
  const int be1 = ea + eb - 995 - n;   // biased exponent of m 2^..., less the implicit bit's one
  uint64_t r;   // its magnitude's bits: m carries the implicit bit into the exponent field
  if (be1 >= 0)
    r = be1 > 2045 ? 0x7ff0000000000000ull : (uint64_t)min((unsigned long long)(((uint64_t)be1 << 52) + m), 0x7ff0000000000000ull);
  else          // subnormal
    r = be1 < -54 ? 0ull : (m + (1ull << (-be1 - 1))) >> -be1;
  return __longlong_as_double((long long)(r | ((uint64_t)neg << 63)));
}

struct EArgs {
  int R, Cn;               // valid rows and columns (of this launch)
  int rt, ct, ks;          // row tiles, column tiles, K ranges
  int nkb, kbs;            // K blocks in all, per range
  int swap;                // 0: out[c * ldc + r]; 1: out[r * ldc + c]
  int vec2;                // swap: pairs of columns may be stored as 16 bytes
  double alpha, beta;
  double* out;
  int64_t ldc;
  int64_t part;            // ks > 1: doubles per K range of the partial sums
  const int *er, *ec;      // row exponents of both operands
  const double *rsrc, *csrc;   // the operands themselves (rows with infinities)
  int64_t ldr, ldcs;
  int K;
  int* err;
};

__global__ void __launch_bounds__(kThreadsE, 1)
    k_gemm_f64e(const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmC, const EArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kBarOff);
  const uint32_t fullA = smem_u32(bars), emptyA = smem_u32(bars + kASlots);
  const uint32_t fullB = smem_u32(bars + 2 * kASlots), emptyB = fullB + 8 * kBStages;
  const uint32_t tfull = emptyB + 8 * kBStages, tempty = tfull + 8, done = tempty + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kASlots + 2 * kBStages + 3);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles = a.rt * a.ct, items = tiles * a.ks;

  if (threadIdx.x == 0) {
    for (int q = 0; q < kASlots; ++q) {
      mbar_init(fullA + 8 * q, 1);
      mbar_init(emptyA + 8 * q, 1);
    }
    for (int q = 0; q < kBStages; ++q) {
      mbar_init(fullB + 8 * q, 1);
      mbar_init(emptyB + 8 * q, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, kEpi);
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
      const uint32_t sB = smem_u32(smem), sA = sB + kBStages * kBBytes;
      int ga = 0, gb = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
        const int tile = t % tiles, r0 = (tile % a.rt) * kBR, c0 = (tile / a.rt) * kBC;
        const int kb0 = (t / tiles) * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
        for (int kb = kb0; kb < kb1 && ok; ++kb, ++gb) {
          const int sb = gb % kBStages;
          if (gb >= kBStages && !mbar_wait(emptyB + 8 * sb, (gb / kBStages - 1) & 1, a.err, kWaitE)) {
            ok = false;
            break;
          }
          mbar_expect_tx(fullB + 8 * sb, kBBytes);
          tma_load_3d(sB + sb * kBBytes, &tmC, fullB + 8 * sb, kb * kBK, c0, 0);
          for (int i = 0; i < kDig; ++i, ++ga) {
            const int sa = ga % kASlots;
            if (ga >= kASlots && !mbar_wait(emptyA + 8 * sa, (ga / kASlots - 1) & 1, a.err, kWaitE)) {
              ok = false;
              break;
            }
            mbar_expect_tx(fullA + 8 * sa, kABytes);
            tma_load_3d(sA + sa * kABytes, &tmR, fullA + 8 * sa, kb * kBK, r0, i);
          }
        }
      }
      // every issued box must have landed before the CTA may exit
      for (int q = (ga > kASlots ? ga - kASlots : 0); q < ga; ++q)
        mbar_wait(fullA + 8 * (q % kASlots), (q / kASlots) & 1, a.err, kWaitE);
      for (int q = (gb > kBStages ? gb - kBStages : 0); q < gb; ++q)
        mbar_wait(fullB + 8 * (q % kBStages), (q / kBStages) & 1, a.err, kWaitE);
    }
  } else if (warp == 9) {
    // ---- MMA issuer: the whole warp follows the loop (uniform operand addresses), one elected
    // lane issues ----
    const uint32_t sB = smem_u32(smem), sA = sB + kBStages * kBBytes;
    int ga = 0, gb = 0, gc = 0;
    bool ok = true;
    auto wait_all = [&](uint32_t bar, int parity) {
      int okw = 1;
      if (lane == 0) okw = mbar_wait(bar, parity, a.err, kWaitE);
      return __shfl_sync(0xffffffffu, okw, 0) != 0;
    };
    for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
      const int kb0 = (t / tiles) * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
      for (int kc = kb0; kc < kb1 && ok; kc += kChunk, ++gc) {
        if (gc > 0 && !wait_all(tempty, (gc - 1) & 1)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int kend = min(kb1, kc + kChunk);
        for (int kb = kc; kb < kend && ok; ++kb, ++gb) {
          const int sb = gb % kBStages;
          if (!wait_all(fullB + 8 * sb, (gb / kBStages) & 1)) { ok = false; break; }
          const uint64_t db = sw128_desc(sB + sb * kBBytes);
#pragma unroll
          for (int i = 0; i < kDig; ++i, ++ga) {
            const int sa = ga % kASlots;
            if (!wait_all(fullA + 8 * sa, (ga / kASlots) & 1)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_lane()) {
              const uint64_t da = sw128_desc(sA + sa * kABytes);
              const uint32_t d = tmem + (uint32_t)(kBC * i);
              const int n = kBC * (kDig - i);
              const uint32_t first = (i == 0 && kb == kc) ? 1u : 0u;
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk) {
                const uint64_t dk = (uint64_t)(2 * kk);   // 16 bf16 inside the swizzle atom
                const uint32_t acc = (first && kk == 0) ? 0u : 1u;
                mma_bf16(d, da + dk, db + dk, idesc_cols(n > 256 ? 256 : n), acc);
                if (n > 256)
                  mma_bf16(d + 256u, da + dk, db + dk + (uint64_t)(256 * 128 >> 4), idesc_cols(n - 256), acc);
              }
              mma_commit(emptyA + 8 * sa);
              if (i == kDig - 1) mma_commit(emptyB + 8 * sb);
            }
            __syncwarp();
          }
        }
        if (ok) {
          if (elect_lane()) mma_commit(tfull);
          __syncwarp();
        }
      }
    }
    if (elect_lane()) mma_commit(done);   // arrives once every issued MMA has completed
    __syncwarp();
  } else {
    // ---- epilogue ----
    const int q4 = warp & 3, half = warp >> 2;
    const uint32_t tl = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(32 * half);
    int gc = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < items && ok; t += gridDim.x) {
      const int tile = t % tiles, r0 = (tile % a.rt) * kBR, c0 = (tile / a.rt) * kBC + 32 * half;
      const int ksi = t / tiles, kb0 = ksi * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
      long long hi[32];
      uint32_t lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        hi[j] = 0;
        lo[j] = 0u;
      }
      for (int kc = kb0; kc < kb1; kc += kChunk, ++gc) {
        const bool okw = mbar_wait(tfull, gc & 1, a.err, 2 * kWaitE);
        if (!__all_sync(0xffffffffu, okw)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          uint32_t v[kDig][4];
#pragma unroll
          for (int l = 0; l < kDig; ++l) tmem_ld4(tl + (uint32_t)(kBC * l + 4 * g), v[l]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            long long s[kDig];
#pragma unroll
            for (int l = 0; l < kDig; ++l) s[l] = (long long)__float2int_rn(__uint_as_float(v[l][q]));
            const long long h = (s[0] << 24) + (s[1] << 16) + (s[2] << 8) + s[3];
            const long long w = (s[4] << 24) + (s[5] << 16) + (s[6] << 8) + s[7] + (long long)lo[4 * g + q];
            lo[4 * g + q] = (uint32_t)w;
            hi[4 * g + q] += h + (w >> 32);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(tempty);
      }
      if (!ok) break;
      const int r = r0 + 32 * q4 + lane;
      if (r < a.R) {
        const int er = __ldg(a.er + r);
        double* out = a.out + (int64_t)ksi * a.part;
        double prev = 0.0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int c = c0 + j;
          if (c < a.Cn) {
            const int ec = __ldg(a.ec + c);
            double x;
            if (er < kExpInf && ec < kExpInf) {
              // partial sums of a split contraction stay free of the rows' scales until they are
              // added, so none of them can underflow or overflow
              x = a.ks > 1 ? level_sum_to_f64(hi[j], lo[j], 1023, 1023) : level_sum_to_f64(hi[j], lo[j], er, ec);
            } else if (er == kExpNaN || ec == kExpNaN) {
              x = __longlong_as_double(0x7ff8000000000000ll);
            } else {
              // an infinity in a row: the products as the FP64 pipe forms them
              x = 0.0;
              const int k1 = min(a.K, kb1 * kBK);
              for (int k = kb0 * kBK; k < k1; ++k)
                x = fma(a.rsrc[(int64_t)r * a.ldr + k], a.csrc[(int64_t)c * a.ldcs + k], x);
            }
            if (a.alpha != 1.0) x *= a.alpha;
            if (a.swap) {
              double* p = out + (int64_t)r * a.ldc + c;
              if (a.beta != 0.0) {
                *p = fma(a.beta, *p, x);
              } else if (!a.vec2) {
                *p = x;
              } else if (j & 1) {
                *reinterpret_cast<double2*>(p - 1) = make_double2(prev, x);
              } else if (c + 1 >= a.Cn) {
                *p = x;
              }
              prev = x;
            } else {
              double* p = out + (int64_t)c * a.ldc + r;
              *p = a.beta != 0.0 ? fma(a.beta, *p, x) : x;
            }
          }
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(done, 0, a.err, kWaitE);   // no MMA may still write TMEM
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// x 2^k, rounded once
__device__ __forceinline__ double scale_pow2(double x, int k) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x), sign = bits & 0x8000000000000000ull;
  const int e = (int)((bits >> 52) & 0x7ffu);
  if (e == 0 || e == 0x7ff) return x;   // zero (the sums are never subnormal) or not finite
  const int ne = e + k;
  const uint64_t f = bits & 0xfffffffffffffull;
  if (ne >= 0x7ff) return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull));
  if (ne >= 1) return __longlong_as_double((long long)(sign | ((uint64_t)ne << 52) | f));
  const int sh = 1 - ne;
  const uint64_t m = f | 0x10000000000000ull;
  return __longlong_as_double((long long)(sign | (sh > 54 ? 0ull : (m + (1ull << (sh - 1))) >> sh)));
}

// out[n * ldc + m] = sum over the K ranges, in their order, of part[s][n][m] (dense, Md columns),
// with the scales of rows m and n (exponents ea, eb) put back
__global__ void k_sum_ranges(const double* __restrict__ part, int64_t stride, int ks, int Md, int64_t total,
                             const int* __restrict__ ea, const int* __restrict__ eb, double alpha, double beta,
                             double* __restrict__ out, int64_t ldc) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = e / Md;
    const int m = (int)(e - n * Md), sa = __ldg(ea + m), sb = __ldg(eb + n);
    double x = 0.0;
    for (int s = 0; s < ks; ++s) x += part[(int64_t)s * stride + e];
    if (sa < kExpInf && sb < kExpInf) x = scale_pow2(x, sa + sb - 2046);
    if (alpha != 1.0) x *= alpha;
    double* p = out + n * ldc + m;
    *p = beta != 0.0 ? fma(beta, *p, x) : x;
  }
}

// Digits of the rows of a float64 matrix: dig[j][r][k] (bf16, rows padded to rp, K to Kp with
// zeros) and the biased exponent of each row's largest element
// (below 1 for a subnormal row).  A warp per row: one pass for
// the exponent, one (from L1) for the digits.  Bytes, not flops, bound it: 8 read and 16
// written per element; the digits are formed on the integer and FP32 pipes (a byte under the
// exponent of 2^23 is the float 2^23 + byte).
__global__ void __launch_bounds__(256) k_digits(const double* __restrict__ in, int64_t ld, int rows, int K,
                                                int Kp, int64_t rp, int vec, __nv_bfloat16* __restrict__ dig,
                                                int* __restrict__ ex) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* row = in + (int64_t)r * ld;
  auto fetch = [&](int k, double (&x)[8]) {
    if (vec && k + 8 <= K) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double2 d = __ldg(reinterpret_cast<const double2*>(row + k) + q);
        x[2 * q] = d.x;
        x[2 * q + 1] = d.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = k + q < K ? __ldg(row + k + q) : 0.0;
    }
  };
  uint32_t mx = 0, nan = 0;
  for (int k = 8 * lane; k < K; k += 256) {
    double x[8];
    fetch(k, x);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint32_t h = (uint32_t)__double2hiint(x[q]) & 0x7fffffffu;
      mx = max(mx, h);
      nan |= h > 0x7ff00000u || (h == 0x7ff00000u && __double2loint(x[q]) != 0);
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx) >> 20;
  nan = __any_sync(0xffffffffu, nan);
  const bool special = mx == 0x7ffu;
  int em = (int)mx;
  if (mx == 0) {   // subnormal (or zero) row: its exponent continues below 1
    long long top = 0;
    for (int k = lane; k < K; k += 32)
      top = max(top, __double_as_longlong(__ldg(row + k)) & 0xfffffffffffffll);
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    em = top ? 12 - __clzll(top) : 1;
  }
  if (lane == 0) ex[r] = nan ? kExpNaN : special ? kExpInf : em;
  for (int k = 8 * lane; k < Kp; k += 256) {
    double x[8];
    fetch(k, x);
    uint32_t b[kDig][4];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      uint32_t w[2][2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const uint64_t bits = (uint64_t)__double_as_longlong(x[q + p]);
        const int e = (int)((bits >> 52) & 0x7ffu);
        uint64_t m = bits & 0xfffffffffffffull;
        if (e) m |= 0x10000000000000ull;
        const int sh = 9 - (em - (e ? e : 1));
        uint64_t y = sh >= 0 ? m << sh : (sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
        if (special) y = 0;
        if (bits >> 63) y = 0 - y;
        y += 0x8080808080808080ull;   // digit + 128 in every byte
        w[p][0] = (uint32_t)(y >> 32);
        w[p][1] = (uint32_t)y;
      }
#pragma unroll
      for (int j = 0; j < kDig; ++j) {
        const uint32_t sel = 0x7440u | (uint32_t)(3 - (j & 3));   // 0x4b, 0, 0, byte
        const float f0 = __uint_as_float(__byte_perm(w[0][j >> 2], 0x4b000000u, sel)) - 8388736.f;
        const float f1 = __uint_as_float(__byte_perm(w[1][j >> 2], 0x4b000000u, sel)) - 8388736.f;
        b[j][q >> 1] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632u);
      }
    }
#pragma unroll
    for (int j = 0; j < kDig; ++j)
      *reinterpret_cast<uint4*>(dig + ((int64_t)j * rp + r) * Kp + k) =
          make_uint4(b[j][0], b[j][1], b[j][2], b[j][3]);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_tiled_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// Digits of one operand in the workspace.
struct Digits {
  __nv_bfloat16* dig;
  int* ex;
  int64_t rp;
  int Kp;
};

int64_t pad128(int64_t r) { return (r + 127) / 128 * 128; }
size_t digit_bytes(int64_t rows, int K) {
  return (size_t)pad128(rows) * ((size_t)pad64(K) * 2 * kDig + sizeof(int));
}

Digits place(uint8_t* p, int64_t rows, int K) {
  Digits d;
  d.rp = pad128(rows);
  d.Kp = pad64(K);
  d.dig = reinterpret_cast<__nv_bfloat16*>(p);
  d.ex = reinterpret_cast<int*>(p + (size_t)d.rp * d.Kp * 2 * kDig);
  return d;
}

cudaError_t make_digits(const double* in, int64_t ld, int rows, int K, const Digits& d, cudaStream_t s) {
  const int vec = ld % 2 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
  k_digits<<<(rows + 7) / 8, 256, 0, s>>>(in, ld, rows, K, d.Kp, d.rp, vec, d.dig, d.ex);
  return cudaGetLastError();
}

cudaError_t digit_map(CUtensorMap* map, const Digits& d, int box_rows, int box_dig) {
  auto fn = encode_tiled_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {(cuuint64_t)d.Kp, (cuuint64_t)d.rp, (cuuint64_t)kDig};
  cuuint64_t strides[2] = {(cuuint64_t)d.Kp * 2, (cuuint64_t)d.rp * d.Kp * 2};
  cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, (cuuint32_t)box_dig};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, d.dig, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

constexpr int kSms = 152;
constexpr size_t kPartBytes = 64u << 20;   // room for the partial sums of a split contraction

// K ranges for `tiles` tiles of nkb K blocks: the split that minimises the waves' length, in
// cycles of one K block (4.8 k) and of an item's fixed part (6 k: pipeline fill, the last
// chunk's drain), with the partial sums' round trip (16 bytes per output and range).
int k_ranges(int64_t tiles, int nkb) {
  int best = 1;
  double bt = 1e300;
  for (int ks = 1; ks <= std::max(1, nkb / 2) && ks <= 64; ++ks) {
    if ((size_t)(tiles * kBR * kBC) * 8 * ks > kPartBytes && ks > 1) break;
    const int kbs = (nkb + ks - 1) / ks;
    if ((nkb + kbs - 1) / kbs != ks) continue;
    const double waves = std::ceil((double)(tiles * ks) / kSms);
    const double t = waves * (kbs * 4800.0 + (kbs + kChunk - 1) / kChunk * 2000.0 + 6000.0) +
                     (ks > 1 ? 8000.0 + (double)tiles * ks * kBR * kBC * 16.0 / 3000.0 : 0.0);
    if (t < bt * 0.98) {
      bt = t;
      best = ks;
    }
  }
  return best;
}

}  // namespace

// The digit form pays where its 3 launches and the tile padding cost less than the FP64 pipe's
// 1.1 TFLOP/s.  (4.1e6 products, M = 8 and 128 walkers, take 17 us on the pipe and two launches
// of at least 4 us more here; from 3e7 on the pipe needs 55 us and more.)
bool gemm_f64e_ok(int Md, int Nd, int Kd) {
  return Kd >= 32 && (double)Md * Nd * Kd >= 3.0e7;
}

size_t gemm_f64e_bytes(int64_t Md, int64_t Nd, int Kd, size_t col_cap) {
  return digit_bytes(Md, Kd) + std::min(digit_bytes(Nd, Kd), std::max(col_cap, digit_bytes(128, Kd))) +
         kPartBytes + 1024;
}

cudaError_t prepare_gemm_f64e() {
  static cudaError_t st = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, []() {
    st = cudaFuncSetAttribute(k_gemm_f64e, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemE);
  });
  return st;
}

// B goes through the workspace in chunks of rows when its digits do not fit beside A's.
// Returns cudaErrorMemoryAllocation, with nothing launched, when not even one 128-row chunk fits.
cudaError_t gemm_f64e(int Md, int Nd, int Kd, double alpha, const double* A, int64_t lda, const double* B,
                      int64_t ldb, double beta, double* C, int64_t ldc, const F64Ws& ws, cudaStream_t s) {
  const size_t ab = (digit_bytes(Md, Kd) + 255) / 256 * 256, wb = ws.bytes / 256 * 256;
  if (!ws.buf || wb < ab + kPartBytes + digit_bytes(128, Kd)) return cudaErrorMemoryAllocation;
  const size_t avail = wb - ab - kPartBytes;
  const int64_t fit = (int64_t)(avail / ((size_t)pad64(Kd) * 2 * kDig + sizeof(int))) / 128 * 128;
  if (fit < 128) return cudaErrorMemoryAllocation;
  const int64_t nch = (Nd + fit - 1) / fit;
  const int64_t rows_per = std::min<int64_t>(fit, pad128((Nd + nch - 1) / nch));
  const Digits da = place(ws.buf, Md, Kd);
  double* part = reinterpret_cast<double*>(ws.buf + wb - kPartBytes);
  cudaError_t e = make_digits(A, lda, Md, Kd, da, s);
  for (int64_t n0 = 0; n0 < Nd && e == cudaSuccess; n0 += rows_per) {
    const int nr = (int)std::min<int64_t>(rows_per, Nd - n0);
    const Digits db = place(ws.buf + ab, nr, Kd);
    if ((e = make_digits(B + n0 * ldb, ldb, nr, Kd, db, s)) != cudaSuccess) break;
    // the operand with less padding in 128-row tiles takes the rows of the MMA
    const int64_t t0 = ((int64_t)(Md + kBR - 1) / kBR) * ((nr + kBC - 1) / kBC);
    const int64_t t1 = ((int64_t)(nr + kBR - 1) / kBR) * ((Md + kBC - 1) / kBC);
    const int swap = t1 < t0;
    const Digits &dr = swap ? db : da, &dc = swap ? da : db;
    CUtensorMap mr, mc;
    if ((e = digit_map(&mr, dr, kBR, 1)) != cudaSuccess) break;
    if ((e = digit_map(&mc, dc, kBC, kDig)) != cudaSuccess) break;
    EArgs a{};
    a.R = swap ? nr : Md;
    a.Cn = swap ? Md : nr;
    a.rt = (a.R + kBR - 1) / kBR;
    a.ct = (a.Cn + kBC - 1) / kBC;
    a.nkb = dr.Kp / kBK;
    a.ks = k_ranges((int64_t)a.rt * a.ct, a.nkb);
    a.kbs = (a.nkb + a.ks - 1) / a.ks;
    a.swap = swap;
    double* Cn = C + n0 * ldc;
    if (a.ks > 1) {
      a.alpha = 1.0;
      a.beta = 0.0;
      a.out = part;
      a.ldc = Md;
      a.part = (int64_t)Md * nr;
    } else {
      a.alpha = alpha;
      a.beta = beta;
      a.out = Cn;
      a.ldc = ldc;
    }
    a.vec2 = a.ldc % 2 == 0 && a.part % 2 == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
    a.er = dr.ex;
    a.ec = dc.ex;
    a.rsrc = swap ? B + n0 * ldb : A;
    a.ldr = swap ? ldb : lda;
    a.csrc = swap ? A : B + n0 * ldb;
    a.ldcs = swap ? lda : ldb;
    a.K = Kd;
    a.err = ws.err;
    const int64_t items = (int64_t)a.rt * a.ct * a.ks;
    k_gemm_f64e<<<(int)std::min<int64_t>(items, kSms), kThreadsE, kSmemE, s>>>(mr, mc, a);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if (a.ks > 1) {
      const int64_t total = (int64_t)Md * nr;
      k_sum_ranges<<<(int)std::min<int64_t>((total + 255) / 256, kSms * 16), 256, 0, s>>>(
          part, a.part, a.ks, Md, total, da.ex, db.ex, alpha, beta, Cn, ldc);
      e = cudaGetLastError();
    }
  }
  return e;
}

}  // namespace afq
