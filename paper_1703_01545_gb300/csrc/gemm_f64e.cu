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
//   Sum.  V = sum_l S_l 2^(48-8l) is accumulated over the chunks as a 96-bit integer and
//   rounded once to float64: no operation touches the FP64 pipe.
// The result carries the rounding of the operands to 62 bits of their row maximum and one final
// rounding, where the multiply-add chain of the SIMT kernel rounds K times.
//
// A_i meets B_0 .. B_(7-i), whose products belong to the levels i .. 7: with the digits of B as
// consecutive 64-row blocks of one shared-memory tile and the levels as consecutive 64-column
// blocks of tensor memory, that is one contiguous window, so a K step of 16 takes 12 MMAs (N up
// to 256) for the 36 products.
//
// One CTA per SM, persistent over (batch, 128 x CN tile, K range) items.  CN = 64: all 512 TMEM
// columns hold the 8 levels of one tile; 16 and 32 (narrow batched products) leave room for two
// tiles, so the sums of one are taken while the next one's MMAs run.
//   warp 16  TMA producer: the 8 digits of a CN-row, 64-wide B block in one box (2 stages), the
//            digits of A as 16 KB boxes (6 slots or more)
//   warp 17  MMA issuer
//   warps 0..15  epilogue: a thread holds one row and CN / 4 columns; per chunk it reads the 8
//            levels and adds them to its 96-bit sums, after the item's last chunk it rounds and
//            stores while the next item's MMAs run.  The rounding is free of branches, so that
//            four columns' chains of dependent integer instructions overlap (with 8 warps and a
//            branch per column a 128 x 64 tile took 62 k cycles)
// Bounds of a 128 x 64 tile and 16 k: 1184 cycles of MMA (of which 32 for windows whose operand
// reads outlast their products), and 49 KB of digits from L2, 42 bytes per clock and SM.
// Measured (GB300, relative 2-norm error against exact rational arithmetic in brackets): the
// contractions of the reverse-mode run at M = 96, X = 480, 128 walkers, 10 steps, 223 ms on the
// FP64 pipe [2.6e-16 .. 1.1e-15 for a float64 multiply-add chain], 9.0 ms here with the digits
// and partial sums [4.3e-17 .. 1.2e-16].  V_HS at M = 64, X = 320, 2048 walkers: 4.47 -> 0.17 ms.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "gemm_f64e.cuh"
#include "internal.h"
#include "tc_device.cuh"

namespace afq {
namespace {

using namespace tc;
using namespace dig;

constexpr int kBR = 128, kBK = 64;             // tile rows, K block
constexpr int kChunk = 4;                      // K blocks per exact chunk (256 k)
constexpr int kABytes = kBR * kBK * 2;
constexpr int kEpiWarps = 16, kEpi = 32 * kEpiWarps, kThreadsE = kEpi + 64;
// CN: tile columns (16, 32, 48 or 64)
template <int CN>
struct ELay {
  static constexpr int kBStages = 2, kBBytes = kDig * CN * kBK * 2;
  static constexpr int kASlots = CN == 64 ? 6 : CN == 48 ? 8 : 9;
  static constexpr int kTBufs = CN <= 32 ? 2 : 1;   // TMEM tiles of 8 CN columns
  static constexpr int kBarOff = kBStages * kBBytes + kASlots * kABytes;
  static constexpr int kSmem = kBarOff + 256 + 1024;
  static_assert(kSmem <= 227 * 1024, "shared memory of a CTA");
};
constexpr uint64_t kWaitE = 2000000000ull;

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

// V = hi 2^32 + lo (96-bit two's complement) as float64, scaled so that a = b = 1 with one k gives
// V = 2^58 and ea = eb = 1023 (biased exponents of the row maxima).  One rounding, to nearest, and no
// branch; `ok` is cleared when the result is not a normal number (nor an exact zero).
__device__ __forceinline__ double level_sum_fast(long long hi, uint32_t lo, int ea, int eb, bool& ok) {
  uint32_t w2 = (uint32_t)((uint64_t)hi >> 32), w1 = (uint32_t)hi, w0 = lo;
  const uint32_t s = (uint32_t)((int)w2 >> 31);   // all ones for a negative V
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %6;\n\tsubc.u32 %2, %5, %6;"
      : "=r"(w0), "=r"(w1), "=r"(w2)
      : "r"(w0 ^ s), "r"(w1 ^ s), "r"(w2 ^ s), "r"(s));
  // the first word that is not zero to the front, then its leading bit to bit 31
  const bool z2 = w2 == 0u, z1 = z2 && w1 == 0u;
  const uint32_t a = z1 ? w0 : z2 ? w1 : w2, b = z1 ? 0u : z2 ? w0 : w1, c = z2 ? 0u : w0;
  const int sh = __clz((int)a) & 31, n = sh + (z1 ? 64 : z2 ? 32 : 0);
  const uint32_t t1 = __funnelshift_l(b, a, sh), t0 = __funnelshift_l(c, b, sh);
  const int be1 = ea + eb - 987 - n;   // biased exponent, less the implicit bit's one
  ok = ok && (a == 0u || (be1 >= 0 && be1 < 2045));
  uint32_t rl = __funnelshift_r(t0, t1, 11), rh = (t1 >> 11) + ((uint32_t)be1 << 20);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(rl), "+r"(rh) : "r"((t0 >> 10) & 1u));
  rh |= s & 0x80000000u;
  return a == 0u ? 0.0 : __hiloint2double((int)rh, (int)rl);
}

// The same for every V and exponent: subnormal results and overflow too.
__device__ __noinline__ double level_sum_any(long long hi, uint32_t lo, int ea, int eb) {
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
  const int be1 = ea + eb - 987 - n;
  uint64_t r;   // its magnitude's bits: m carries the implicit bit into the exponent field
  if (be1 >= 0) {
    r = be1 > 2045 ? 0x7ff0000000000000ull : ((uint64_t)be1 << 52) + m;
    if (r > 0x7ff0000000000000ull) r = 0x7ff0000000000000ull;
  } else {      // subnormal
    r = be1 < -54 ? 0ull : (m + (1ull << (-be1 - 1))) >> -be1;
  }
  return __longlong_as_double((long long)(r | ((uint64_t)neg << 63)));
}

struct EArgs {
  int R, Cn;               // valid rows and columns (of one batch element)
  int rt, ct, nz, ks;      // row tiles, column tiles, batch, K ranges
  int rz, cz;              // digit rows from one batch element to the next, both operands
  int nkb, kbs;            // K blocks in all, per range
  int swap;                // 0: out[c * ldc + r]; 1: out[r * ldc + c]
  int vec2;                // swap: pairs of columns may be stored as 16 bytes
  int scaled, added;       // alpha is not 1, beta is not 0 (setup and derivatives only)
  double alpha, beta;
  double* out;
  int64_t ldc, outz;       // column stride, batch stride
  int64_t part;            // ks > 1: doubles per K range of the partial sums
  const int *er, *ec;      // row exponents of both operands
  const double *rsrc, *csrc;   // the operands themselves for rows with infinities, or null: NaN
  int64_t ldr, ldcs;
  int K;
  int* err;
};

template <int CN>
__global__ void __launch_bounds__(kThreadsE, 1)
    k_gemm_f64e(const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmC, const EArgs a) {
  using Lay = ELay<CN>;
  constexpr int kASlots = Lay::kASlots, kBStages = Lay::kBStages, kTBufs = Lay::kTBufs;
  constexpr int CH = CN / 4;   // columns of one epilogue thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Lay::kBarOff);
  const uint32_t fullA = smem_u32(bars), emptyA = fullA + 8 * kASlots;
  const uint32_t fullB = emptyA + 8 * kASlots, emptyB = fullB + 8 * kBStages;
  const uint32_t tfull = emptyB + 8 * kBStages, tempty = tfull + 8 * kTBufs, done = tempty + 8 * kTBufs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kASlots + 2 * kBStages + 2 * kTBufs + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles = a.rt * a.ct, work = tiles * a.nz, items = work * a.ks;
  // Item n of this CTA.  One K block (sticky): a run of consecutive items, columns fastest, so that
  // the 8 digit tiles of a row tile are loaded once for all its columns (fresh: the first of them).
  // Longer contractions: row tiles fastest over the CTAs, which then share the column tiles in L2.
  const bool sticky = a.nkb == 1;
  const int first_item = sticky ? (int)((int64_t)items * blockIdx.x / gridDim.x) : blockIdx.x;
  const int last_item = sticky ? (int)((int64_t)items * (blockIdx.x + 1) / gridDim.x) : items;
  const int step_item = sticky ? 1 : gridDim.x;
  auto place_of = [&](int t, int& ksi, int& z, int& rtile, int& ctile) {
    ksi = t / work;
    z = (t - ksi * work) / tiles;
    const int tile = t % tiles;
    rtile = sticky ? tile / a.ct : tile % a.rt;
    ctile = sticky ? tile % a.ct : tile / a.rt;
  };

  if (threadIdx.x == 0) {
    for (int q = 0; q < kASlots; ++q) {
      mbar_init(fullA + 8 * q, 1);
      mbar_init(emptyA + 8 * q, 1);
    }
    for (int q = 0; q < kBStages; ++q) {
      mbar_init(fullB + 8 * q, 1);
      mbar_init(emptyB + 8 * q, 1);
    }
    for (int q = 0; q < kTBufs; ++q) {
      mbar_init(tfull + 8 * q, 1);
      mbar_init(tempty + 8 * q, kEpi);
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

  if (warp == kEpiWarps) {
    if (lane == 0) {
      // ---- TMA producer ----
      const uint32_t sB = smem_u32(smem), sA = sB + kBStages * Lay::kBBytes;
      int ga = 0, gb = 0;
      bool ok = true;
      for (int t = first_item; t < last_item && ok; t += step_item) {
        int ksi, z, rtile, ctile;
        place_of(t, ksi, z, rtile, ctile);
        const int r0 = z * a.rz + rtile * kBR, c0 = z * a.cz + ctile * CN;
        const bool fresh = !sticky || t == first_item || ctile == 0;
        const int kb0 = ksi * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
        for (int kb = kb0; kb < kb1 && ok; ++kb, ++gb) {
          const int sb = gb % kBStages;
          if (gb >= kBStages && !mbar_wait(emptyB + 8 * sb, (gb / kBStages - 1) & 1, a.err, kWaitE)) {
            ok = false;
            break;
          }
          mbar_expect_tx(fullB + 8 * sb, Lay::kBBytes);
          tma_load_3d(sB + sb * Lay::kBBytes, &tmC, fullB + 8 * sb, kb * kBK, c0, 0);
          for (int i = 0; i < kDig && fresh; ++i, ++ga) {
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
  } else if (warp == kEpiWarps + 1) {
    // ---- MMA issuer: the whole warp follows the loop (uniform operand addresses), one elected
    // lane issues ----
    const uint32_t sB = smem_u32(smem), sA = sB + kBStages * Lay::kBBytes;
    int ga = 0, gb = 0, gc = 0;
    bool ok = true;
    auto wait_all = [&](uint32_t bar, int parity) {
      int okw = 1;
      if (lane == 0) okw = mbar_wait(bar, parity, a.err, kWaitE);
      return __shfl_sync(0xffffffffu, okw, 0) != 0;
    };
    for (int t = first_item; t < last_item && ok; t += step_item) {
      int ksi, z, rtile, ctile;
      place_of(t, ksi, z, rtile, ctile);
      const int kb0 = ksi * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
      const bool fresh = !sticky || t == first_item || ctile == 0;
      const bool release = !sticky || t + 1 == last_item || ctile + 1 == a.ct;   // the row tile's last use
      if (!fresh) ga -= kDig;   // the slots of the previous item again
      for (int kc = kb0; kc < kb1 && ok; kc += kChunk, ++gc) {
        const int tb = gc % kTBufs;
        if (gc >= kTBufs && !wait_all(tempty + 8 * tb, (gc / kTBufs - 1) & 1)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int kend = min(kb1, kc + kChunk);
        for (int kb = kc; kb < kend && ok; ++kb, ++gb) {
          const int sb = gb % kBStages;
          if (!wait_all(fullB + 8 * sb, (gb / kBStages) & 1)) { ok = false; break; }
          const uint64_t db = sw128_desc(sB + sb * Lay::kBBytes);
#pragma unroll
          for (int i = 0; i < kDig; ++i, ++ga) {
            const int sa = ga % kASlots;
            if (fresh && !wait_all(fullA + 8 * sa, (ga / kASlots) & 1)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_lane()) {
              const uint64_t da = sw128_desc(sA + sa * kABytes);
              const uint32_t d = tmem + (uint32_t)(tb * kDig * CN + CN * i);
              const int n = CN * (kDig - i);
              const uint32_t first = (i == 0 && kb == kc) ? 1u : 0u;
#pragma unroll
              for (int kk = 0; kk < kBK / 16; ++kk) {
                const uint64_t dk = (uint64_t)(2 * kk);   // 16 bf16 inside the swizzle atom
                const uint32_t acc = (first && kk == 0) ? 0u : 1u;
                mma_bf16(d, da + dk, db + dk, idesc_cols(n > 256 ? 256 : n), acc);
                if (n > 256)
                  mma_bf16(d + 256u, da + dk, db + dk + (uint64_t)(256 * 128 >> 4), idesc_cols(n - 256), acc);
              }
              if (release) mma_commit(emptyA + 8 * sa);
              if (i == kDig - 1) mma_commit(emptyB + 8 * sb);
            }
            __syncwarp();
          }
        }
        if (ok) {
          if (elect_lane()) mma_commit(tfull + 8 * tb);
          __syncwarp();
        }
      }
    }
    if (elect_lane()) mma_commit(done);   // arrives once every issued MMA has completed
    __syncwarp();
  } else {
    // ---- epilogue ----
    const int q4 = warp & 3, part = warp >> 2;
    const uint32_t tl = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(CH * part);
    int gc = 0;
    bool ok = true;
    for (int t = first_item; t < last_item && ok; t += step_item) {
      int ksi, z, rtile, ctile;
      place_of(t, ksi, z, rtile, ctile);
      const int r0 = rtile * kBR, c0 = ctile * CN + CH * part;
      const int kb0 = ksi * a.kbs, kb1 = min(a.nkb, kb0 + a.kbs);
      long long hi[CH];
      uint32_t lo[CH];
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        hi[j] = 0;
        lo[j] = 0u;
      }
      for (int kc = kb0; kc < kb1; kc += kChunk, ++gc) {
        const int tb = gc % kTBufs;
        const bool okw = mbar_wait(tfull + 8 * tb, (gc / kTBufs) & 1, a.err, 2 * kWaitE);
        if (!__all_sync(0xffffffffu, okw)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int g = 0; g < CH / 4; ++g) {
          uint32_t v[kDig][4];
#pragma unroll
          for (int l = 0; l < kDig; ++l)
            tmem_ld4(tl + (uint32_t)(tb * kDig * CN + CN * l + 4 * g), v[l]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // |S_0|, |S_1| <= 2^22: integers by the exponent of 2^23; S_6 + 2^-8 S_7 rounded to an
            // integer (2^-60 of the row maxima's product); conversions for the rest
            const int s0 = (int)__float_as_uint(__uint_as_float(v[0][q]) + 12582912.f) - 0x4b400000;
            const int s1 = (int)__float_as_uint(__uint_as_float(v[1][q]) + 12582912.f) - 0x4b400000;
            const int s2 = __float2int_rn(__uint_as_float(v[2][q])), s3 = __float2int_rn(__uint_as_float(v[3][q]));
            const int s4 = __float2int_rn(__uint_as_float(v[4][q])), s5 = __float2int_rn(__uint_as_float(v[5][q]));
            const int s6 = __float2int_rn(fmaf(__uint_as_float(v[7][q]), 0x1p-8f, __uint_as_float(v[6][q])));
            const long long h = (long long)(s0 * 256 + s1) * 256 + s2;
            const long long w = ((long long)s3 * 256 + s4) * 65536 + ((long long)s5 * 256 + s6) +
                                (long long)lo[4 * g + q];
            lo[4 * g + q] = (uint32_t)w;
            hi[4 * g + q] += h + (w >> 32);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(tempty + 8 * tb);
      }
      if (!ok) break;
      const int r = r0 + 32 * q4 + lane;
      if (r < a.R) {
        const int er0 = __ldg(a.er + (int64_t)z * a.rz + r);
        // partial sums of a split contraction stay free of the rows' scales until they are added,
        // so none of them can underflow or overflow
        const int er = a.ks > 1 && er0 < kExpInf ? 1023 : er0;
        double* out = a.out + (int64_t)ksi * a.part + (int64_t)z * a.outz;
#pragma unroll
        for (int g = 0; g < CH / 4; ++g) {
          const int c = c0 + 4 * g;
          double x[4];
          int ec[4];
          bool ok4 = er0 < kExpInf && !a.scaled && !a.added;   // (a multiplication here would hold the FP64 pipe even unused)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            ec[q] = c + q < a.Cn ? __ldg(a.ec + (int64_t)z * a.cz + c + q) : 1023;
            ok4 = ok4 && ec[q] < kExpInf;
            if (a.ks > 1 && ec[q] < kExpInf) ec[q] = 1023;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = level_sum_fast(hi[4 * g + q], lo[4 * g + q], er, ec[q], ok4);
          if (!ok4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (er0 < kExpInf && ec[q] < kExpInf) {
                x[q] = level_sum_any(hi[4 * g + q], lo[4 * g + q], er, ec[q]);
              } else if (er0 == kExpNaN || ec[q] == kExpNaN || !a.rsrc) {
                x[q] = __longlong_as_double(0x7ff8000000000000ll);
              } else {
                // an infinity in a row: the products as the FP64 pipe forms them
                x[q] = 0.0;
                const int k1 = c + q < a.Cn ? min(a.K, kb1 * kBK) : 0;
                for (int k = kb0 * kBK; k < k1; ++k)
                  x[q] = fma(a.rsrc[(int64_t)r * a.ldr + k], a.csrc[(int64_t)(c + q) * a.ldcs + k], x[q]);
              }
              if (a.scaled) x[q] *= a.alpha;
              if (a.added && c + q < a.Cn)
                x[q] = fma(a.beta, a.swap ? out[(int64_t)r * a.ldc + c + q] : out[(int64_t)(c + q) * a.ldc + r], x[q]);
            }
          }
          if (a.swap) {
            double* p = out + (int64_t)r * a.ldc + c;
            if (a.vec2 && c + 4 <= a.Cn) {
              reinterpret_cast<double2*>(p)[0] = make_double2(x[0], x[1]);
              reinterpret_cast<double2*>(p)[1] = make_double2(x[2], x[3]);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (c + q < a.Cn) p[q] = x[q];
            }
          } else {
            double* p = out + (int64_t)c * a.ldc + r;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (c + q < a.Cn) p[q * a.ldc] = x[q];
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
// exponent of 2^23 is the float 2^23 + byte).  Row r is the source's row (r / grp) gstep + goff +
// r % grp: a spin's columns of every walker, or (grp = rows) consecutive rows.
__global__ void __launch_bounds__(256) k_digits(const double* __restrict__ in, int64_t ld, int rows, int grp,
                                                int64_t gstep, int goff, int K,
                                                int Kp, int64_t rp, int vec, __nv_bfloat16* __restrict__ dig,
                                                int* __restrict__ ex) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* row = in + ((int64_t)(r / grp) * gstep + goff + r % grp) * ld;
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
    for (int q = 0; q < 8; ++q) row_scan(x[q], mx, nan);
  }
  int mark;
  const int em = row_exponent(mx, nan, mark, [&]() {
    long long top = 0;
    for (int k = lane; k < K; k += 32) top = max(top, fraction_of(__ldg(row + k)));
    return top;
  });
  if (lane == 0) ex[r] = mark;
  for (int k = 8 * lane; k < Kp; k += 256) {
    double x[8];
    fetch(k, x);
    uint32_t b[kDig][4];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      uint32_t w0[2], w1[2];
      digit_bytes_of(x[q], em, mark >= kExpInf, w0[0], w0[1]);
      digit_bytes_of(x[q + 1], em, mark >= kExpInf, w1[0], w1[1]);
#pragma unroll
      for (int j = 0; j < kDig; ++j) b[j][q >> 1] = digit_pair(j, w0, w1);
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

constexpr int kSms = 152;
constexpr size_t kPartBytes = 64u << 20;   // room for the partial sums of a split contraction

// K ranges for `tiles` tiles of nkb K blocks: the split that minimises the waves' length, in
// cycles of one K block (4.8 k) and of an item's fixed part (6 k: pipeline fill, the last
// chunk's drain), with the partial sums' round trip (16 bytes per output and range).
int k_ranges(int64_t tiles, int nkb, size_t part_bytes) {
  int best = 1;
  double bt = 1e300;
  for (int ks = 1; ks <= std::max(1, nkb / 2) && ks <= 64; ++ks) {
    if ((size_t)(tiles * kBR * 64) * 8 * ks > part_bytes && ks > 1) break;
    const int kbs = (nkb + ks - 1) / ks;
    if ((nkb + kbs - 1) / kbs != ks) continue;
    const double waves = std::ceil((double)(tiles * ks) / kSms);
    const double t = waves * (kbs * 4800.0 + (kbs + kChunk - 1) / kChunk * 2000.0 + 6000.0) +
                     (ks > 1 ? 8000.0 + (double)tiles * ks * kBR * 64 * 16.0 / 3000.0 : 0.0);
    if (t < bt * 0.98) {
      bt = t;
      best = ks;
    }
  }
  return best;
}

cudaError_t digit_map(CUtensorMap* map, const DigitOp& d, int box_rows, int box_dig) {
  auto fn = encode_tiled_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {(cuuint64_t)d.Kp, (cuuint64_t)(d.rp - d.off), (cuuint64_t)kDig};
  cuuint64_t strides[2] = {(cuuint64_t)d.Kp * 2, (cuuint64_t)d.rp * d.Kp * 2};
  cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, (cuuint32_t)box_dig};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, d.dig, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int CN>
cudaError_t launch_cn(const CUtensorMap& mr, const CUtensorMap& mc, const EArgs& a, cudaStream_t s) {
  const int64_t items = (int64_t)a.rt * a.ct * a.nz * a.ks;
  if (items > 0x7fffffff) return cudaErrorInvalidConfiguration;
  k_gemm_f64e<CN><<<(int)std::min<int64_t>(items, kSms), kThreadsE, ELay<CN>::kSmem, s>>>(mr, mc, a);
  return cudaGetLastError();
}

int64_t pad128(int64_t r) { return (r + 127) / 128 * 128; }

}  // namespace

size_t digit_bytes(int64_t rows, int K) {
  return ((size_t)pad128(rows) * ((size_t)pad64(K) * 2 * kDig + sizeof(int)) + 255) / 256 * 256;
}

DigitOp digit_place(void* p, int64_t rows, int K) {
  DigitOp d;
  d.rp = pad128(rows);
  d.Kp = pad64(K);
  d.dig = static_cast<__nv_bfloat16*>(p);
  d.ex = reinterpret_cast<int*>(static_cast<uint8_t*>(p) + (size_t)d.rp * d.Kp * 2 * kDig);
  return d;
}

cudaError_t digits_of(const double* in, int64_t ld, int rows, int K, const DigitOp& d, cudaStream_t s, int grp,
                      int64_t gstep, int goff) {
  if (grp <= 0) grp = rows;
  const int vec = ld % 2 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
  k_digits<<<(rows + 7) / 8, 256, 0, s>>>(in, ld, rows, grp, gstep, goff, K, d.Kp, d.rp, vec, d.dig, d.ex);
  return cudaGetLastError();
}

// Columns per tile: the narrowest form that takes all columns at once.  More columns: with one K
// block 32 (two tiles in tensor memory: the sums of one, 7 k cycles of issue for 8192 outputs, run
// beside the 4.7 k cycles of MMAs of the other, and the row tile's digits stay in shared memory),
// else 64, whose operand reads (42 bytes per clock and SM against 65) serve the most products.
cudaError_t digit_gemm(const DigitOp& rows, const DigitOp& cols, const DigitGemm& g, cudaStream_t s) {
  if (rows.Kp != cols.Kp || g.R < 1 || g.Cn < 1 || g.nz < 1) return cudaErrorInvalidValue;
  const int cn = g.Cn <= 16 ? 16 : g.Cn <= 32 || rows.Kp == kBK ? 32 : g.Cn <= 48 ? 48 : 64;
  CUtensorMap mr, mc;
  cudaError_t e = digit_map(&mr, rows, kBR, 1);
  if (e == cudaSuccess) e = digit_map(&mc, cols, cn, kDig);
  if (e != cudaSuccess) return e;
  EArgs a{};
  a.R = g.R;
  a.Cn = g.Cn;
  a.rt = (g.R + kBR - 1) / kBR;
  a.ct = (g.Cn + cn - 1) / cn;
  a.nz = g.nz;
  a.rz = g.rz;
  a.cz = g.cz;
  a.nkb = rows.Kp / kBK;
  a.ks = std::max(1, g.ks);
  a.kbs = (a.nkb + a.ks - 1) / a.ks;
  a.swap = g.swap;
  a.alpha = g.alpha;
  a.beta = g.beta;
  a.out = g.out;
  a.ldc = g.ldc;
  a.outz = g.outz;
  a.part = g.part;
  a.scaled = g.alpha != 1.0;
  a.added = g.beta != 0.0;
  a.vec2 = g.ldc % 2 == 0 && g.outz % 2 == 0 && g.part % 2 == 0 && (reinterpret_cast<uintptr_t>(g.out) & 15) == 0;
  a.er = rows.ex;
  a.ec = cols.ex;
  a.rsrc = g.rsrc;
  a.ldr = g.ldr;
  a.csrc = g.csrc;
  a.ldcs = g.ldcs;
  a.K = g.K;
  a.err = g.err;
  switch (cn) {
    case 16: return launch_cn<16>(mr, mc, a, s);
    case 32: return launch_cn<32>(mr, mc, a, s);
    case 48: return launch_cn<48>(mr, mc, a, s);
    default: return launch_cn<64>(mr, mc, a, s);
  }
}

// digit_gemm of one batch element over as many K ranges as pay, their partial sums in `part`.
cudaError_t digit_gemm_sum(const DigitOp& rows, const DigitOp& cols, DigitGemm g, double* part, size_t part_bytes,
                           cudaStream_t s) {
  const int64_t tiles = ((int64_t)(g.R + kBR - 1) / kBR) * ((g.Cn + 63) / 64);
  g.ks = k_ranges(tiles, rows.Kp / kBK, part_bytes);
  if (g.ks <= 1) return digit_gemm(rows, cols, g, s);
  // the partial sums are dense, the operand whose index is contiguous in `out` innermost
  const int in = g.swap ? g.Cn : g.R, outer = g.swap ? g.R : g.Cn;
  DigitGemm q = g;
  q.alpha = 1.0;
  q.beta = 0.0;
  q.out = part;
  q.ldc = in;
  q.part = (int64_t)in * outer;
  cudaError_t e = digit_gemm(rows, cols, q, s);
  if (e != cudaSuccess) return e;
  const int64_t total = (int64_t)in * outer;
  k_sum_ranges<<<(int)std::min<int64_t>((total + 255) / 256, kSms * 16), 256, 0, s>>>(
      part, q.part, g.ks, in, total, g.swap ? cols.ex : rows.ex, g.swap ? rows.ex : cols.ex, g.alpha, g.beta, g.out,
      g.ldc);
  return cudaGetLastError();
}

// The digit form pays where its launches (about 12 us in all) and its 36 products of the padded
// operands (1.2 PFLOP/s) take less than the FP64 pipe's 1.1 TFLOP/s.  At M = 8 and 128 walkers the
// pipe's 17 us win; from 3e7 products on it needs 55 us and more.
bool gemm_f64e_ok(int Md, int Nd, int Kd) {
  const double pad = (double)((Md + 63) / 64 * 64) * ((Nd + 63) / 64 * 64) * pad64(Kd);
  return 2.0 * Md * Nd * Kd / 1.1e6 > 1.3 * (12.0 + 2.0 * 36.0 * pad / 1.2e9);
}

size_t gemm_f64e_bytes(int64_t Md, int64_t Nd, int Kd, size_t col_cap) {
  return digit_bytes(Md, Kd) + std::min(digit_bytes(Nd, Kd), std::max(col_cap, digit_bytes(128, Kd))) +
         kPartBytes + 1024;
}

cudaError_t prepare_gemm_f64e() {
  static SmemLimits limits;   // per device: a handle of another device raises its own
  auto raise = [&](int slot, auto k, int bytes) {
    return limits.raise(slot, (size_t)bytes, [&] {
      return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    });
  };
  cudaError_t e = raise(0, k_gemm_f64e<16>, ELay<16>::kSmem);
  if (e == cudaSuccess) e = raise(1, k_gemm_f64e<32>, ELay<32>::kSmem);
  if (e == cudaSuccess) e = raise(2, k_gemm_f64e<48>, ELay<48>::kSmem);
  if (e == cudaSuccess) e = raise(3, k_gemm_f64e<64>, ELay<64>::kSmem);
  return e;
}

// B goes through the workspace in chunks of rows when its digits do not fit beside A's.
// Returns cudaErrorMemoryAllocation, with nothing launched, when not even one 128-row chunk fits.
cudaError_t gemm_f64e(int Md, int Nd, int Kd, double alpha, const double* A, int64_t lda, const double* B,
                      int64_t ldb, double beta, double* C, int64_t ldc, const F64Ws& ws, cudaStream_t s) {
  const size_t ab = digit_bytes(Md, Kd), wb = ws.bytes / 256 * 256;
  if (!ws.buf || wb < ab + kPartBytes + digit_bytes(128, Kd)) return cudaErrorMemoryAllocation;
  const size_t avail = wb - ab - kPartBytes;
  const int64_t fit = (int64_t)(avail / ((size_t)pad64(Kd) * 2 * kDig + sizeof(int))) / 128 * 128;
  if (fit < 128) return cudaErrorMemoryAllocation;
  const int64_t nch = (Nd + fit - 1) / fit;
  const int64_t rows_per = std::min<int64_t>(fit, pad128((Nd + nch - 1) / nch));
  const DigitOp da = digit_place(ws.buf, Md, Kd);
  double* part = reinterpret_cast<double*>(ws.buf + wb - kPartBytes);
  cudaError_t e = digits_of(A, lda, Md, Kd, da, s);
  for (int64_t n0 = 0; n0 < Nd && e == cudaSuccess; n0 += rows_per) {
    const int nr = (int)std::min<int64_t>(rows_per, Nd - n0);
    const DigitOp db = digit_place(ws.buf + ab, nr, Kd);
    if ((e = digits_of(B + n0 * ldb, ldb, nr, Kd, db, s)) != cudaSuccess) break;
    // the operand with less padding in 128-row tiles takes the rows of the MMA
    const int64_t t0 = ((int64_t)(Md + kBR - 1) / kBR) * ((nr + 63) / 64);
    const int64_t t1 = ((int64_t)(nr + kBR - 1) / kBR) * ((Md + 63) / 64);
    double* Cn = C + n0 * ldc;
    DigitGemm g;
    g.swap = t1 < t0;
    g.R = g.swap ? nr : Md;
    g.Cn = g.swap ? Md : nr;
    g.alpha = alpha;
    g.beta = beta;
    g.out = Cn;
    g.ldc = ldc;
    g.rsrc = g.swap ? B + n0 * ldb : A;
    g.ldr = g.swap ? ldb : lda;
    g.csrc = g.swap ? A : B + n0 * ldb;
    g.ldcs = g.swap ? lda : ldb;
    g.K = Kd;
    g.err = ws.err;
    e = digit_gemm_sum(g.swap ? db : da, g.swap ? da : db, g, part, kPartBytes, s);
  }
  return e;
}

}  // namespace afq
