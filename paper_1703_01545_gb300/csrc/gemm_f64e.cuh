// Device helpers of the digit form of float64 numbers (gemm_f64e.cu): x 2^(62-E) as a 62-bit
// integer in 8 balanced base-256 digits, BF16 each, E the exponent of the row's largest element.
#pragma once
#include <cstdint>

namespace afq {
namespace dig {

constexpr int kDig = 8;                        // digits per element
constexpr int kExpNaN = 4095, kExpInf = 4094;  // exponent marks of rows with NaN / infinities

// Largest element so far of a row, as the high word of its magnitude, and whether a NaN was seen.
__device__ __forceinline__ void row_scan(double x, uint32_t& mx, uint32_t& nan) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  mx = max(mx, h);
  nan |= h > 0x7ff00000u || (h == 0x7ff00000u && __double2loint(x) != 0);
}

// The 8 digits + 128, most significant first in the bytes of hi, then lo, for a row whose largest
// element has the biased exponent em (below 1: subnormal); all zero digits with `zero`.
__device__ __forceinline__ void digit_bytes_of(double x, int em, bool zero, uint32_t& hi, uint32_t& lo) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ffu);
  uint64_t m = bits & 0xfffffffffffffull;
  if (e) m |= 0x10000000000000ull;
  const int sh = 9 - (em - (e ? e : 1));
  uint64_t y = sh >= 0 ? m << sh : (sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
  if (zero) y = 0;
  if (bits >> 63) y = 0 - y;
  y += 0x8080808080808080ull;   // digit + 128 in every byte
  hi = (uint32_t)(y >> 32);
  lo = (uint32_t)y;
}

// Digit j of two elements as a BF16 pair (the first in the low half); hi / lo as above.  A byte
// under the exponent of 2^23 is the float 2^23 + byte, and a digit has at most 8 bits.
__device__ __forceinline__ uint32_t digit_pair(int j, const uint32_t (&a)[2], const uint32_t (&b)[2]) {
  const uint32_t sel = 0x7440u | (uint32_t)(3 - (j & 3));   // 0x4b, 0, 0, byte
  const float f0 = __uint_as_float(__byte_perm(a[j >> 2], 0x4b000000u, sel)) - 8388736.f;
  const float f1 = __uint_as_float(__byte_perm(b[j >> 2], 0x4b000000u, sel)) - 8388736.f;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632u);
}

// Exponent of a row from the warp's scans, and its mark for the contraction.  A row of
// subnormals needs its largest fraction: `top` gives this lane's share when it is asked for.
template <class F>
__device__ __forceinline__ int row_exponent(uint32_t mx, uint32_t nan, int& mark, F top) {
  mx = __reduce_max_sync(0xffffffffu, mx) >> 20;
  nan = __any_sync(0xffffffffu, nan);
  int em = (int)mx;
  if (mx == 0) {
    long long t = top();
    for (int o = 16; o > 0; o >>= 1) t = max(t, __shfl_xor_sync(0xffffffffu, t, o));
    em = t ? 12 - __clzll(t) : 1;
  }
  mark = nan ? kExpNaN : mx == 0x7ffu ? kExpInf : em;
  return em;
}

__device__ __forceinline__ long long fraction_of(double x) {
  return __double_as_longlong(x) & 0xfffffffffffffll;
}

// Rows r0 .. of a batch element as digits, K strided in memory: a CTA per batch element and 32 rows,
// element (row, k) from f.at(z, row, k), which is contiguous in the row.  The first pass takes the
// rows' exponents, the second cuts 64 k x 32 rows at a time through shared memory (32 warps, as a
// single batch element has few rows and a long K).  `quarter`: pairs
// (k even: re, odd: im) give a second set of rows, rows2 further on, with (-im, re).
template <class F>
__global__ void __launch_bounds__(1024) k_strided_digits(const F f, int rows, int K, int Kp, int64_t rp, int rz,
                                                        int rows2, uint16_t* __restrict__ out,
                                                        int* __restrict__ ex) {
  __shared__ double tile[32][65];
  __shared__ uint32_t smx[32][32], snan[32][32];
  __shared__ long long sfr[32][32];
  __shared__ int sem[32], smark[32];
  const int z = blockIdx.x, r0 = blockIdx.y * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = r0 + lane;
  uint32_t mx = 0, nan = 0;
  long long fr = 0;
  for (int k = warp; k < K; k += 32) {
    const double x = row < rows ? f.at(z, row, k) : 0.0;
    row_scan(x, mx, nan);
    fr = max(fr, fraction_of(x));
  }
  smx[warp][lane] = mx;
  snan[warp][lane] = nan;
  sfr[warp][lane] = fr;
  __syncthreads();
  if (warp == 0) {
    for (int w = 1; w < 32; ++w) {
      mx = max(mx, smx[w][lane]);
      nan |= snan[w][lane];
      fr = max(fr, sfr[w][lane]);
    }
    mx >>= 20;
    // (the largest fraction is the row's largest element only in a subnormal row)
    const int em = mx ? (int)mx : fr ? 12 - __clzll(fr) : 1;
    const int mark = nan ? kExpNaN : mx == 0x7ffu ? kExpInf : em;
    sem[lane] = em;
    smark[lane] = mark;
    if (row < rows) {
      ex[(int64_t)z * rz + row] = mark;
      if (rows2) ex[(int64_t)z * rz + rows2 + row] = mark;
    }
  }
  for (int k0 = 0; k0 < Kp; k0 += 64) {
    __syncthreads();
    for (int k = warp; k < 64; k += 32)
      tile[lane][k] = row < rows && k0 + k < K ? f.at(z, row, k0 + k) : 0.0;
    __syncthreads();
    const int q = warp;
    if (r0 + q < rows) {
      uint32_t a[2], b[2];
      digit_bytes_of(tile[q][2 * lane], sem[q], smark[q] >= kExpInf, a[0], a[1]);
      digit_bytes_of(tile[q][2 * lane + 1], sem[q], smark[q] >= kExpInf, b[0], b[1]);
      const int64_t o = ((int64_t)z * rz + r0 + q) * Kp + k0 + 2 * lane;
#pragma unroll
      for (int j = 0; j < kDig; ++j) {
        const uint32_t d = digit_pair(j, a, b);
        *reinterpret_cast<uint32_t*>(out + (int64_t)j * rp * Kp + o) = d;
        if (rows2)
          *reinterpret_cast<uint32_t*>(out + (int64_t)j * rp * Kp + o + (int64_t)rows2 * Kp) =
              __byte_perm(d, d, 0x1032u) ^ 0x00008000u;
      }
    }
  }
}

}  // namespace dig
}  // namespace afq
