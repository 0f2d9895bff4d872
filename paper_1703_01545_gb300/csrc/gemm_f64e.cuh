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

}  // namespace dig
}  // namespace afq
