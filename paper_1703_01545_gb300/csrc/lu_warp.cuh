// LU factorisation of one small complex block by the lanes of a warp.
#pragma once
#include <cstdint>

namespace afq {
namespace {

// Scalar-type details of the LU: the integer magnitude key of a component (the high word of
// |x|, monotone in |x|) and its bounds (below: zero or subnormal, above: non-finite), the
// biased exponent, the exact power of two 2^(bias - e), and a reciprocal.
template <typename T> struct LuT;
template <> struct LuT<double> {
  static constexpr unsigned kMin = 0x00100000u, kInf = 0x7ff00000u;
  static constexpr int kMaxE = 2046;
  static __device__ __forceinline__ unsigned key(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
  static __device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
  static __device__ __forceinline__ double pow2(int eh) { return __hiloint2double((2046 - eh) << 20, 0); }
  static __device__ __forceinline__ int bias() { return 1023; }
  static __device__ __forceinline__ double rcp(double x) { return __drcp_rn(x); }
  static __device__ __forceinline__ double fm(double a, double b, double c) { return fma(a, b, c); }
};
template <> struct LuT<float> {
  static constexpr unsigned kMin = 0x00800000u, kInf = 0x7f800000u;
  static constexpr int kMaxE = 254;
  static __device__ __forceinline__ unsigned key(float x) { return __float_as_uint(x) & 0x7fffffffu; }
  static __device__ __forceinline__ int expo(float x) { return (int)((__float_as_uint(x) >> 23) & 0xffu); }
  static __device__ __forceinline__ float pow2(int eh) { return __uint_as_float((unsigned)(254 - eh) << 23); }
  static __device__ __forceinline__ int bias() { return 127; }
  static __device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }
  static __device__ __forceinline__ float fm(float a, float b, float c) { return fmaf(a, b, c); }
};

// LU factorisation with partial (row) pivoting of one spin block, P O = L U, in FP64 (or FP32,
// T = float) by W lanes of a warp (W = 16: both halves of the warp factorise one block each, in step; W = 32:
// one block per warp).  Pivot k interchanges whole rows, scales row k right of the diagonal by
// 1 / pivot (U is unit upper triangular), stores 1 / pivot on the diagonal and updates the
// trailing block; L, with the pivots as its diagonal, is left below the diagonal.  The pivots
// and the determinant are those of Gauss-Jordan elimination with the same pivoting.  Every
// FP64 warp instruction occupies the FP64 pipe whatever its active lanes, so the per-pivot
// scalar work is short and runs in all lanes: the pivot is chosen on an integer magnitude key
// (the high word of |re| or |im|, monotone in the magnitude), the determinant is the product
// of the pivots renormalised by an exact power of two built from its exponent bits, the row
// scale uses one reciprocal, and row blocks of the trailing update that no lane needs are
// skipped.  Each complex update is 4 FP64 fused multiply-adds.  Lane l owns column l % ns and
// rows l / ns + q (W / ns), q < Q.  kmax: the larger block of the warp (uniform loop bound).
template <int W, int Q, int LD, typename T = double>
__device__ __forceinline__ void lu_block(T* __restrict__ ar, T* __restrict__ ai, int l,
                                         int ns, int kmax, int* __restrict__ piv, T& dr,
                                         T& di, int& dexp, bool& bad) {
  using S = LuT<T>;
  const int nsd = ns > 0 ? ns : 1, RS = W / nsd;
  const int c = l % nsd, r0 = l / nsd;
  const bool active = ns > 0 && r0 < RS;
  dr = T(1);
  di = T(0);
  dexp = 0;
  bad = false;
  for (int k = 0; k < kmax; ++k) {
    const bool live = k < ns && !bad;
    unsigned key = 0u;
    if (live && l >= k && l < ns) {
      const unsigned hr = S::key(ar[l * LD + k]);
      const unsigned hi = S::key(ai[l * LD + k]);
      key = hr > hi ? hr : hi;
    }
    int p = l;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
      const unsigned ok = __shfl_xor_sync(0xffffffffu, key, o);
      const int op = __shfl_xor_sync(0xffffffffu, p, o);
      if (ok > key || (ok == key && op < p)) { key = ok; p = op; }
    }
    // zero, subnormal-only or non-finite column: singular for this kernel
    if (live && (key < S::kMin || key >= S::kInf)) bad = true;
    const bool go = live && !bad;
    if (go && l == 0) piv[k] = p;
    if (go && p != k && l < ns) {
      T t = ar[k * LD + l]; ar[k * LD + l] = ar[p * LD + l]; ar[p * LD + l] = t;
      t = ai[k * LD + l]; ai[k * LD + l] = ai[p * LD + l]; ai[p * LD + l] = t;
    }
    __syncwarp();
    const T vr = go ? ar[k * LD + k] : T(1), vi = go ? ai[k * LD + k] : T(0);
    {
      const T tr = S::fm(dr, vr, -di * vi);
      T ti = S::fm(dr, vi, di * vr);
      T trr = tr;
      if (go && p != k) { trr = -tr; ti = -ti; }
      if (go) { dr = trr; di = ti; }
      const int e1 = S::expo(dr), e2 = S::expo(di);
      const int eh = e1 > e2 ? e1 : e2;
      if (eh > 0 && eh < S::kMaxE) {
        const T sc = S::pow2(eh);   // 2^(bias - eh), exact
        dr *= sc;
        di *= sc;
        dexp += eh - S::bias();
      }
    }
    const T vv = S::fm(vr, vr, vi * vi);
    // FP64: a pivot whose square leaves the range counts as singular (or not finite) too
    if (sizeof(T) == 8 && go && !(vv > T(0) && S::key(vv) < S::kInf)) bad = true;
    const T rinv = S::rcp(vv);
    const T ir = vr * rinv, ii = -vi * rinv;          // 1 / pivot
    __syncwarp();
    if (go && l >= k && l < ns) {
      const T xr = ar[k * LD + l], xi = ai[k * LD + l];
      ar[k * LD + l] = (l == k) ? ir : S::fm(xr, ir, -xi * ii);
      ai[k * LD + l] = (l == k) ? ii : S::fm(xr, ii, xi * ir);
    }
    __syncwarp();
    // A[r][c] -= A[r][k] U[k][c] for r, c > k: column k and row k are not written, so no
    // synchronisation separates these reads from the update
    const bool colk = go && active && c > k;
    const int qf = colk ? max(0, (k + 1 - r0 + RS - 1) / RS) : Q;
    const int q0 = __reduce_min_sync(0xffffffffu, qf);
    const T kr = colk ? ar[k * LD + c] : T(0), ki = colk ? ai[k * LD + c] : T(0);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      if (q >= q0) {
        const int r = r0 + q * RS;
        if (colk && r < ns && r > k) {
          const T fr = ar[r * LD + k], fi = ai[r * LD + k];
          ar[r * LD + c] = S::fm(-fr, kr, S::fm(fi, ki, ar[r * LD + c]));
          ai[r * LD + c] = S::fm(-fr, ki, S::fm(-fi, kr, ai[r * LD + c]));
        }
      }
    }
    __syncwarp();
  }
}

}  // namespace
}  // namespace afq
