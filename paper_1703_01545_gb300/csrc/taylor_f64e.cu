// FP64 Taylor exponential sum_{m <= n} A^m Phi / m! of every walker with its products in digit form
// (gemm_f64e.cu): A is complex symmetric and differs from walker to walker, so a round is a batched
// contraction, one walker per batch element.
//
// Complex products as real ones, by what fills the 128 rows of an MMA:
//   M <= 64 (stacked rows)   [A_re; A_im] [T_re | T_im]: K = M, four real products, combined when
//                            the next term is formed
//   M > 64 (joined K)        [A_re | A_im] [T_re T_im; -T_im T_re]: K = 2 M2 (M2 = M rounded up to
//                            even), the real and imaginary columns of A T at once
// The terms are kept without their factorial, U_m = A U_(m-1), and Phi += U_m / m!, so that a round
// costs the FP64 pipe one multiply-add per real number (and one addition more for stacked rows).
//
// Walkers go in chunks whose digits (16 bytes per element of A) and products stay in L2 over the
// rounds: A is cut into digits once per chunk and read once per round.
//
// Measured at M = 64, 8/8, 2048 walkers, order 6: 5.73 ms in the FP64-pipe kernel (k_taylor, still
// taken for small populations), 1.03 ms here: products 0.61, terms 0.26, digits of A 0.16.  Bound by
// the products' operand reads (128 KB of digits of A per walker and round) and their epilogues.
#include <algorithm>
#include <cstdint>

#include "gemm_f64e.cuh"
#include "internal.h"

namespace afq {
namespace {

using namespace dig;

constexpr int kMaxM = 256;                         // a warp holds a term's column in registers
constexpr size_t kChunkBytes = (size_t)110 << 20;  // digits and products of a chunk: within L2

bool stacked(int M) { return M <= 64; }
int even(int M) { return (M + 1) / 2 * 2; }

struct Plan {
  int R, K, Cn;        // rows and K of a walker's A, columns
  int nw;              // walkers per chunk
  size_t per;          // bytes per walker: digits of A and of the term, products
};

Plan plan_of(int M, int N, int Nw) {
  Plan p;
  p.R = stacked(M) ? 2 * M : M;
  p.K = stacked(M) ? M : 2 * even(M);
  p.Cn = 2 * N;
  p.per = (size_t)(p.R + p.Cn) * ((size_t)pad64(p.K) * 2 * kDig + 4) + sizeof(double) * (size_t)p.R * p.Cn;
  // whole waves of tiles, as many as fit the chunk, one at least
  const int tiles = ((p.R + 127) / 128) * ((p.Cn + 63) / 64);
  const int wave = std::max(1, 152 / tiles);
  const int64_t fit = (int64_t)(kChunkBytes / p.per);
  p.nw = (int)std::min<int64_t>(Nw, std::max<int64_t>(wave, fit / wave * wave));
  const int nch = (Nw + p.nw - 1) / p.nw;
  if (p.nw > wave) p.nw = std::min(p.nw, std::max(wave, ((Nw + nch - 1) / nch + wave - 1) / wave * wave));
  p.nw = std::min(p.nw, Nw);
  return p;
}

// Digits of the rows of A from the packed upper triangles [2][Nw][P] of walkers w0 .. : a CTA per
// walker, a warp per row, lanes over pairs of k.  The row's part left of the diagonal is a column
// of the triangle; both parts come from L1, which holds a walker's planes (33 KB each at M = 64).
__global__ void __launch_bounds__(512) k_vhs_digits(const double* __restrict__ Ap, int64_t P, int M, int Nw, int w0,
                                                    int stack, int M2, int Kp, int64_t rp,
                                                    __nv_bfloat16* __restrict__ out, int* __restrict__ ex) {
  const int z = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rows = stack ? 2 * M : M;
  const double* re = Ap + (int64_t)(w0 + z) * P;
  const double* im = re + (int64_t)Nw * P;
  for (int r = warp; r < rows; r += 16) {
    const int i = r >= M ? r - M : r;
    const int64_t ri = (int64_t)i * (M - 1) - (int64_t)i * (i - 1) / 2;   // A[i][j] at ri + j, j >= i
    // element k of the row: plane and column j, zero beyond
    auto elem = [&](int k) -> double {
      const int p = stack ? (r >= M) : (k >= M2), j = stack ? k : (k >= M2 ? k - M2 : k);
      if (j >= M) return 0.0;
      const int64_t o = j >= i ? ri + j : (int64_t)j * (M - 1) - (int64_t)j * (j - 1) / 2 + i;
      return __ldg((p ? im : re) + o);
    };
    uint32_t mx = 0, nan = 0;
    for (int k = 2 * lane; k < Kp; k += 64) {
      row_scan(elem(k), mx, nan);
      row_scan(elem(k + 1), mx, nan);
    }
    int mark;
    const int em = row_exponent(mx, nan, mark, [&]() {
      long long t = 0;
      for (int k = lane; k < Kp; k += 32) t = max(t, fraction_of(elem(k)));
      return t;
    });
    const int64_t row = (int64_t)z * rows + r;
    if (lane == 0) ex[row] = mark;
    for (int k = 2 * lane; k < Kp; k += 64) {
      uint32_t a[2], b[2];
      digit_bytes_of(elem(k), em, mark >= kExpInf, a[0], a[1]);
      digit_bytes_of(elem(k + 1), em, mark >= kExpInf, b[0], b[1]);
#pragma unroll
      for (int j = 0; j < kDig; ++j)
        *reinterpret_cast<uint32_t*>(out + ((int64_t)j * rp + row) * Kp + k) = digit_pair(j, a, b);
    }
  }
}

// One term of walkers w0 .. : a warp per (walker, column n), lanes over pairs of orbitals.
// FIRST: U = Phi; else U = the round's products and Phi += coef U.  `more`: the digits of U as the
// next round's columns.
template <int NP, bool FIRST>
__global__ void __launch_bounds__(256) k_term(const double* __restrict__ prod, double* __restrict__ phi, int M, int N,
                                              int Nw, int w0, int nw, int stack, int M2, double coef, int more,
                                              int Kp, int64_t rp, __nv_bfloat16* __restrict__ out,
                                              int* __restrict__ ex) {
  const int task = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (task >= nw * N) return;
  const int z = task / N, n = task - z * N, R = stack ? 2 * M : M;
  const int64_t base = ((int64_t)(w0 + z) * N + n) * M, plane = (int64_t)Nw * N * M;
  const double* pr = prod + ((int64_t)z * 2 * N + n) * R;       // column n of the real half
  const double* pi = pr + (int64_t)N * R;
  double x[NP][2][2];   // [pair][element][re, im]
  uint32_t mx = 0, nan = 0;
#pragma unroll
  for (int t = 0; t < NP; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = 64 * t + 2 * lane + q;
      double re = 0.0, im = 0.0;
      if (i < M) {
        if (FIRST) {
          re = phi[base + i];
          im = phi[plane + base + i];
        } else {
          if (stack) {
            re = pr[i] - pi[M + i];
            im = pi[i] + pr[M + i];
          } else {
            re = pr[i];
            im = pi[i];
          }
          phi[base + i] = fma(coef, re, phi[base + i]);
          phi[plane + base + i] = fma(coef, im, phi[plane + base + i]);
        }
      }
      x[t][q][0] = re;
      x[t][q][1] = im;
      row_scan(re, mx, nan);
      row_scan(im, mx, nan);
    }
  if (!more) return;
  int mark;
  const int em = row_exponent(mx, nan, mark, [&]() {
    long long f = 0;
#pragma unroll
    for (int t = 0; t < NP; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) f = max(f, fraction_of(x[t][q >> 1][q & 1]));
    return f;
  });
  const int64_t r0 = (int64_t)z * 2 * N + n, r1 = r0 + N;
  if (lane == 0) ex[r0] = ex[r1] = mark;
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    const int k = 64 * t + 2 * lane;
    if (k >= M) break;
    uint32_t a[2], b[2], c[2], d[2];
    digit_bytes_of(x[t][0][0], em, mark >= kExpInf, a[0], a[1]);
    digit_bytes_of(x[t][1][0], em, mark >= kExpInf, b[0], b[1]);
    digit_bytes_of(x[t][0][1], em, mark >= kExpInf, c[0], c[1]);
    digit_bytes_of(x[t][1][1], em, mark >= kExpInf, d[0], d[1]);
#pragma unroll
    for (int j = 0; j < kDig; ++j) {
      const uint32_t re = digit_pair(j, a, b), im = digit_pair(j, c, d);
      uint32_t* p0 = reinterpret_cast<uint32_t*>(out + ((int64_t)j * rp + r0) * Kp + k);
      uint32_t* p1 = reinterpret_cast<uint32_t*>(out + ((int64_t)j * rp + r1) * Kp + k);
      *p0 = re;
      *p1 = im;
      if (!stack) {
        p0[M2 / 2] = im ^ 0x80008000u;
        p1[M2 / 2] = re;
      }
    }
  }
}

template <bool FIRST>
cudaError_t launch_term(const Ctx& c, const Plan& p, const double* prod, double* phi, int w0, int nw, double coef,
                        int more, const DigitOp& b, cudaStream_t s) {
  const int grid = (nw * c.N + 7) / 8, st = stacked(c.M), M2 = even(c.M);
  switch ((c.M + 63) / 64) {
#define AFQ_TERM(NP)                                                                                        \
  case NP:                                                                                                  \
    k_term<NP, FIRST><<<grid, 256, 0, s>>>(prod, phi, c.M, c.N, c.Nw, w0, nw, st, M2, coef, more, b.Kp, b.rp, \
                                           b.dig, b.ex);                                                    \
    break;
    AFQ_TERM(1)
    AFQ_TERM(2)
    AFQ_TERM(3)
    AFQ_TERM(4)
#undef AFQ_TERM
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

// The digit form against k_taylor at 1.05 TFLOP/s: 2 launches of about 4 us per round and chunk,
// and the padded products at 1.0 PFLOP/s with their columns in tiles of 16, 32, 48 or 64.
bool taylor_f64e_ok(int M, int N, int Nw, int order) {
  if (M > kMaxM || M < 12) return false;
  const Plan p = plan_of(M, N, Nw);
  const double cols = p.Cn <= 48 ? (p.Cn + 15) / 16 * 16 : (p.Cn + 63) / 64 * 64;
  const double nch = (double)((Nw + p.nw - 1) / p.nw);
  const double pipe = 8.0 * order * M * M * N * (double)Nw / 1.05e6;
  const double dig = nch * (12.0 + 8.0 * order) +
                     72.0 * order * (double)Nw * ((p.R + 127) / 128 * 128) * cols * pad64(p.K) / 1.0e9;
  return pipe > 1.3 * dig;
}

size_t taylor_f64e_ws(int M, int N, int Nw) {
  const Plan p = plan_of(M, N, Nw);
  return digit_bytes((int64_t)p.nw * p.R, p.K) + digit_bytes((int64_t)p.nw * p.Cn, p.K) +
         sizeof(double) * (size_t)p.nw * p.R * p.Cn + 1024;
}

// Phi <- sum_m A^m Phi / m! in place, A from c.Avhs.
cudaError_t launch_taylor_f64e(const Ctx& c, double* phi, cudaStream_t s) {
  const Plan p = plan_of(c.M, c.N, c.Nw);
  const int order = c.opt.taylor_order;
  cudaError_t e = cudaSuccess;
  for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += p.nw) {
    const int nw = std::min(p.nw, c.Nw - w0);
    const DigitOp a = digit_place(c.ws64.buf, (int64_t)nw * p.R, p.K);
    uint8_t* pb = c.ws64.buf + digit_bytes((int64_t)nw * p.R, p.K);
    const DigitOp b = digit_place(pb, (int64_t)nw * p.Cn, p.K);
    double* prod = reinterpret_cast<double*>(pb + digit_bytes((int64_t)nw * p.Cn, p.K));
    k_vhs_digits<<<nw, 512, 0, s>>>(c.Avhs, c.P, c.M, c.Nw, w0, stacked(c.M), even(c.M), a.Kp, a.rp, a.dig, a.ex);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    // the columns' padding in K meets zero digits of A, but must be finite
    if ((e = cudaMemsetAsync(b.dig, 0, (size_t)b.rp * b.Kp * 2 * kDig, s)) != cudaSuccess) break;
    if ((e = launch_term<true>(c, p, prod, phi, w0, nw, 0.0, 1, b, s)) != cudaSuccess) break;
    double coef = 1.0;
    for (int m = 1; m <= order && e == cudaSuccess; ++m) {
      DigitGemm g;
      g.R = p.R;
      g.Cn = p.Cn;
      g.nz = nw;
      g.rz = p.R;
      g.cz = p.Cn;
      g.out = prod;
      g.ldc = p.R;
      g.outz = (int64_t)p.R * p.Cn;
      g.K = p.K;
      g.err = c.ws64.err;
      if ((e = digit_gemm(a, b, g, s)) != cudaSuccess) break;
      coef /= m;
      e = launch_term<false>(c, p, prod, phi, w0, nw, coef, m < order, b, s);
    }
  }
  return e;
}

}  // namespace afq
