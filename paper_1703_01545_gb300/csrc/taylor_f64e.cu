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

// What a term kernel does with the round's product U (of A, or of conj(A) in the reverse sweep).
enum TermKind {
  kFirst = 0,   // x = in
  kSum = 1,     // x = U, acc += coef x
  kKeep = 2,    // x = U, out = coef x
  kRev = 3      // x = in + coef U, out = x (where the walker's mask allows)
};

struct TermArgs {
  const double* prod;    // products of walkers w0 .., [z][2 N][R]
  const double* in;      // [2][Nw][N][M]
  double* out;           // [2][Nw][N][M], or null
  const int* mask;       // kRev: walkers whose out is written, or null
  double coef;
  int M, N, Nw, w0, nw, stack, M2;
  int conj;              // the digits' products are with conj(A) (and so were kRev's)
  int more;              // digits of x as the next round's columns
  int Kp;
  int64_t rp;
  __nv_bfloat16* dig;
  int* ex;
};

// One term of walkers w0 .. : a warp per (walker, column n), lanes over pairs of orbitals.
// Columns n and N + n of the next product, joined K: [x_r | -x_i], [x_i | x_r] for A, [x_r | x_i],
// [x_i | -x_r] for conj(A); stacked rows: x_r, x_i for both.
template <int NP, int KIND>
__global__ void __launch_bounds__(256) k_term(const TermArgs a) {
  const int task = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, M = a.M, N = a.N;
  if (task >= a.nw * N) return;
  const int z = task / N, n = task - z * N, R = a.stack ? 2 * M : M;
  const int64_t base = ((int64_t)(a.w0 + z) * N + n) * M, plane = (int64_t)a.Nw * N * M;
  const double* pr = a.prod + ((int64_t)z * 2 * N + n) * R;     // column n of the real half
  const double* pi = pr + (int64_t)N * R;
  const bool write = KIND != kRev || (a.out && (!a.mask || a.mask[a.w0 + z]));
  double x[NP][2][2];   // [pair][element][re, im]
  uint32_t mx = 0, nan = 0;
#pragma unroll
  for (int t = 0; t < NP; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = 64 * t + 2 * lane + q;
      double re = 0.0, im = 0.0;
      if (i < M) {
        if (KIND == kFirst) {
          re = a.in[base + i];
          im = a.in[plane + base + i];
        } else {
          if (!a.stack) {
            re = pr[i];
            im = pi[i];
          } else if (KIND == kRev) {
            re = pr[i] + pi[M + i];
            im = pi[i] - pr[M + i];
          } else {
            re = pr[i] - pi[M + i];
            im = pi[i] + pr[M + i];
          }
          if (KIND == kSum) {
            a.out[base + i] = fma(a.coef, re, a.out[base + i]);
            a.out[plane + base + i] = fma(a.coef, im, a.out[plane + base + i]);
          }
          if (KIND == kRev) {
            re = fma(a.coef, re, a.in[base + i]);
            im = fma(a.coef, im, a.in[plane + base + i]);
          }
          if (KIND == kKeep) {
            a.out[base + i] = a.coef * re;
            a.out[plane + base + i] = a.coef * im;
          }
          if (KIND == kRev && write) {
            a.out[base + i] = re;
            a.out[plane + base + i] = im;
          }
        }
      }
      x[t][q][0] = re;
      x[t][q][1] = im;
      row_scan(re, mx, nan);
      row_scan(im, mx, nan);
    }
  if (!a.more) return;
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
  if (lane == 0) a.ex[r0] = a.ex[r1] = mark;
  const uint32_t neg_re = a.conj ? 0u : 0x80008000u, neg_im = a.conj ? 0x80008000u : 0u;
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    const int k = 64 * t + 2 * lane;
    if (k >= M) break;
    uint32_t b[2], c[2], d[2], e[2];
    digit_bytes_of(x[t][0][0], em, mark >= kExpInf, b[0], b[1]);
    digit_bytes_of(x[t][1][0], em, mark >= kExpInf, c[0], c[1]);
    digit_bytes_of(x[t][0][1], em, mark >= kExpInf, d[0], d[1]);
    digit_bytes_of(x[t][1][1], em, mark >= kExpInf, e[0], e[1]);
#pragma unroll
    for (int j = 0; j < kDig; ++j) {
      const uint32_t re = digit_pair(j, b, c), im = digit_pair(j, d, e);
      uint32_t* p0 = reinterpret_cast<uint32_t*>(a.dig + ((int64_t)j * a.rp + r0) * a.Kp + k);
      uint32_t* p1 = reinterpret_cast<uint32_t*>(a.dig + ((int64_t)j * a.rp + r1) * a.Kp + k);
      *p0 = re;
      *p1 = im;
      if (!a.stack) {
        p0[a.M2 / 2] = im ^ neg_re;
        p1[a.M2 / 2] = re ^ neg_im;
      }
    }
  }
}

template <int KIND>
cudaError_t launch_term(const TermArgs& a, cudaStream_t s) {
  const int grid = (a.nw * a.N + 7) / 8;
  switch ((a.M + 63) / 64) {
    case 1: k_term<1, KIND><<<grid, 256, 0, s>>>(a); break;
    case 2: k_term<2, KIND><<<grid, 256, 0, s>>>(a); break;
    case 3: k_term<3, KIND><<<grid, 256, 0, s>>>(a); break;
    case 4: k_term<4, KIND><<<grid, 256, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Tangent mode: U = A U' and dU = dA U' + A dU' of a round; products of [U' | dU'] with A ([z][4 N][R])
// and of U' with dA ([z][2 N][R]).  FIRST: U = Phi, dU = dPhi; else Phi += coef U, dPhi += coef dU.
// Columns of a walker: U's real, U's imaginary, dU's real, dU's imaginary ones.
template <int NP, bool FIRST>
__global__ void __launch_bounds__(256) k_term_tan(const double* __restrict__ prod, const double* __restrict__ dprod,
                                                  double* __restrict__ phi, double* __restrict__ dphi, int M, int N,
                                                  int Nw, int w0, int nw, int stack, int M2, double coef, int more,
                                                  int Kp, int64_t rp, __nv_bfloat16* __restrict__ out,
                                                  int* __restrict__ ex) {
  const int task = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (task >= 2 * nw * N) return;
  const int d = task & 1, zn = task >> 1, z = zn / N, n = zn - z * N, R = stack ? 2 * M : M;   // d = 1: dU
  const int64_t base = ((int64_t)(w0 + z) * N + n) * M, plane = (int64_t)Nw * N * M;
  double* x0 = d ? dphi : phi;
  const double* pr = prod + ((int64_t)z * 4 * N + d * 2 * N + n) * R;
  const double* pi = pr + (int64_t)N * R;
  const double* qr = dprod + ((int64_t)z * 2 * N + n) * R;
  const double* qi = qr + (int64_t)N * R;
  double x[NP][2][2];
  uint32_t mx = 0, nan = 0;
#pragma unroll
  for (int t = 0; t < NP; ++t)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = 64 * t + 2 * lane + q;
      double re = 0.0, im = 0.0;
      if (i < M) {
        if (FIRST) {
          re = x0[base + i];
          im = x0[plane + base + i];
        } else {
          re = stack ? pr[i] - pi[M + i] : pr[i];
          im = stack ? pi[i] + pr[M + i] : pi[i];
          if (d) {
            re += stack ? qr[i] - qi[M + i] : qr[i];
            im += stack ? qi[i] + qr[M + i] : qi[i];
          }
          x0[base + i] = fma(coef, re, x0[base + i]);
          x0[plane + base + i] = fma(coef, im, x0[plane + base + i]);
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
  const int64_t r0 = (int64_t)z * 4 * N + d * 2 * N + n, r1 = r0 + N;
  if (lane == 0) ex[r0] = ex[r1] = mark;
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    const int k = 64 * t + 2 * lane;
    if (k >= M) break;
    uint32_t a[2], b[2], c[2], e[2];
    digit_bytes_of(x[t][0][0], em, mark >= kExpInf, a[0], a[1]);
    digit_bytes_of(x[t][1][0], em, mark >= kExpInf, b[0], b[1]);
    digit_bytes_of(x[t][0][1], em, mark >= kExpInf, c[0], c[1]);
    digit_bytes_of(x[t][1][1], em, mark >= kExpInf, e[0], e[1]);
#pragma unroll
    for (int j = 0; j < kDig; ++j) {
      const uint32_t re = digit_pair(j, a, b), im = digit_pair(j, c, e);
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

// A chunk of walkers in the workspace: digits of A and of the terms, products.
struct Chunk {
  DigitOp a, b;
  double* prod;
  uint8_t* end;
  DigitGemm g;
  TermArgs t;
};

cudaError_t start_chunk(const Ctx& c, const F64Ws& ws, const Plan& p, int w0, int nw, Chunk& k, cudaStream_t s) {
  k.a = digit_place(ws.buf, (int64_t)nw * p.R, p.K);
  uint8_t* pb = ws.buf + digit_bytes((int64_t)nw * p.R, p.K);
  k.b = digit_place(pb, (int64_t)nw * p.Cn, p.K);
  k.prod = reinterpret_cast<double*>(pb + digit_bytes((int64_t)nw * p.Cn, p.K));
  k.end = reinterpret_cast<uint8_t*>(k.prod) + (sizeof(double) * (size_t)nw * p.R * p.Cn + 255) / 256 * 256;
  DigitGemm& g = k.g;
  g.R = p.R;
  g.Cn = p.Cn;
  g.nz = nw;
  g.rz = p.R;
  g.cz = p.Cn;
  g.out = k.prod;
  g.ldc = p.R;
  g.outz = (int64_t)p.R * p.Cn;
  g.K = p.K;
  g.err = ws.err;
  k.t = TermArgs{k.prod, nullptr, nullptr, nullptr, 0.0, c.M, c.N, c.Nw, w0, nw, stacked(c.M), even(c.M),
                 0, 1, k.b.Kp, k.b.rp, k.b.dig, k.b.ex};
  k_vhs_digits<<<nw, 512, 0, s>>>(c.Avhs, c.P, c.M, c.Nw, w0, stacked(c.M), even(c.M), k.a.Kp, k.a.rp, k.a.dig,
                                  k.a.ex);
  cudaError_t e = cudaGetLastError();
  // the columns' padding in K meets zero digits of A, but must be finite
  if (e == cudaSuccess) e = cudaMemsetAsync(k.b.dig, 0, (size_t)k.b.rp * k.b.Kp * 2 * kDig, s);
  return e;
}

// Terms of the Taylor series at orbital i, k = (n N + b) 2 + re / im: x[n][plane][w][b][i].
struct TermRows {
  const double* x;
  int64_t nstride, plane;   // one term, one plane
  int N, M, w0;
  __device__ double at(int z, int i, int k) const {
    const int p = k & 1, nb = k >> 1, n = nb / N, b = nb - n * N;
    return x[n * nstride + p * plane + ((int64_t)(w0 + z) * N + b) * M + i];
  }
};

// Abar of the walkers that are out of the reverse sweep
__global__ void __launch_bounds__(256) k_zero_masked(double* __restrict__ Abar, const int* __restrict__ mask, int MM,
                                                     int Nw) {
  const int w = blockIdx.x;
  if (mask[w]) return;
  for (int p = 0; p < 2; ++p)
    for (int e = threadIdx.x; e < MM; e += 256) Abar[((int64_t)p * Nw + w) * MM + e] = 0.0;
}

size_t outer_bytes(int M, int K2, int nw) {
  return digit_bytes((int64_t)nw * M, K2) + digit_bytes(2 * (int64_t)nw * M, K2);
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
    Chunk k;
    if ((e = start_chunk(c, c.ws64, p, w0, std::min(p.nw, c.Nw - w0), k, s)) != cudaSuccess) break;
    k.t.in = phi;
    if ((e = launch_term<kFirst>(k.t, s)) != cudaSuccess) break;
    k.t.out = phi;
    k.t.coef = 1.0;
    for (int m = 1; m <= order && e == cudaSuccess; ++m) {
      if ((e = digit_gemm(k.a, k.b, k.g, s)) != cudaSuccess) break;
      k.t.coef /= m;
      k.t.more = m < order;
      e = launch_term<kSum>(k.t, s);
    }
  }
  return e;
}

namespace {
// bytes of the workspace a walker takes in tangent mode: digits of A, dA and four sets of columns
// (each with its padding to 128 rows over the chunk, below), products
size_t tan_per(const Plan& p) {
  return (size_t)(2 * p.R + 2 * p.Cn) * ((size_t)pad64(p.K) * 2 * kDig + 4) + sizeof(double) * 3 * (size_t)p.R * p.Cn;
}
int tan_chunk(const Ctx& c, const Plan& p) {
  const size_t pad = 3 * digit_bytes(128, p.K) + 4096;
  if (!c.ws64.buf || c.ws64.bytes <= pad) return 0;
  return (int)std::min<size_t>((size_t)c.Nw, (c.ws64.bytes - pad) / tan_per(p));
}
}  // namespace

// Where the plain series runs in digit form and the handle's workspace holds a chunk of some size.
bool taylor_tan_f64e_ok(const Ctx& c) {
  if (!c.taylor_dig || !taylor_f64e_ok(c.M, c.N, c.Nw, c.opt.taylor_order)) return false;
  return tan_chunk(c, plan_of(c.M, c.N, c.Nw)) >= std::min(c.Nw, 38);
}

// Phi <- T_n(A) Phi and dPhi <- its derivative along dA and dPhi, in place.
cudaError_t launch_taylor_tan_f64e(const Ctx& c, double* phi, double* dphi, cudaStream_t s) {
  const Plan p = plan_of(c.M, c.N, c.Nw);
  const int nwc = tan_chunk(c, p), order = c.opt.taylor_order, M2 = even(c.M), st = stacked(c.M);
  cudaError_t e = cudaSuccess;
  for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += nwc) {
    const int nw = std::min(nwc, c.Nw - w0), cn = 2 * p.Cn;
    uint8_t* at = c.ws64.buf;
    DigitOp a[2];
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
      a[q] = digit_place(at, (int64_t)nw * p.R, p.K);
      at += digit_bytes((int64_t)nw * p.R, p.K);
      k_vhs_digits<<<nw, 512, 0, s>>>(q ? c.dAvhs : c.Avhs, c.P, c.M, c.Nw, w0, st, M2, a[q].Kp, a[q].rp, a[q].dig,
                                      a[q].ex);
      e = cudaGetLastError();
    }
    const DigitOp b = digit_place(at, (int64_t)nw * cn, p.K);
    at += digit_bytes((int64_t)nw * cn, p.K);
    double* prod = reinterpret_cast<double*>(at);
    double* dprod = prod + (size_t)nw * p.R * cn;
    if (e == cudaSuccess) e = cudaMemsetAsync(b.dig, 0, (size_t)b.rp * b.Kp * 2 * kDig, s);
    auto term = [&](bool first, double coef, int more) -> cudaError_t {
      const int grid = (2 * nw * c.N + 7) / 8;
#define AFQ_TERM(NP)                                                                                             \
  case NP:                                                                                                       \
    if (first)                                                                                                   \
      k_term_tan<NP, true><<<grid, 256, 0, s>>>(prod, dprod, phi, dphi, c.M, c.N, c.Nw, w0, nw, st, M2, coef, more, \
                                                b.Kp, b.rp, b.dig, b.ex);                                        \
    else                                                                                                         \
      k_term_tan<NP, false><<<grid, 256, 0, s>>>(prod, dprod, phi, dphi, c.M, c.N, c.Nw, w0, nw, st, M2, coef,   \
                                                 more, b.Kp, b.rp, b.dig, b.ex);                                 \
    break;
      switch ((c.M + 63) / 64) {
        AFQ_TERM(1)
        AFQ_TERM(2)
        AFQ_TERM(3)
        AFQ_TERM(4)
        default: return cudaErrorInvalidValue;
      }
#undef AFQ_TERM
      return cudaGetLastError();
    };
    if (e != cudaSuccess || (e = term(true, 0.0, 1)) != cudaSuccess) break;
    double coef = 1.0;
    for (int m = 1; m <= order && e == cudaSuccess; ++m) {
      DigitGemm g;
      g.R = p.R;
      g.Cn = cn;
      g.nz = nw;
      g.rz = p.R;
      g.cz = cn;
      g.out = prod;
      g.ldc = p.R;
      g.outz = (int64_t)p.R * cn;
      g.K = p.K;
      g.err = c.ws64.err;
      if ((e = digit_gemm(a[0], b, g, s)) != cudaSuccess) break;
      g.Cn = p.Cn;
      g.out = dprod;
      g.outz = (int64_t)p.R * p.Cn;
      if ((e = digit_gemm(a[1], b, g, s)) != cudaSuccess) break;
      coef /= m;
      e = term(false, coef, m < order);
    }
  }
  return e;
}

size_t taylor_rev_f64e_ws(int M, int N, int Nw, int order) {
  const Plan p = plan_of(M, N, Nw);
  return taylor_f64e_ws(M, N, Nw) + outer_bytes(M, 2 * order * N, p.nw);
}

// Reverse of the Taylor series at the walkers' A (adj_taylor): with U_n = A^n Phi1 and
//   V_order = Pbar2,  V_(n-1) = Pbar2 + conj(A) V_n / n,
// pbar <- V_0 and Abar = sum_n V_n (U_(n-1) / n!)^H (u keeps U_(n-1) / n!), the last as one contraction over (n, b, re / im)
// per walker.  u, v: [order][2][Nw][N][M] each.  Abar comes out transposed, [2][Nw][j][i], which its
// only use, the trace with the symmetric L_g, does not see.  At M = 96, 12/12, 128 walkers, order 6:
// 4.93 ms in the walker kernel (k_taylor_rev), 0.55 ms here.
cudaError_t launch_taylor_rev_f64e(const Ctx& c, const F64Ws& ws, const double* phi1, double* pbar, double* u,
                                   double* v, double* Abar, const int* mask, cudaStream_t s) {
  const Plan p = plan_of(c.M, c.N, c.Nw);
  const int order = c.opt.taylor_order, M = c.M, MM = M * M, K2 = 2 * order * c.N;
  const int64_t nphi = 2 * (int64_t)c.Nw * c.N * M;
  cudaError_t e = cudaSuccess;
  for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += p.nw) {
    const int nw = std::min(p.nw, c.Nw - w0);
    // U_0 and V_order of the chunk as they are
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
      const int64_t o = ((int64_t)q * c.Nw + w0) * c.N * M;
      const size_t by = sizeof(double) * (size_t)nw * c.N * M;
      e = cudaMemcpyAsync(u + o, phi1 + o, by, cudaMemcpyDeviceToDevice, s);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(v + (order - 1) * nphi + o, pbar + o, by, cudaMemcpyDeviceToDevice, s);
    }
    Chunk k;
    if (e != cudaSuccess || (e = start_chunk(c, ws, p, w0, nw, k, s)) != cudaSuccess) break;
    k.t.in = phi1;
    k.t.more = order > 1;
    if ((e = launch_term<kFirst>(k.t, s)) != cudaSuccess) break;
    k.t.coef = 1.0;
    for (int m = 1; m < order && e == cudaSuccess; ++m) {
      if ((e = digit_gemm(k.a, k.b, k.g, s)) != cudaSuccess) break;
      k.t.coef /= m + 1;
      k.t.out = u + m * nphi;
      k.t.more = m + 1 < order;
      e = launch_term<kKeep>(k.t, s);
    }
    k.t.conj = 1;
    k.t.more = 1;
    k.t.in = v + (order - 1) * nphi;
    if (e == cudaSuccess) e = launch_term<kFirst>(k.t, s);
    for (int n = order; n >= 1 && e == cudaSuccess; --n) {
      if ((e = digit_gemm(k.a, k.b, k.g, s)) != cudaSuccess) break;
      k.t.coef = 1.0 / n;
      k.t.out = n > 1 ? v + (n - 2) * nphi : pbar;
      k.t.mask = n > 1 ? nullptr : mask;
      k.t.more = n > 1;
      e = launch_term<kRev>(k.t, s);
    }
    if (e != cudaSuccess) break;
    // V[(n-1)] holds V_n, u[(n-1)] U_(n-1): both at index n - 1
    const DigitOp dv = digit_place(k.end, (int64_t)nw * M, K2);
    const DigitOp du = digit_place(k.end + digit_bytes((int64_t)nw * M, K2), 2 * (int64_t)nw * M, K2);
    const dim3 grid(nw, (M + 31) / 32);
    const TermRows fv{v, nphi, nphi / 2, c.N, M, w0}, fu{u, nphi, nphi / 2, c.N, M, w0};
    k_strided_digits<<<grid, 1024, 0, s>>>(fv, M, K2, dv.Kp, dv.rp, M, 0, reinterpret_cast<uint16_t*>(dv.dig), dv.ex);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    k_strided_digits<<<grid, 1024, 0, s>>>(fu, M, K2, du.Kp, du.rp, 2 * M, M, reinterpret_cast<uint16_t*>(du.dig), du.ex);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {   // re: [U_r | U_i], im: [-U_i | U_r]
      DigitOp dq = du;
      dq.dig += (int64_t)q * M * du.Kp;
      dq.ex += q * M;
      dq.off = q * M;
      DigitGemm g;
      g.R = g.Cn = M;
      g.nz = nw;
      g.rz = M;
      g.cz = 2 * M;
      g.out = Abar + ((int64_t)q * c.Nw + w0) * MM;
      g.ldc = M;
      g.outz = MM;
      g.K = K2;
      g.err = ws.err;
      e = digit_gemm(dv, dq, g, s);
    }
  }
  if (e != cudaSuccess) return e;
  k_zero_masked<<<c.Nw, 256, 0, s>>>(Abar, mask, MM, c.Nw);
  return cudaGetLastError();
}

}  // namespace afq
