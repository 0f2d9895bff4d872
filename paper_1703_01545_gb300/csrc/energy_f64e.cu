// FP64 local energy (Eq. 7 with Wick's theorem) with the half-rotated products in digit form:
//   E_L = sum_(n,i) htil[n][i] Theta[n][i]
//       + 1/2 sum_g [ (sum_s tr T^s_g)^2 - sum_s sum_ab T^s_g[a][b] T^s_g[b][a] ],
//   T^s_g[a][b] = sum_i Ltil[g][n0+a][i] Theta[n0+b][i].
//
// T of every Cholesky vector is 4 X M sum_s N_s^2 operations per walker, all of the energy's work
// but a few per cent: as one contraction per spin, rows (g, a) by columns (re/im, w, b), it runs as
// exact BF16 digit products on the tensor cores (gemm_f64e.cu) instead of on the FP64 pipe (2
// multiply-adds per clock and SM).  T is X N_s^2 complex numbers per walker, too many to keep for
// all walkers: it goes through a buffer of walker chunks small enough to stay in the 129 MB L2,
// where the exchange and trace sums read it back, each pair (a, b), (b, a) once.  Those sums, half
// of N_s^2 complex products per (g, w), are what is left on the FP64 pipe.
// Measured at M = 64, X = 320, 8/8, 2048 walkers: 19.25 ms in the per-walker FP64 kernel (k_energy,
// still the faster one for small products), 2.38 ms here: contraction 1.07, exchange sums 1.11 (FP64
// pipe; 0.29 at its full rate), digits 0.14.  Error of E_L against float64 arithmetic 1.4e-16.
#include <algorithm>
#include <cstdint>

#include "device_util.cuh"
#include "internal.h"

namespace afq {
namespace {

constexpr size_t kTBytes = (size_t)80 << 20;   // T chunk: leaves L2 room for the digits of the next
constexpr size_t kStage = 40 * 1024;           // staged T of one step of k_exchange
constexpr int kMaxSplit = 16;                  // ranges of g that share a walker's exchange sum
constexpr int kEx = 256;

// Exchange sums and traces of one spin for walkers w0 .. w0 + gridDim.x - 1; T[(p, wl, b)][(g, a)]
// with rows of ldt = X ns.  CTA (wl, q) takes the q-th range of g, gb (a power of two up to 32) of
// them staged at a time (one coalesced read) as [p][b][a][g]: the lanes of a warp are consecutive g
// (32 / gb pairs side by side for gb < 32), so the staged reads touch every bank once, and a warp
// takes the pairs a <= b in turn:
//   ex[q][p][w] = sum_g sum_ab T_ab T_ba,   tr[p][w][g] = sum_a T_aa.
// Bound by the FP64 pipe: 4 multiply-adds per pair and g, 2 per clock and SM.
__global__ void __launch_bounds__(kEx) k_exchange(const double* __restrict__ T, int64_t ldt, int ns, int X,
                                                  int w0, int Nw, int gb, double* __restrict__ ex,
                                                  double* __restrict__ tr) {
  extern __shared__ double sm[];
  __shared__ double red[2 * (kEx / 32)];
  const int wl = blockIdx.x, nwc = gridDim.x, q = blockIdx.y, tid = threadIdx.x, w = w0 + wl;
  const int g0 = (int)((int64_t)X * q / gridDim.y), g1 = (int)((int64_t)X * (q + 1) / gridDim.y);
  const int np = ns * (ns + 1) / 2, gs = gb + 1;   // odd row length: the staging writes spread too
  const int pl = ns * ns * gs;                     // imaginary plane
  const int lg = tid & (gb - 1), slot = tid / gb, nslot = kEx / gb;
  // sums over a = b (xr^2 - xi^2, xr xi) and over a < b (T_ab T_ba), doubled where due at the end
  double d[2] = {0.0, 0.0}, o[2] = {0.0, 0.0};
  for (int gc = g0; gc < g1; gc += gb) {
    const int ng = min(gb, g1 - gc), len = ng * ns;
    __syncthreads();
    for (int col = tid >> 5; col < 2 * ns; col += kEx / 32) {
      const int p = col / ns, b = col - p * ns;
      const double* src = T + ((int64_t)(p * nwc + wl) * ns + b) * ldt + (int64_t)gc * ns;
      for (int k = tid & 31; k < len; k += 32) {
        const int g = k / ns;
        sm[(col * ns + k - g * ns) * gs + g] = src[k];
      }
    }
    __syncthreads();
    if (lg < ng) {
      int b = 0, a = slot;   // pair r = b (b + 1) / 2 + a, a <= b
      while (a > b) a -= ++b;
      for (int r = slot; r < np; r += nslot) {
        const double* xy = sm + (b * ns + a) * gs + lg;   // T_ab
        const double xr = xy[0], xi = xy[pl];
        if (a == b) {
          d[0] = fma(xr, xr, fma(-xi, xi, d[0]));
          d[1] = fma(xr, xi, d[1]);
        } else {
          const double* yx = sm + (a * ns + b) * gs + lg;
          const double yr = yx[0], yi = yx[pl];
          o[0] = fma(xr, yr, fma(-xi, yi, o[0]));
          o[1] = fma(xr, yi, fma(xi, yr, o[1]));
        }
        a += nslot;
        while (a > b) a -= ++b;
      }
    }
    for (int e = tid; e < 2 * ng; e += kEx) {
      const int p = e / ng, g = e - p * ng;
      double t = 0.0;
      for (int a = 0; a < ns; ++a) t += sm[p * pl + (a * ns + a) * gs + g];
      tr[((int64_t)p * Nw + w) * X + gc + g] = t;
    }
  }
  double acc[2] = {fma(2.0, o[0], d[0]), 2.0 * (o[1] + d[1])};
  block_sum<2>(acc, red);
  if (tid == 0) {
    ex[((int64_t)q * 2) * Nw + w] = acc[0];
    ex[((int64_t)q * 2 + 1) * Nw + w] = acc[1];
  }
}

// E_L of a walker from its one-body sum, the traces [spin][p][w][g] of both spins and the exchange
// sums [spin][range][p][w].
__global__ void __launch_bounds__(128) k_energy_sum(const double* __restrict__ theta, const double* __restrict__ htil,
                                                    const double* __restrict__ tr, const double* __restrict__ ex,
                                                    int nspin, int nsplit, int NM, int X, int Nw,
                                                    double* __restrict__ eloc) {
  __shared__ double red[2 * 4];
  const int w = blockIdx.x;
  const int64_t plane = (int64_t)Nw * NM, base = (int64_t)w * NM, tsp = 2 * (int64_t)Nw * X;
  double acc[2] = {0.0, 0.0};
  for (int e = threadIdx.x; e < NM; e += 128) {
    const double h = __ldg(htil + e);
    acc[0] = fma(h, theta[base + e], acc[0]);
    acc[1] = fma(h, theta[plane + base + e], acc[1]);
  }
  for (int g = threadIdx.x; g < X; g += 128) {
    double cr = 0.0, ci = 0.0;
    for (int s = 0; s < nspin; ++s) {
      cr += tr[s * tsp + (int64_t)w * X + g];
      ci += tr[s * tsp + ((int64_t)Nw + w) * X + g];
    }
    acc[0] = fma(0.5 * cr, cr, fma(-0.5 * ci, ci, acc[0]));
    acc[1] = fma(cr, ci, acc[1]);
  }
  block_sum<2>(acc, red);
  if (threadIdx.x == 0) {
    double er = 0.0, ei = 0.0;
    for (int q = 0; q < nspin * nsplit; ++q) {
      er += ex[((int64_t)q * 2) * Nw + w];
      ei += ex[((int64_t)q * 2 + 1) * Nw + w];
    }
    eloc[w] = acc[0] - 0.5 * er;
    eloc[Nw + w] = acc[1] - 0.5 * ei;
  }
}

// Walkers per chunk: T of both planes within kTBytes for the larger spin (one at least).
int chunk_walkers(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  const size_t per = 2 * (size_t)c.X * ns * ns * sizeof(double);
  return (int)std::max<size_t>(1, std::min<size_t>((size_t)c.Nw, kTBytes / per));
}

// CTAs over g so that a chunk of walkers fills the SMs a few times over
int splits(const Ctx& c, int nwc) {
  return std::max(1, std::min({kMaxSplit, (8 * 152 + nwc - 1) / nwc, c.X / 16}));
}

}  // namespace

// Where the contraction of the larger spin pays in digit form; a chunk of few walkers would
// slice the rows (g, a) anew for too few columns, so its T has to be at least as large as Ltil.
bool energy_f64e_ok(int M, int X, int n_up, int n_dn, int Nw) {
  const int ns = std::max(n_up, n_dn);
  return (int64_t)X * ns < (int64_t)1 << 30 && 2 * (size_t)X * ns * ns * 8 <= kTBytes &&
         gemm_f64e_ok(X * ns, (int)std::min<int64_t>(2 * (int64_t)Nw * ns, 1 << 30), M);
}

// Scratch: T, traces of both spins, exchange sums, and the digits (of the rows (g, a) of a spin,
// and of a chunk's columns) in the contractions' workspace.
size_t energy_f64e_scratch(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  const size_t t = 2 * (size_t)c.X * ns * ns * chunk_walkers(c);
  return sizeof(double) * (t + 4 * (size_t)c.Nw * c.X + 4 * (size_t)kMaxSplit * c.Nw);
}
size_t energy_f64e_ws(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  return digit_bytes((int64_t)c.X * ns, c.M) + digit_bytes(2 * (int64_t)chunk_walkers(c) * ns, c.M);
}

cudaError_t launch_energy_f64e(const Ctx& c, cudaStream_t s) {
  const int NM = c.N * c.M, nwc = chunk_walkers(c), nsmax = std::max(c.n_up, c.N - c.n_up);
  const int nsplit = splits(c, nwc);
  double* T = c.e64;
  double* tr = T + 2 * (size_t)c.X * nsmax * nsmax * nwc;
  double* ex = tr + 4 * (size_t)c.Nw * c.X;
  cudaError_t e = cudaSuccess;
  int sp = 0;
  for (int s0 = 0; s0 < 2 && e == cudaSuccess; ++s0) {
    const int n0 = s0 ? c.n_up : 0, ns = s0 ? c.N - c.n_up : c.n_up;
    if (ns == 0) continue;
    const int rows = c.X * ns;
    const DigitOp da = digit_place(c.ws64.buf, rows, c.M);
    e = digits_of(c.Ltil, c.M, rows, c.M, da, s, ns, c.N, n0);
    for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += nwc) {
      const int nw = std::min(nwc, c.Nw - w0), cols = 2 * nw * ns;
      const DigitOp db = digit_place(c.ws64.buf + digit_bytes(rows, c.M), cols, c.M);
      for (int p = 0; p < 2 && e == cudaSuccess; ++p) {
        DigitOp dp = db;
        dp.dig += (int64_t)p * nw * ns * db.Kp;
        dp.ex += p * nw * ns;
        e = digits_of(c.theta + ((int64_t)p * c.Nw + w0) * NM, c.M, nw * ns, c.M, dp, s, ns, c.N, n0);
      }
      if (e != cudaSuccess) break;
      DigitGemm g;
      g.R = rows;
      g.Cn = cols;
      g.out = T;
      g.ldc = rows;
      g.K = c.M;
      g.err = c.ws64.err;
      if ((e = digit_gemm(da, db, g, s)) != cudaSuccess) break;
      int gb = 32;
      while (gb > 1 && (size_t)2 * ns * ns * (gb + 1) * sizeof(double) > kStage) gb /= 2;
      k_exchange<<<dim3(nw, nsplit), kEx, (size_t)2 * ns * ns * (gb + 1) * sizeof(double), s>>>(
          T, rows, ns, c.X, w0, c.Nw, gb, ex + (size_t)sp * nsplit * 2 * c.Nw,
          tr + (size_t)sp * 2 * c.Nw * c.X);
      e = cudaGetLastError();
    }
    ++sp;
  }
  if (e != cudaSuccess) return e;
  k_energy_sum<<<c.Nw, 128, 0, s>>>(c.theta, c.htil, tr, ex, sp, nsplit, NM, c.X, c.Nw, c.eloc);
  return cudaGetLastError();
}

}  // namespace afq
