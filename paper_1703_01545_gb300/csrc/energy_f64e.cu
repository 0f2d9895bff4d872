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
#include "gemm_f64e.cuh"
#include "internal.h"

namespace afq {
namespace {

constexpr size_t kTBytes = (size_t)80 << 20;   // T chunk: leaves L2 room for the digits of the next
constexpr size_t kStage = 40 * 1024;           // staged T of one step of k_exchange
constexpr int kMaxSplit = 16;                  // ranges of g that share a walker's exchange sum
constexpr int kEx = 256;

// Row length of gb staged Cholesky vectors: odd, so that the staging writes spread over the banks too (single
// vectors are staged in their order as they are).
__host__ __device__ constexpr int staged_row(int gb) { return gb > 1 ? gb + 1 : 1; }

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
  const int np = ns * (ns + 1) / 2, gs = staged_row(gb);
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

// Tangent mode: beside ex and tr of T, the derivatives dex = sum_g sum_ab T_ab dT_ba (of half the
// exchange sum) and dtr = sum_a dT_aa, from dT = Ltil dTheta in the same layout.
__global__ void __launch_bounds__(kEx) k_exchange_tan(const double* __restrict__ T, const double* __restrict__ dT,
                                                      int64_t ldt, int ns, int X, int w0, int Nw, int gb,
                                                      double* __restrict__ ex, double* __restrict__ tr) {
  extern __shared__ double sm[];
  __shared__ double red[4 * (kEx / 32)];
  const int wl = blockIdx.x, nwc = gridDim.x, q = blockIdx.y, tid = threadIdx.x, w = w0 + wl;
  const int g0 = (int)((int64_t)X * q / gridDim.y), g1 = (int)((int64_t)X * (q + 1) / gridDim.y);
  const int nsq = ns * ns, gs = staged_row(gb), pl = nsq * gs;   // planes: T re, T im, dT re, dT im
  const int lg = tid & (gb - 1), slot = tid / gb, nslot = kEx / gb;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int gc = g0; gc < g1; gc += gb) {
    const int ng = min(gb, g1 - gc), len = ng * ns;
    __syncthreads();
    for (int col = tid >> 5; col < 4 * ns; col += kEx / 32) {
      const int pp = col / ns, b = col - pp * ns;
      const double* src = (pp >= 2 ? dT : T) + ((int64_t)((pp & 1) * nwc + wl) * ns + b) * ldt + (int64_t)gc * ns;
      for (int k = tid & 31; k < len; k += 32) {
        const int g = k / ns;
        sm[(col * ns + k - g * ns) * gs + g] = src[k];
      }
    }
    __syncthreads();
    if (lg < ng)
      for (int r = slot; r < nsq; r += nslot) {
        const int b = r / ns, a = r - b * ns;
        const double* xy = sm + r * gs + lg;               // (a, b)
        const double* yx = sm + (a * ns + b) * gs + lg;    // (b, a)
        const double xr = xy[0], xi = xy[pl], dr = yx[2 * pl], di = yx[3 * pl];
        acc[2] = fma(xr, dr, fma(-xi, di, acc[2]));
        acc[3] = fma(xr, di, fma(xi, dr, acc[3]));
        if (a <= b) {
          const double f = a == b ? 1.0 : 2.0, yr = f * yx[0], yi = f * yx[pl];
          acc[0] = fma(xr, yr, fma(-xi, yi, acc[0]));
          acc[1] = fma(xr, yi, fma(xi, yr, acc[1]));
        }
      }
    for (int e = tid; e < 4 * ng; e += kEx) {
      const int p = e / ng, g = e - p * ng;
      double t = 0.0;
      for (int a = 0; a < ns; ++a) t += sm[p * pl + (a * ns + a) * gs + g];
      tr[((int64_t)p * Nw + w) * X + gc + g] = t;
    }
  }
  block_sum<4>(acc, red);
  if (tid == 0)
    for (int p = 0; p < 4; ++p) ex[((int64_t)q * 4 + p) * Nw + w] = acc[p];
}

// E_L and dE_L of a walker; tr[spin][4][w][g], ex[spin][range][4][w] as above
__global__ void __launch_bounds__(128) k_energy_sum_tan(const double* __restrict__ theta, const double* __restrict__ dtheta,
                                                        const double* __restrict__ htil, const double* __restrict__ htilP,
                                                        const double* __restrict__ tr, const double* __restrict__ ex,
                                                        int nspin, int nsplit, int NM, int X, int Nw,
                                                        double* __restrict__ eloc, double* __restrict__ deloc) {
  __shared__ double red[4 * 4];
  const int w = blockIdx.x;
  const int64_t plane = (int64_t)Nw * NM, base = (int64_t)w * NM, tp = (int64_t)Nw * X;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int e = threadIdx.x; e < NM; e += 128) {
    const double h = __ldg(htil + e), hp = __ldg(htilP + e), vr = theta[base + e], vi = theta[plane + base + e];
    acc[0] = fma(h, vr, acc[0]);
    acc[1] = fma(h, vi, acc[1]);
    acc[2] = fma(hp, vr, fma(h, dtheta[base + e], acc[2]));
    acc[3] = fma(hp, vi, fma(h, dtheta[plane + base + e], acc[3]));
  }
  for (int g = threadIdx.x; g < X; g += 128) {
    double c[4] = {0.0, 0.0, 0.0, 0.0};
    for (int s = 0; s < nspin; ++s)
      for (int p = 0; p < 4; ++p) c[p] += tr[(4 * s + p) * tp + (int64_t)w * X + g];
    acc[0] = fma(0.5 * c[0], c[0], fma(-0.5 * c[1], c[1], acc[0]));
    acc[1] = fma(c[0], c[1], acc[1]);
    acc[2] = fma(c[0], c[2], fma(-c[1], c[3], acc[2]));
    acc[3] = fma(c[0], c[3], fma(c[1], c[2], acc[3]));
  }
  block_sum<4>(acc, red);
  if (threadIdx.x == 0) {
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    for (int q = 0; q < nspin * nsplit; ++q)
      for (int p = 0; p < 4; ++p) x[p] += ex[((int64_t)q * 4 + p) * Nw + w];
    eloc[w] = acc[0] - 0.5 * x[0];
    eloc[Nw + w] = acc[1] - 0.5 * x[1];
    deloc[w] = acc[2] - x[2];
    deloc[Nw + w] = acc[3] - x[3];
  }
}

// Ltil rows (g, b) of a spin as columns: element (orbital i, k = g ns + b)
struct LtilColumns {
  const double* ltil;
  int ns, n0, N, M;
  __device__ double at(int, int i, int k) const {
    const int g = k / ns;
    return ltil[((int64_t)g * N + n0 + k - g * ns) * M + i];
  }
};

// W[(p, wl, a)][(g, b)] = conj(rhobar_g) delta_ab - conj(T_g[a][b]) as digits, from the chunk's T
// ([(p, wl, b)][(g, a)]) and the traces tr[spin][p][w][g] of both spins.  A CTA per (wl, p): the rows'
// exponents in a first pass, then gb Cholesky vectors at a time staged as [a][(g, b)], so that T is
// read along its rows and the digits are written along theirs.  gb ns is even.
__global__ void __launch_bounds__(256) k_energy_w(const double* __restrict__ T, int64_t ldt, int ns, int X, int w0, int Nw,
                                                  const double* __restrict__ tr, int nspin, int gb, int Kp, int64_t rp,
                                                  uint16_t* __restrict__ out, int* __restrict__ ex) {
  using namespace dig;
  extern __shared__ double sm[];   // [ns][gb ns + 1]
  __shared__ uint32_t smx[32], snan[32];
  __shared__ unsigned long long sfr[32];
  __shared__ int sem[32], smark[32];
  const int wl = blockIdx.x, nwc = gridDim.x, p = blockIdx.y, tid = threadIdx.x, K = X * ns;
  const int lane = tid & 31, warp = tid >> 5, ld = gb * ns + 1;
  const int64_t tsp = 2 * (int64_t)Nw * X, to = ((int64_t)p * Nw + w0 + wl) * X;
  const double* Tw = T + ((int64_t)(p * nwc + wl) * ns) * ldt;
  auto value = [&](int a, int b, int g, double t) -> double {
    double v = p ? t : -t;
    if (a == b) {
      double rho = 0.0;
      for (int s = 0; s < nspin; ++s) rho += tr[s * tsp + to + g];
      v += p ? -rho : rho;
    }
    return v;
  };
  if (tid < 32) {
    smx[tid] = snan[tid] = 0u;
    sfr[tid] = 0ull;
  }
  __syncthreads();
  for (int b = 0; b < ns; ++b)
    for (int r = tid; r < K; r += 256) {
      const int g = r / ns, a = r - g * ns;
      const double x = value(a, b, g, Tw[(int64_t)b * ldt + r]);
      uint32_t mx = 0, nan = 0;
      row_scan(x, mx, nan);
      if (mx > smx[a]) atomicMax(&smx[a], mx);
      if (nan) snan[a] = 1u;
      if ((mx >> 20) == 0) atomicMax(&sfr[a], (unsigned long long)fraction_of(x));
    }
  __syncthreads();
  if (tid < ns) {
    const uint32_t mx = smx[tid] >> 20;
    const int em = mx ? (int)mx : sfr[tid] ? 12 - __clzll((long long)sfr[tid]) : 1;
    sem[tid] = em;
    smark[tid] = snan[tid] ? kExpNaN : mx == 0x7ffu ? kExpInf : em;
    ex[(int64_t)(p * nwc + wl) * ns + tid] = smark[tid];
  }
  for (int k0 = 0; k0 < Kp; k0 += gb * ns) {
    const int g0 = k0 / ns, len = min(gb * ns, Kp - k0);   // (the last step pads K with zeros)
    __syncthreads();
    for (int b = warp; b < ns; b += 8)
      for (int r = lane; r < gb * ns; r += 32) {
        const int g = r / ns, a = r - g * ns;
        sm[a * ld + g * ns + b] = g0 + g < X ? value(a, b, g0 + g, Tw[(int64_t)b * ldt + (int64_t)g0 * ns + r]) : 0.0;
      }
    __syncthreads();
    for (int a = warp; a < ns; a += 8)
      for (int k = 2 * lane; k < len; k += 64) {
        uint32_t x[2], y[2];
        digit_bytes_of(sm[a * ld + k], sem[a], smark[a] >= kExpInf, x[0], x[1]);
        digit_bytes_of(sm[a * ld + k + 1], sem[a], smark[a] >= kExpInf, y[0], y[1]);
        const int64_t row = (int64_t)(p * nwc + wl) * ns + a;
#pragma unroll
        for (int j = 0; j < kDig; ++j)
          *reinterpret_cast<uint32_t*>(out + ((int64_t)j * rp + row) * Kp + k0 + k) = digit_pair(j, x, y);
      }
  }
}

// thb[(p, w, n0 + a)][i] = ebar_w (htil[n0 + a][i] (real plane) + G[(p, wl, a)][i]), 0 for walkers out
// of the sweep
__global__ void __launch_bounds__(256) k_energy_thb(const double* __restrict__ G, const double* __restrict__ htil,
                                                    const double* __restrict__ ebar, const int* __restrict__ mask,
                                                    int ns, int n0, int N, int M, int w0, int nwc, int Nw,
                                                    double* __restrict__ thb) {
  const int64_t total = 2 * (int64_t)nwc * ns * M;
  for (int64_t e = blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256) {
    const int i = (int)(e % M), a = (int)(e / M % ns), wl = (int)(e / ((int64_t)M * ns) % nwc);
    const int p = (int)(e / ((int64_t)M * ns * nwc)), w = w0 + wl;
    const double v = mask[w] ? ebar[w] * (p ? G[e] : G[e] + htil[(n0 + a) * M + i]) : 0.0;
    thb[(((int64_t)p * Nw + w) * N + n0 + a) * M + i] = v;
  }
}

__global__ void k_energy_masked(const double* __restrict__ el, const int* __restrict__ mask, int Nw,
                                double* __restrict__ eloc) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w < Nw) eloc[w] = mask[w] ? el[w] : 0.0;
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

// Tangent mode: T and dT share the T chunk of c.e64, half of its walkers each; c.e64_tan holds the traces of
// both and both spins, then the exchange sums.  A chunk of one walker has no room for its dT (one walker in
// all, or a T above half of kTBytes), which then follows the sums in c.e64_tan.
struct TanPlace {
  int nwc;                    // walkers at a time
  size_t len, ex, dt;         // doubles of T; offsets in c.e64_tan of the sums, and of dT or the end
  bool own;                   // dT in c.e64_tan
};
static TanPlace tan_place(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up), chunk = chunk_walkers(c);
  TanPlace t;
  t.own = chunk < 2;
  t.nwc = t.own ? 1 : chunk / 2;
  t.len = 2 * (size_t)c.X * ns * ns * t.nwc;
  t.ex = 8 * (size_t)c.Nw * c.X;
  t.dt = t.ex + 8 * (size_t)kMaxSplit * c.Nw;
  return t;
}
size_t energy_tan_f64e_scratch(const Ctx& c) {
  const TanPlace t = tan_place(c);
  return sizeof(double) * (t.dt + (t.own ? t.len : 0));
}
// doubles at the head of c.e64 that hold T of a chunk, and that tangent mode fills with T and dT
int64_t energy_chunk_doubles(const Ctx& c, bool tangent) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  if (!tangent) return 2 * (int64_t)c.X * ns * ns * chunk_walkers(c);
  const TanPlace t = tan_place(c);
  return (int64_t)(t.own ? t.len : 2 * t.len);
}
size_t energy_f64e_ws(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  return digit_bytes((int64_t)c.X * ns, c.M) + digit_bytes(2 * (int64_t)chunk_walkers(c) * ns, c.M);
}

namespace {

// T of one spin for walkers w0 .. w0 + nw - 1; `cols` memory for the columns' digits
cudaError_t products_of(const Ctx& c, const F64Ws& ws, const double* theta, const DigitOp& da, void* cols, int n0,
                        int ns, int w0, int nw, double* T, cudaStream_t s) {
  const int NM = c.N * c.M, nc = 2 * nw * ns, rows = c.X * ns;
  const DigitOp db = digit_place(cols, nc, c.M);
  for (int p = 0; p < 2; ++p) {
    DigitOp dp = db;
    dp.dig += (int64_t)p * nw * ns * db.Kp;
    dp.ex += p * nw * ns;
    const cudaError_t e = digits_of(theta + ((int64_t)p * c.Nw + w0) * NM, c.M, nw * ns, c.M, dp, s, ns, c.N, n0);
    if (e != cudaSuccess) return e;
  }
  DigitGemm g;
  g.R = rows;
  g.Cn = nc;
  g.out = T;
  g.ldc = rows;
  g.K = c.M;
  g.err = ws.err;
  return digit_gemm(da, db, g, s);
}

// Cholesky vectors staged at a time by the exchange kernels: a power of two within kStage.  A single one takes
// 32 KB at most (4 planes, ns = 32), so no launch asks for more than the 48 KB that need no attribute.
size_t staged_bytes(int ns, int planes, int gb) { return (size_t)planes * ns * ns * staged_row(gb) * sizeof(double); }
int staged(int ns, int planes) {
  int gb = 32;
  while (gb > 1 && staged_bytes(ns, planes, gb) > kStage) gb /= 2;
  return gb;
}

// T of a spin and from it the exchange sums and traces (spin index sp)
cudaError_t chunk_of(const Ctx& c, const F64Ws& ws, const double* theta, const DigitOp& da, void* cols, int sp, int n0,
                     int ns, int w0, int nw, int nsplit, double* T, double* tr, double* ex, cudaStream_t s) {
  const cudaError_t e = products_of(c, ws, theta, da, cols, n0, ns, w0, nw, T, s);
  if (e != cudaSuccess) return e;
  const int gb = staged(ns, 2);
  k_exchange<<<dim3(nw, nsplit), kEx, staged_bytes(ns, 2, gb), s>>>(
      T, c.X * ns, ns, c.X, w0, c.Nw, gb, ex + (size_t)sp * nsplit * 2 * c.Nw, tr + (size_t)sp * 2 * c.Nw * c.X);
  return cudaGetLastError();
}

}  // namespace

int64_t exchange_smem(int ns, bool tangent) { return (int64_t)staged_bytes(ns, tangent ? 4 : 2, staged(ns, tangent ? 4 : 2)); }

// E_L and dE_L of every walker from Theta and dTheta (tangent mode)
cudaError_t launch_energy_tan_f64e(const Ctx& c, cudaStream_t s) {
  const TanPlace at = tan_place(c);
  const int NM = c.N * c.M, nwc = at.nwc, nsplit = splits(c, nwc);
  double* T = c.e64;
  double* dT = at.own ? c.e64_tan + at.dt : T + at.len;
  double* tr = c.e64_tan;
  double* ex = tr + at.ex;
  cudaError_t e = cudaSuccess;
  int sp = 0;
  for (int s0 = 0; s0 < 2 && e == cudaSuccess; ++s0) {
    const int n0 = s0 ? c.n_up : 0, ns = s0 ? c.N - c.n_up : c.n_up;
    if (ns == 0) continue;
    const DigitOp da = digit_place(c.ws64.buf, c.X * ns, c.M);
    uint8_t* cols = c.ws64.buf + digit_bytes(c.X * ns, c.M);
    e = digits_of(c.Ltil, c.M, c.X * ns, c.M, da, s, ns, c.N, n0);
    for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += nwc) {
      const int nw = std::min(nwc, c.Nw - w0), gb = staged(ns, 4);
      e = products_of(c, c.ws64, c.theta, da, cols, n0, ns, w0, nw, T, s);
      if (e == cudaSuccess) e = products_of(c, c.ws64, c.dtheta, da, cols, n0, ns, w0, nw, dT, s);
      if (e != cudaSuccess) break;
      k_exchange_tan<<<dim3(nw, nsplit), kEx, staged_bytes(ns, 4, gb), s>>>(
          T, dT, c.X * ns, ns, c.X, w0, c.Nw, gb, ex + (size_t)sp * nsplit * 4 * c.Nw,
          tr + (size_t)sp * 4 * c.Nw * c.X);
      e = cudaGetLastError();
    }
    ++sp;
  }
  if (e != cudaSuccess) return e;
  k_energy_sum_tan<<<c.Nw, 128, 0, s>>>(c.theta, c.dtheta, c.htil, c.htilP, tr, ex, sp, nsplit, NM, c.X, c.Nw, c.eloc,
                                        c.deloc);
  return cudaGetLastError();
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
    const DigitOp da = digit_place(c.ws64.buf, c.X * ns, c.M);
    e = digits_of(c.Ltil, c.M, c.X * ns, c.M, da, s, ns, c.N, n0);
    for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += nwc)
      e = chunk_of(c, c.ws64, c.theta, da, c.ws64.buf + digit_bytes(c.X * ns, c.M), sp, n0, ns, w0,
                   std::min(nwc, c.Nw - w0), nsplit, T, tr, ex, s);
    ++sp;
  }
  if (e != cudaSuccess) return e;
  k_energy_sum<<<c.Nw, 128, 0, s>>>(c.theta, c.htil, tr, ex, sp, nsplit, NM, c.X, c.Nw, c.eloc);
  return cudaGetLastError();
}

// Reverse: T of both spins of a chunk, W and Ltil's columns as digits, G and its partial sums.
namespace {
constexpr size_t kRevPart = (size_t)64 << 20;
// walkers whose T (both spins) takes 320 MB at most: the reverse reads it twice only, and needs as
// many (walker, plane) CTAs as there are SMs
int rev_chunk(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up);
  const size_t per = 4 * (size_t)c.X * ns * ns * sizeof(double);
  return (int)std::max<size_t>(1, std::min<size_t>((size_t)c.Nw, ((size_t)320 << 20) / per));
}
}  // namespace

size_t energy_rev_f64e_scratch(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up), nwc = rev_chunk(c);
  return sizeof(double) * (4 * (size_t)c.X * ns * ns * nwc + 2 * (size_t)nwc * ns * c.M + 4 * (size_t)c.Nw * c.X +
                           4 * (size_t)kMaxSplit * c.Nw + 2 * (size_t)c.Nw) + kRevPart;
}

size_t energy_rev_f64e_ws(const Ctx& c) {
  const int ns = std::max(c.n_up, c.N - c.n_up), nwc = rev_chunk(c);
  return 2 * digit_bytes((int64_t)c.X * ns, c.M) + 2 * digit_bytes(c.M, c.X * ns) +
         std::max(digit_bytes(2 * (int64_t)nwc * ns, c.M), digit_bytes(2 * (int64_t)nwc * ns, c.X * ns));
}

// 15.7 ms in the walker kernel (k_energy_rev) at M = 96, X = 480, 12/12, 128 walkers, 3.6 ms here.
// E_L of every walker and thb = ebar (htil + sum_g conj(rhobar_g) Ltil_g - sum_g conj(T_g) Ltil_g), the
// second product as one contraction over (g, b).
cudaError_t launch_energy_rev_f64e(const Ctx& c, const F64Ws& ws, double* scratch, const double* theta,
                                   const double* ebar, double* thb, double* eloc, const int* mask, cudaStream_t s) {
  const int NM = c.N * c.M, nwc = rev_chunk(c), nsmax = std::max(c.n_up, c.N - c.n_up);
  const int nsplit = splits(c, nwc);
  const size_t tlen = 2 * (size_t)c.X * nsmax * nsmax * nwc;
  double* part = scratch;
  double* T[2] = {part + kRevPart / sizeof(double), part + kRevPart / sizeof(double) + tlen};
  double* G = T[1] + tlen;
  double* tr = G + 2 * (size_t)nwc * nsmax * c.M;
  double* ex = tr + 4 * (size_t)c.Nw * c.X;
  double* el = ex + 4 * (size_t)kMaxSplit * c.Nw;
  uint8_t* at = ws.buf;
  DigitOp da[2], dl[2];
  int n0s[2], nss[2], nspin = 0;
  cudaError_t e = cudaSuccess;
  for (int s0 = 0; s0 < 2 && e == cudaSuccess; ++s0) {
    const int n0 = s0 ? c.n_up : 0, ns = s0 ? c.N - c.n_up : c.n_up;
    if (ns == 0) continue;
    const int rows = c.X * ns;
    n0s[nspin] = n0;
    nss[nspin] = ns;
    da[nspin] = digit_place(at, rows, c.M);
    at += digit_bytes(rows, c.M);
    dl[nspin] = digit_place(at, c.M, rows);
    at += digit_bytes(c.M, rows);
    e = digits_of(c.Ltil, c.M, rows, c.M, da[nspin], s, ns, c.N, n0);
    if (e != cudaSuccess) break;
    const LtilColumns f{c.Ltil, ns, n0, c.N, c.M};
    dig::k_strided_digits<<<dim3(1, (c.M + 31) / 32), 1024, 0, s>>>(
        f, c.M, rows, dl[nspin].Kp, dl[nspin].rp, c.M, 0, reinterpret_cast<uint16_t*>(dl[nspin].dig), dl[nspin].ex);
    e = cudaGetLastError();
    ++nspin;
  }
  for (int w0 = 0; w0 < c.Nw && e == cudaSuccess; w0 += nwc) {
    const int nw = std::min(nwc, c.Nw - w0);
    for (int sp = 0; sp < nspin && e == cudaSuccess; ++sp)
      e = chunk_of(c, ws, theta, da[sp], at, sp, n0s[sp], nss[sp], w0, nw, nsplit, T[sp], tr, ex, s);
    for (int sp = 0; sp < nspin && e == cudaSuccess; ++sp) {
      const int ns = nss[sp], rows = c.X * ns;
      const DigitOp dw = digit_place(at, 2 * nw * ns, rows);
      // staged vectors: an even number (gb ns has to be even) within kStage
      const int gb = std::max(2, (int)(kStage / (sizeof(double) * ns * ns)) / 2 * 2);
      const int gs = std::min(gb, 32);
      k_energy_w<<<dim3(nw, 2), 256, sizeof(double) * ns * ((size_t)gs * ns + 1), s>>>(T[sp], rows, ns, c.X, w0, c.Nw, tr, nspin, gs, dw.Kp, dw.rp,
                                             reinterpret_cast<uint16_t*>(dw.dig), dw.ex);
      if ((e = cudaGetLastError()) != cudaSuccess) break;
      DigitGemm g;
      g.R = 2 * nw * ns;
      g.Cn = c.M;
      g.swap = 1;
      g.out = G;
      g.ldc = c.M;
      g.K = rows;
      g.err = ws.err;
      if ((e = digit_gemm_sum(dw, dl[sp], g, part, kRevPart, s)) != cudaSuccess) break;
      const int64_t total = 2 * (int64_t)nw * ns * c.M;
      k_energy_thb<<<(int)std::min<int64_t>((total + 255) / 256, 152 * 8), 256, 0, s>>>(
          G, c.htil, ebar, mask, ns, n0s[sp], c.N, c.M, w0, nw, c.Nw, thb);
      e = cudaGetLastError();
    }
  }
  if (e != cudaSuccess) return e;
  k_energy_sum<<<c.Nw, 128, 0, s>>>(theta, c.htil, tr, ex, nspin, nsplit, NM, c.X, c.Nw, el);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_energy_masked<<<(c.Nw + 255) / 256, 256, 0, s>>>(el, mask, c.Nw, eloc);
  return cudaGetLastError();
}

}  // namespace afq
