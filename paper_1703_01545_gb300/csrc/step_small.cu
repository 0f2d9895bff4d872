// Whole FP64 steps of small systems (M <= 16, spin blocks of at most 8): one CTA per walker runs up to
// kSteps propagation steps (Eqs. 3-5, 8-9, 11 and the hybrid weight) out of shared memory, in place of
// eight kernels per step.
//
// At these sizes a step is latency: some ten thousand multiply-adds per walker, in kernels of 3 to 13 us
// each.  What sets a kernel's time is that GB300 issues an FP64 instruction of a warp every 64 cycles per
// scheduler whatever its active lanes, so
//   * every product is spread over all 4 warps (S lanes per output, combined by shuffles),
//   * the normals of all steps are drawn at once (one lane per pair and step: a Box-Muller chain of about
//     100 FP64 instructions is paid once per launch, not per step),
//   * the logarithm, phase, exponential and cosine of the weights are taken for all steps at once, one
//     lane per step, after the steps: a step that kills the walker is found then, and the walker is put
//     back to that step's determinant (every step's is kept in shared memory).  The steps computed
//     beyond it are dropped.
// Constants (packed Cholesky tensor, half-rotated tensor, e^{-dt K/2}, trial) are staged once per launch.
// Still bound by the chains of dependent FP64 instructions (a term of the series about 2 us with two CTAs on
// an SM, the LU of a 2 x 2 block 5 us).  M = 8, X = 24, 2/2, 128 walkers: 16 us a step (51 us of eight
// kernels); the pair with 2/1, 40 steps and 8 measurements: 2.83 -> 1.51 ms.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "device_util.cuh"
#include "internal.h"
#include "lu_warp.cuh"

namespace afq {
namespace {

constexpr int kSteps = 8;      // steps per launch at most
constexpr int kT = 128;
constexpr int kNs = 8;         // largest spin block
constexpr int kSpin = 2 * kNs * kNs;   // LU factors of a spin: re, im [kNs][kNs]

struct SmallArgs {
  const double *Lt, *Ltil, *expK, *psi, *rho;   // [P][X], [X][N][M], [M][M], [N][M], [X]
  const double* fields;                         // [n][Nw][X] or null
  double *phi, *theta, *logO, *w;
  int *alive, *flags;
  const unsigned long long* step;
  uint2 key;
  uint32_t k0;
  int M, N, nu, X, P, Nw, n, order, free_proj;
  double sqrt_dt, fb_cap, log_shift;
};

// Shared memory, in doubles.
struct Lay {
  int lt, ltil, ek, psi, rho, x, u, q, rb, a, t0, t1, acc, snap, lu, aux, det, total;
  int ldx, ldn, ldm, nm2;
};
__host__ __device__ inline Lay layout(int M, int N, int X, int P, int n) {
  Lay l;
  l.ldx = X | 1;            // odd rows: the lanes of an output's neighbours read distinct banks
  l.ldn = (N * M) | 1;
  l.ldm = M | 1;
  l.nm2 = 2 * N * M;
  int o = 0;
  auto take = [&](int k) { const int r = o; o += k; return r; };
  l.lt = take(P * l.ldx);
  l.ltil = take(X * l.ldn);
  l.ek = take(M * l.ldm);
  l.psi = take(N * M);
  l.rho = take(X);
  l.x = take(n * X);        // fields of all steps
  l.u = take(2 * X);
  l.q = take(4 * X);        // terms of the four sums
  l.rb = take(2 * X);
  l.a = take(2 * M * l.ldm);
  l.t0 = take(l.nm2);
  l.t1 = take(l.nm2);
  l.acc = take(l.nm2);
  l.snap = take((n + 1) * 2 * l.nm2);   // per step (0: before the first): Phi, Theta
  l.lu = take(2 * kSpin);
  l.aux = take(4 * n);
  l.det = take(8 * n);      // det mantissas of both spins, exponent, singular
  l.total = o;
  return l;
}

__device__ __forceinline__ double sum_lanes(double v, int S) {
  for (int o = 1; o < S; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Lanes per output: as many as the block has for `count` outputs, a power of two up to 8.
__device__ __forceinline__ int lanes_for(int count) {
  int S = 1;
  while (S < 8 && 2 * S * count <= kT) S *= 2;
  return S;
}

// NS: both spin blocks' size at most (2, 4 or 8).  The solves are unrolled to it, and what is beyond a
// lane's block still takes its FP64 issue slots: a step at 2/2 and 128 walkers takes 19 us in the form for 8
// and 16 us in this one.
template <int NS>
__global__ void __launch_bounds__(kT) k_steps_small(const SmallArgs g) {
  extern __shared__ double sm[];
  __shared__ int s_piv[2][16], s_last;
  __shared__ unsigned char s_i[160], s_j[160];
  __shared__ double s_inv[65];   // 1 / m: a division costs every warp of the CTA some ten FP64 instructions
  const int wk = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M = g.M, N = g.N, X = g.X, P = g.P, NM = N * M, nu = g.nu, nd = N - nu, n = g.n;
  if (!g.alive[wk]) return;   // a dead walker does not change (nor its Theta and log O)
  const Lay l = layout(M, N, X, P, n);
  const int64_t plane = (int64_t)g.Nw * NM, base = (int64_t)wk * NM;
  const uint32_t t0 = (uint32_t)(*g.step);
  // ---- constants, walker, fields ----
  for (int e = tid; e < P * X; e += kT) sm[l.lt + (e / X) * l.ldx + e % X] = g.Lt[e];
  if (!g.free_proj)
    for (int e = tid; e < X * NM; e += kT) sm[l.ltil + (e / NM) * l.ldn + e % NM] = g.Ltil[e];
  for (int e = tid; e < M * M; e += kT) sm[l.ek + (e / M) * l.ldm + e % M] = g.expK[e];
  for (int e = tid; e < NM; e += kT) {
    sm[l.psi + e] = g.psi[e];
    sm[l.snap + e] = g.phi[base + e];
    sm[l.snap + NM + e] = g.phi[plane + base + e];
    sm[l.snap + l.nm2 + e] = g.theta[base + e];
    sm[l.snap + l.nm2 + NM + e] = g.theta[plane + base + e];
  }
  for (int e = tid; e < X; e += kT) sm[l.rho + e] = g.rho[e];
  if (tid < g.order) s_inv[tid + 1] = 1.0 / (double)(tid + 1);
  for (int e = tid; e < P; e += kT) {   // packed index -> (i, j), i <= j
    int i = 0, r = e;
    while (r >= M - i) r -= M - i++;
    s_i[e] = (unsigned char)i;
    s_j[e] = (unsigned char)(i + r);
  }
  const int npair = (X + 1) / 2;
  for (int e = tid; e < n * npair; e += kT) {
    const int t = e / npair, j = e - t * npair;
    double z[2];
    if (g.fields) {
      const double* f = g.fields + ((int64_t)t * g.Nw + wk) * X;
      z[0] = f[2 * j];
      z[1] = 2 * j + 1 < X ? f[2 * j + 1] : 0.0;
    } else {
      philox_normal2(philox4x32_10(make_uint4((uint32_t)j, g.k0 + (uint32_t)wk, t0 + (uint32_t)t, 0u), g.key), z[0],
                     z[1]);
    }
    sm[l.x + t * X + 2 * j] = z[0];
    if (2 * j + 1 < X) sm[l.x + t * X + 2 * j + 1] = z[1];
  }
  __syncthreads();

  // out(o, sum_k term(o, k)) for o < count: S lanes per output (0: as many as there are), whole warps
  // without outputs skipped
  auto outputs = [&](int count, int K, int S, auto term, auto out) {
    if (S == 0) S = lanes_for(count);
    for (int b = 0; b < count * S; b += kT) {
      if (b + (tid & ~31) >= count * S) break;
      const int o = (b + tid) / S, part = (b + tid) & (S - 1);
      double v = 0.0;
      if (o < count)
        for (int k = part; k < K; k += S) v = term(o, k, v);
      v = sum_lanes(v, S);
      if (o < count && part == 0) out(o, v);
    }
  };

  for (int t = 0; t < n; ++t) {
    const double* phi = sm + l.snap + t * 2 * l.nm2;
    const double* th = phi + l.nm2;
    double* phn = sm + l.snap + (t + 1) * 2 * l.nm2;
    double* thn = phn + l.nm2;
    // rhobar_g (Eq. 9)
    if (!g.free_proj) {
      outputs(2 * X, NM, 0,
              [&](int o, int k, double v) { return fma(sm[l.ltil + (o >> 1) * l.ldn + k], th[(o & 1) * NM + k], v); },
              [&](int o, double v) { sm[l.rb + (o & 1) * X + (o >> 1)] = v; });
      __syncthreads();
    }
    // force bias, shifted fields, U = i sqrt(dt) c, and the terms of c.<rho> and x.xbar - xbar^2 / 2
    for (int e = tid; e < X; e += kT) {
      const double x = sm[l.x + t * X + e], rm = sm[l.rho + e];
      double xr = 0.0, xi = 0.0;
      if (!g.free_proj) {
        xr = g.sqrt_dt * sm[l.rb + X + e];
        xi = -g.sqrt_dt * (sm[l.rb + e] - rm);
        if (g.fb_cap > 0.0) {
          const double m2 = xr * xr + xi * xi;
          if (m2 > g.fb_cap * g.fb_cap) {
            const double sc = g.fb_cap / sqrt(m2);
            xr *= sc;
            xi *= sc;
          }
        }
      }
      const double cr = x - xr, ci = -xi;
      sm[l.u + e] = -g.sqrt_dt * ci;
      sm[l.u + X + e] = g.sqrt_dt * cr;
      sm[l.q + e] = cr * rm;
      sm[l.q + X + e] = ci * rm;
      sm[l.q + 2 * X + e] = x * xr - 0.5 * (xr * xr - xi * xi);
      sm[l.q + 3 * X + e] = x * xi - xr * xi;
    }
    __syncthreads();
    {   // warp q adds the q-th terms
      double v = 0.0;
      for (int e = lane; e < X; e += 32) v += sm[l.q + warp * X + e];
      v = sum_lanes(v, 32);
      if (lane == 0) sm[l.aux + 4 * t + warp] = v;
    }
    // A = sum_g U_g L_g (Eq. 11), both halves of the symmetric matrix
    outputs(2 * P, X, 0,
            [&](int o, int k, double v) { return fma(sm[l.lt + (o >> 1) * l.ldx + k], sm[l.u + (o & 1) * X + k], v); },
            [&](int o, double v) {
              double* a = sm + l.a + (o & 1) * M * l.ldm;
              const int i = s_i[o >> 1], j = s_j[o >> 1];
              a[i * l.ldm + j] = v;
              a[j * l.ldm + i] = v;
            });
    // e^{-dt K/2} Phi
    auto onebody = [&](const double* src, double* dst, double* dst2) {
      outputs(2 * NM, M, 0,
              [&](int o, int k, double v) {
                const int r = o % NM, i = r % M;
                return fma(sm[l.ek + i * l.ldm + k], src[o - i + k], v);
              },
              [&](int o, double v) {
                dst[o] = v;
                if (dst2) dst2[o] = v;
              });
    };
    onebody(phi, sm + l.t0, sm + l.acc);
    __syncthreads();
    // Taylor terms: an output's lanes share the sum over j; lane 0 keeps its real part, lane 1 (or 0)
    // its imaginary part
    double* cur = sm + l.t0;
    double* nxt = sm + l.t1;
    const int S = lanes_for(NM);
    for (int m = 1; m <= g.order; ++m) {
      const double inv = s_inv[m];
      for (int b = 0; b < NM * S; b += kT) {
        if (b + (tid & ~31) >= NM * S) break;
        const int o = (b + tid) / S, part = (b + tid) & (S - 1);
        double sr = 0.0, si = 0.0;
        if (o < NM) {
          const int i = o % M;
          const double* ar = sm + l.a + i * l.ldm;
          const double* ai = ar + M * l.ldm;
          const double* tr = cur + (o - i);
          for (int j = part; j < M; j += S) {
            sr = fma(ar[j], tr[j], fma(-ai[j], tr[NM + j], sr));
            si = fma(ar[j], tr[NM + j], fma(ai[j], tr[j], si));
          }
        }
        sr = sum_lanes(sr, S);
        si = sum_lanes(si, S);
        if (o < NM && part < 2) {
          for (int c = part; c < 2; c += S > 1 ? 2 : 1) {
            const double v = (c ? si : sr) * inv;
            nxt[c * NM + o] = v;
            sm[l.acc + c * NM + o] += v;
          }
        }
      }
      __syncthreads();
      double* x = cur;
      cur = nxt;
      nxt = x;
    }
    onebody(sm + l.acc, phn, nullptr);
    __syncthreads();
    // O_s = Psi_s^T Phi_s, by 4 lanes an entry, as k_overlap64: O, its factors and Theta then have the bits
    // that a refresh of the same walker gives
    const int nn = nu * nu + nd * nd;
    outputs(2 * nn, M, 4,
            [&](int o, int k, double v) {
              const int p = o & 1, e = o >> 1, sp = e >= nu * nu, ns = sp ? nd : nu, e2 = sp ? e - nu * nu : e;
              const int n0 = sp ? nu : 0;
              return fma(sm[l.psi + (n0 + e2 / ns) * M + k], phn[p * NM + (n0 + e2 % ns) * M + k], v);
            },
            [&](int o, double v) {
              const int p = o & 1, e = o >> 1, sp = e >= nu * nu, ns = sp ? nd : nu, e2 = sp ? e - nu * nu : e;
              sm[l.lu + sp * kSpin + p * kNs * kNs + (e2 / ns) * kNs + e2 % ns] = v;
            });
    __syncthreads();
    if (warp == 0) {   // both spin blocks, 16 lanes each
      const int h = lane >> 4, l16 = lane & 15, ns = h ? nd : nu;
      double* ar = sm + l.lu + h * kSpin;
      double dr, di;
      int dexp;
      bool bad;
      lu_block<16, (NS > 4 ? 4 : 1), kNs>(ar, ar + kNs * kNs, l16, ns, nu > nd ? nu : nd, s_piv[h], dr, di, dexp, bad);
      if (l16 == 0) {
        double* d = sm + l.det + 8 * t;
        d[2 * h] = dr;
        d[2 * h + 1] = di;
        d[4 + h] = (double)dexp;
        d[6 + h] = bad ? 1.0 : 0.0;
      }
    }
    __syncthreads();
    const bool bad = sm[l.det + 8 * t + 6] != 0.0 || sm[l.det + 8 * t + 7] != 0.0;
    // Theta_s = Phi_s O_s^{-1}: y U = phi_i, z L = y, theta_i[perm[j]] = z_j
    for (int e = tid; e < 2 * M; e += kT) {
      const int sp = e / M, i = e - sp * M, ns = sp ? nd : nu, n0 = sp ? nu : 0;
      const double* Lr = sm + l.lu + sp * kSpin;
      const double* Li = Lr + kNs * kNs;
      unsigned perm = 0x76543210u;   // row j of P O is row (perm >> 4 j) & 15 of O
      if (!bad)
        for (int k = 0; k < ns; ++k) {
          const int p = s_piv[sp][k];
          const unsigned x = (perm >> (4 * k)) & 15u, y = (perm >> (4 * p)) & 15u;
          perm ^= ((x ^ y) << (4 * k)) | ((x ^ y) << (4 * p));
        }
      double yr[NS], yi[NS];
#pragma unroll
      for (int j = 0; j < NS; ++j)
        if (j < ns) {
          yr[j] = phn[(n0 + j) * M + i];
          yi[j] = phn[NM + (n0 + j) * M + i];
        }
#pragma unroll
      for (int j = 1; j < NS; ++j)
        if (j < ns) {
#pragma unroll
          for (int k = 0; k < j; ++k) {
            const double ur = Lr[k * kNs + j], ui = Li[k * kNs + j];
            yr[j] = fma(-yr[k], ur, fma(yi[k], ui, yr[j]));
            yi[j] = fma(-yr[k], ui, fma(-yi[k], ur, yi[j]));
          }
        }
#pragma unroll
      for (int j = NS - 1; j >= 0; --j)
        if (j < ns) {
          double tr = yr[j], ti = yi[j];
#pragma unroll
          for (int k = j + 1; k < NS; ++k)
            if (k < ns) {
              const double lr = Lr[k * kNs + j], li = Li[k * kNs + j];
              tr = fma(-yr[k], lr, fma(yi[k], li, tr));
              ti = fma(-yr[k], li, fma(-yi[k], lr, ti));
            }
          const double qr = Lr[j * kNs + j], qi = Li[j * kNs + j];
          yr[j] = fma(tr, qr, -ti * qi);
          yi[j] = fma(tr, qi, ti * qr);
        }
#pragma unroll
      for (int j = 0; j < NS; ++j)
        if (j < ns) {
          const int c = n0 + (int)((perm >> (4 * j)) & 15u);
          thn[c * M + i] = bad ? 0.0 : yr[j];
          thn[NM + c * M + i] = bad ? 0.0 : yi[j];
        }
    }
    __syncthreads();
  }

  // ---- weights of all steps by one warp, lane t for step t ----
  if (warp == 0) {
    double ld_re, ld_im, f_re, f_im = 0.0;
    const int t = lane < n ? lane : 0;
    const double* d = sm + l.det + 8 * t;
    const double* q = sm + l.aux + 4 * t;
    bool bad = d[6] != 0.0 || d[7] != 0.0;
    const double pr = fma(d[0], d[2], -d[1] * d[3]), pi = fma(d[0], d[3], d[1] * d[2]);
    ld_re = fma(d[4] + d[5], M_LN2, 0.5 * log(fma(pr, pr, pi * pi)));
    ld_im = atan2(pi, pr);
    bad = bad || !isfinite(ld_re) || !isfinite(ld_im);
    double pv_re = __shfl_up_sync(0xffffffffu, ld_re, 1), pv_im = __shfl_up_sync(0xffffffffu, ld_im, 1);
    if (lane == 0) {
      pv_re = g.logO[wk];
      pv_im = g.logO[g.Nw + wk];
    }
    // log s = sqrt(dt) (S_im - i S_re)
    const double lr_re = g.sqrt_dt * q[1] + ld_re - pv_re, lr_im = -g.sqrt_dt * q[0] + ld_im - pv_im;
    const double mag = exp(lr_re + q[2] + g.log_shift);
    if (g.free_proj) {
      double sn, cs;
      sincos(lr_im + q[3], &sn, &cs);
      f_re = mag * cs;
      f_im = mag * sn;
    } else {
      f_re = mag * fmax(0.0, cos(lr_im));
    }
    double w_re = g.w[wk], w_im = g.w[g.Nw + wk];
    int last = n, alive = 1, sing = 0;
    for (int t = 0; t < n; ++t) {
      const double fr = __shfl_sync(0xffffffffu, f_re, t), fi = __shfl_sync(0xffffffffu, f_im, t);
      if (__shfl_sync(0xffffffffu, (int)bad, t)) {
        w_re = w_im = 0.0;
        alive = 0;
        sing = 1;
        last = t + 1;
        break;
      }
      if (g.free_proj) {
        const cplx v = cmul({w_re, w_im}, {fr, fi});
        w_re = v.re;
        w_im = v.im;
      } else {
        w_re *= fr;
        w_im = 0.0;
        if (!(w_re > 0.0)) {
          w_re = 0.0;
          alive = 0;
          last = t + 1;
          break;
        }
      }
    }
    // log O of the last step taken (a singular one leaves the step's before it)
    const int src = last - 1 - sing;
    const double out_re = __shfl_sync(0xffffffffu, ld_re, max(src, 0)), out_im = __shfl_sync(0xffffffffu, ld_im, max(src, 0));
    if (lane == 0) {
      s_last = last;
      if (src >= 0) {
        g.logO[wk] = out_re;
        g.logO[g.Nw + wk] = out_im;
      }
      g.w[wk] = w_re;
      g.w[g.Nw + wk] = w_im;
      if (!alive) g.alive[wk] = 0;
      if (sing) atomicAdd(g.flags, 1);
    }
  }
  __syncthreads();
  const int last = s_last;
  for (int e = tid; e < NM; e += kT) {
    const double* p = sm + l.snap + last * 2 * l.nm2;
    g.phi[base + e] = p[e];
    g.phi[plane + base + e] = p[NM + e];
    g.theta[base + e] = p[l.nm2 + e];
    g.theta[plane + base + e] = p[l.nm2 + NM + e];
  }
}

SmemLimits g_small_limits;

}  // namespace

// M <= 16 and blocks of at most 8, with the constants and kSteps snapshots within 96 KB (two CTAs per SM).
bool step_small_ok(const Ctx& c) {
  return c.opt.precision == AFQMC_FP64 && c.n_det == 0 && c.M <= 16 && c.n_up <= kNs && c.N - c.n_up <= kNs &&
         c.X >= 1 && c.X <= 4096 && sizeof(double) * (size_t)layout(c.M, c.N, c.X, (int)c.P, kSteps).total <= 96 * 1024;
}

// Whether a call of n steps takes this kernel, of a handle that can.  A few waves of CTAs are latency, where it
// beats the separate kernels two to four times.  Beyond, it pays per walker and step (the separate kernels:
// 65 to 75 us plus 46 ns at M = 8, 100 ns at M = 12), so what it stages and draws per launch (a third of a
// one-step launch) and how many CTAs an SM holds (4 by registers, fewer above 56 KB) count.  us per step, separate kernels -> this one:
//   M = 8, X = 24, 2/2 (23 to 32 KB a CTA)      n = 1        n = 2         n = 5         n = 8
//     128 walkers                              74 -> 38     70 -> 27      67 -> 19      67 -> 17
//     1000                                     105 -> 82    101 -> 64     98 -> 54      98 -> 52
//     2000                                     148 -> 150   144 -> 121    142 -> 106    141 -> 102
//     8000                                     437 -> 481   434 -> 400    431 -> 358    430 -> 352
//     40000                                    1832 -> 2244 1826 -> 1885  1825 -> 1689  1825 -> 1654
//   M = 12, X = 40, 3/3 (67 to 85 KB)
//     300                                      94 -> 63     90 -> 51      88 -> 43      87 -> 42
//     1000                                     177 -> 203   174 -> 176    172 -> 165    171 -> 162
//     2000                                     296 -> 330   291 -> 288    289 -> 288    288 -> 282
//     4000                                     486 -> 586   481 -> 517    479 -> 572    478 -> 561
// The populations at which the two meet grow with the number of CTAs whose memory an SM's would hold, up to
// some 10 (M = 4, X = 8, 1/1, single steps: 2000 walkers), so they are counted in waves of these: one for single
// steps, seven for two steps or where fewer than 6 fit, and any number else.
bool step_small_pays(const Ctx& c, int n) {
  if (!step_small_ok(c)) return false;
  const size_t sm = sizeof(double) * (size_t)layout(c.M, c.N, c.X, (int)c.P, std::min(n, kSteps)).total + 2048;
  const int fit = (int)std::min<size_t>(10, (size_t)228 * 1024 / sm);
  const int waves = (c.Nw + 152 * fit - 1) / (152 * fit);
  return n <= 1 ? waves <= 1 : (n == 2 || fit < 6) ? waves <= 7 : true;
}

cudaError_t prepare_step_small(const Ctx& c) {
  const size_t sm = sizeof(double) * (size_t)layout(c.M, c.N, c.X, (int)c.P, kSteps).total;
  return g_small_limits.raise(0, sm, [&] {
    cudaError_t e = cudaSuccess;
    for (auto k : {k_steps_small<2>, k_steps_small<4>, k_steps_small<8>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    return e;
  });
}

// n_steps steps of every walker from the device step counter on, which is advanced by them; fields
// [n_steps][Nw][X] or null.
cudaError_t launch_steps_small(const Ctx& c, int n_steps, const double* fields, cudaStream_t s) {
  for (int t = 0; t < n_steps; t += kSteps) {
    SmallArgs a;
    a.Lt = c.Lt; a.Ltil = c.Ltil; a.expK = c.expK; a.psi = c.psi; a.rho = c.rho_mf;
    a.fields = fields ? fields + (int64_t)t * c.Nw * c.X : nullptr;
    a.phi = c.phi; a.theta = c.theta; a.logO = c.logO; a.w = c.w; a.alive = c.alive; a.flags = c.d_flags;
    a.step = c.d_step;
    a.key = make_uint2((uint32_t)(c.opt.seed & 0xffffffffull), (uint32_t)(c.opt.seed >> 32));
    a.k0 = (uint32_t)c.opt.walker_offset;
    a.M = c.M; a.N = c.N; a.nu = c.n_up; a.X = c.X; a.P = (int)c.P; a.Nw = c.Nw;
    a.n = std::min(kSteps, n_steps - t);
    a.order = c.opt.taylor_order;
    a.free_proj = c.opt.mode == AFQMC_FREE;
    a.sqrt_dt = c.sqrt_dt; a.fb_cap = c.opt.fb_cap;
    a.log_shift = -c.opt.dt * (c.c_mf - c.e_trial);
    const size_t sm = sizeof(double) * (size_t)layout(c.M, c.N, c.X, a.P, a.n).total;
    const int ns = std::max(c.n_up, c.N - c.n_up);
    (ns <= 2 ? k_steps_small<2> : ns <= 4 ? k_steps_small<4> : k_steps_small<8>)<<<c.Nw, kT, sm, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_step_advance(c, s, a.n);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace afq
