// kite_recon.cu -- FP64 reconstruction of the density of states from raw moments.
//
// rho(E) = [g_0 mu_0 + 2 sum_{n>=1} g_n mu_n T_n(eps)] / (pi sqrt(1-eps^2) de_minus) with
// eps = (E - de_plus)/de_minus: the delta-function expansion of Sec. 2a
// (Delta_n = 2 T_n / (pi sqrt(1-eps^2)), weight 1/(1+delta_n0)) traced as in Eq. e7,
// truncated at M terms (Eq. e8a) and damped by a kernel g_n (Sec. 2a).
#include <math.h>

#include <algorithm>

#include <vector>

#include "kite_internal.h"
#include "kite_nufft.cuh"

namespace kite {
namespace {

// c_n = (2 - delta_n0) g_n mu_n, kernel built for M terms.
__global__ void k_dos_coef(const double* __restrict__ mu, int M, int kernel, double param,
                           double* __restrict__ coef) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= M) return;
  double g = 1.0;
  if (kernel == KITE_KERNEL_JACKSON) {
    // Jackson kernel (Weisse et al., Rev. Mod. Phys. 78, 275 (2006)):
    // g_n = [(M-n+1) cos(pi n/(M+1)) + sin(pi n/(M+1)) cot(pi/(M+1))] / (M+1)
    const double q = 3.141592653589793 / (double)(M + 1);
    const double cot = cos(q) / sin(q);
    g = ((double)(M - n + 1) * cos(q * n) + sin(q * n) * cot) / (double)(M + 1);
  } else if (kernel == KITE_KERNEL_LORENTZ) {
    g = sinh(param * (1.0 - (double)n / (double)M)) / sinh(param);
  }
  coef[n] = (n == 0 ? 1.0 : 2.0) * g * mu[n];
}

// One thread per energy; the Chebyshev polynomials follow the recurrence of Eq. e3.
// Coefficients are staged through shared memory in tiles.
__global__ void k_dos_eval(const double* __restrict__ coef, int M, double de_plus,
                           double de_minus, const double* __restrict__ E, int K,
                           double* __restrict__ rho) {
  __shared__ double tile[1024];
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  double eps = 0.0;
  bool inside = false;
  if (k < K) {
    eps = (E[k] - de_plus) / de_minus;
    inside = eps > -1.0 && eps < 1.0;
  }
  double tm1 = 1.0, t = eps, sum = 0.0;
  for (int base = 0; base < M; base += 1024) {
    const int len = min(1024, M - base);
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += blockDim.x) tile[i] = coef[base + i];
    __syncthreads();
    for (int i = 0; i < len; ++i) {
      const int n = base + i;
      if (n == 0) {
        sum += tile[i];
      } else {
        sum += tile[i] * t;
        const double tn = 2.0 * eps * t - tm1;
        tm1 = t;
        t = tn;
      }
    }
  }
  if (k < K) rho[k] = inside ? sum / (3.141592653589793 * sqrt(1.0 - eps * eps)) / de_minus : 0.0;
}

// Average Green's function G(E + i eta) per eV (Eqs. green_function_cheb_expansion/b traced
// as in Eq. e7): sum_n (c_n / 2) g^{+,eta~}_n(eps) / de_minus with c_n = (2 - d_n0) g_n mu_n
// from k_dos_coef, and the retarded CPGF coefficients g_n = -2i q^n / sqrt(1 - z^2),
// q = z - i sqrt(1 - z^2), z = eps + i eta~ (geometric in n).  One thread per energy.
struct gcplx {
  double re, im;
};
__device__ __forceinline__ gcplx gmul(gcplx a, gcplx b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ gcplx gsqrt(gcplx z) {  // principal branch
  const double r = hypot(z.re, z.im);
  if (r == 0.0) return {0.0, 0.0};
  if (z.re >= 0.0) {
    const double t = sqrt(0.5 * (r + z.re));
    return {t, z.im / (2.0 * t)};
  }
  const double t = sqrt(0.5 * (r - z.re));
  return {fabs(z.im) / (2.0 * t), z.im >= 0.0 ? t : -t};
}

__global__ void k_green_eval(const double* __restrict__ coef, int M, double de_plus, double de_minus,
                             double eta_t, const double* __restrict__ E, int K, double* __restrict__ G,
                             double* __restrict__ rho) {
  __shared__ double tile[1024];
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const double eps = k < K ? (E[k] - de_plus) / de_minus : 0.0;
  const gcplx z = {eps, eta_t};
  const gcplx r = gsqrt({1.0 - (z.re * z.re - z.im * z.im), -2.0 * z.re * z.im});
  const gcplx q = {z.re + r.im, z.im - r.re};  // z - i r
  // g_0 = -2i / r
  const double rr = r.re * r.re + r.im * r.im;
  gcplx g = {-2.0 * r.im / rr, -2.0 * r.re / rr};
  double are = 0.0, aim = 0.0;
  for (int base = 0; base < M; base += 1024) {
    const int len = min(1024, M - base);
    __syncthreads();
    for (int i = threadIdx.x; i < len; i += blockDim.x) tile[i] = 0.5 * coef[base + i];
    __syncthreads();
    for (int i = 0; i < len; ++i) {
      are += tile[i] * g.re;
      aim += tile[i] * g.im;
      g = gmul(g, q);
    }
  }
  if (k < K) {
    if (G) {
      G[2 * k] = are / de_minus;
      G[2 * k + 1] = aim / de_minus;
    }
    if (rho) rho[k] = -aim / de_minus / 3.141592653589793;
  }
}

}  // namespace

int reconstruct_green_impl(kite_ctx* ctx, const double* mu_dev, int M_use, int kernel, double param,
                           const Scale& sc, double eta, const double* E_dev, int K, double* G_dev,
                           double* rho_dev, double* coef_dev) {
  k_dos_coef<<<(M_use + 255) / 256, 256, 0, ctx->stream>>>(mu_dev, M_use, kernel, param, coef_dev);
  KITE_CUDA_TRY(ctx, cudaGetLastError());
  k_green_eval<<<(K + 127) / 128, 128, 0, ctx->stream>>>(coef_dev, M_use, sc.de_plus, sc.de_minus,
                                                         eta / sc.de_minus, E_dev, K, G_dev, rho_dev);
  KITE_CUDA_TRY(ctx, cudaGetLastError());
  return KITE_OK;
}

int reconstruct_dos_impl(kite_ctx* ctx, const double* mu_dev, int M_use, int kernel,
                         double param, const Scale& sc, const double* E_dev, int K,
                         double* rho_dev, double* coef_dev) {
  k_dos_coef<<<(M_use + 255) / 256, 256, 0, ctx->stream>>>(mu_dev, M_use, kernel, param, coef_dev);
  KITE_CUDA_TRY(ctx, cudaGetLastError());
  k_dos_eval<<<(K + 127) / 128, 128, 0, ctx->stream>>>(coef_dev, M_use, sc.de_plus, sc.de_minus,
                                                       E_dev, K, rho_dev);
  KITE_CUDA_TRY(ctx, cudaGetLastError());
  return KITE_OK;
}

}  // namespace kite

// ====================================================================================
// First-order optical conductivity sigma_xx(omega) from the 2D moments (Sec. 2b):
//   Gamma_nm = -g_n g_m mu_nm / ((1 + d_n0)(1 + d_m0))            (Eq. Gammanm, damped)
//   S(w) = int de f(e) sum_nm Gamma_nm [g^R_n(e + w) Delta_m(e) + Delta_n(e) g^A_m(e - w)]
//   sigma(w) = -i (n_orb a^2/Omega_c) / w * S(w)   [units e^2/hbar, w = hbar omega/de_minus]
// (Eq. conductivity_1st_order in rescaled units).  With e = cos(theta), Delta_m(e) de =
// (2/pi) cos(m theta) d theta, integrated by Gauss-Legendre quadrature in theta.  Then
// U[n][k] = sum_m Gamma_nm D[m][k] and W[m][k] = sum_n Gamma_nm D[n][k] (cosine sums at the
// nodes, kite_nufft.cuh; dense FP64 products outside its range of orders and nodes), and per frequency
// S = sum_k sum_n (g^R_n(e_k + w) U[n][k] + g^A_n(e_k - w) W[n][k]).
// The CPGF coefficients (Eq. green_function_cheb_expansionb) are geometric in n:
// g^{s}_n(z) = -2 s i q^n / sqrt(1 - z^2) with q = exp(-s i arccos z) = z - s i sqrt(1 - z^2)
// for the principal branches, so only a complex square root is needed per (w, node).
// ====================================================================================
namespace kite {
namespace {

struct cplx {
  double re, im;
};
__device__ __forceinline__ cplx cmul(cplx a, cplx b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ cplx cdiv(cplx a, cplx b) {
  const double d = b.re * b.re + b.im * b.im;
  return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
// principal square root (Re >= 0), cancellation-free in both half planes
__device__ __forceinline__ cplx csqrt_p(cplx z) {
  const double r = hypot(z.re, z.im);
  if (r == 0.0) return {0.0, 0.0};
  if (z.re >= 0.0) {
    const double t = sqrt(0.5 * (r + z.re));
    return {t, z.im / (2.0 * t)};
  }
  const double t = sqrt(0.5 * (r - z.re));
  return {fabs(z.im) / (2.0 * t), z.im >= 0.0 ? t : -t};
}

__global__ void k_sig_gamma(const double* __restrict__ mu, int M_avail, int M, int kernel,
                            double* __restrict__ gam) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)M * M) return;
  const int n = (int)(e / M), m = (int)(e - (e / M) * M);
  auto jackson = [&](int k) {
    const double q = 3.141592653589793 / (double)(M + 1);
    return ((double)(M - k + 1) * cos(q * k) + sin(q * k) * (cos(q) / sin(q))) / (double)(M + 1);
  };
  double w = (n == 0 ? 0.5 : 1.0) * (m == 0 ? 0.5 : 1.0);
  if (kernel == KITE_KERNEL_JACKSON) w *= jackson(n) * jackson(m);
  const double* p = mu + 2 * ((int64_t)n * M_avail + m);
  gam[2 * e] = -w * p[0];
  gam[2 * e + 1] = -w * p[1];
}

// D[m][k] = (2/pi) cos(m theta_k) w_k
__global__ void k_sig_dmat(const double* __restrict__ theta, const double* __restrict__ wq, int M,
                           int K, double* __restrict__ D) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)M * K) return;
  const int m = (int)(e / K), k = (int)(e - (e / K) * K);
  D[e] = 0.6366197723675814 * cos((double)m * theta[k]) * wq[k];
}

// C[i][k] = sum_j A(i,j) B[j][k], A complex [M][M] (A(i,j) = G[i][j] or, if trans, G[j][i]),
// B real [M][K], C complex [M][K].  16x16 tiles through shared memory.
__global__ void k_zgemm_real(const double* __restrict__ G, int trans, const double* __restrict__ B,
                             int M, int K, double* __restrict__ Cm) {
  __shared__ double As_re[16][17], As_im[16][17], Bs[16][17];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int i = blockIdx.y * 16 + ty, k = blockIdx.x * 16 + tx;
  double re = 0.0, im = 0.0;
  for (int j0 = 0; j0 < M; j0 += 16) {
    const int ia = blockIdx.y * 16 + ty, ja = j0 + tx;
    double ar = 0.0, ai = 0.0;
    if (ia < M && ja < M) {
      const int64_t idx = trans ? (int64_t)ja * M + ia : (int64_t)ia * M + ja;
      ar = G[2 * idx];
      ai = G[2 * idx + 1];
    }
    As_re[ty][tx] = ar;
    As_im[ty][tx] = ai;
    const int jb = j0 + ty;
    Bs[ty][tx] = (jb < M && k < K) ? B[(int64_t)jb * K + k] : 0.0;
    __syncthreads();
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
      re += As_re[ty][jj] * Bs[jj][tx];
      im += As_im[ty][jj] * Bs[jj][tx];
    }
    __syncthreads();
  }
  if (i < M && k < K) {
    Cm[2 * ((int64_t)i * K + k)] = re;
    Cm[2 * ((int64_t)i * K + k) + 1] = im;
  }
}

// Partial sums of S(w): a block takes 128 nodes, kSigW frequencies and one branch (retarded
// with U, advanced with W).  The CPGF sum of a node is a polynomial in q, by Horner's rule
// (four FP64 multiply-adds per term instead of eight with the powers carried along: the FP64
// pipe is the bound), kSigW of them side by side on each loaded coefficient.  M = 512, 1088
// nodes, 128 frequencies: 3.34 ms with one block per frequency and carried powers, 1.09 ms so
// (0.57 G multiply-adds: 0.9 ms at the FP64 pipe's rate); the whole call 19.8 -> 1.5 ms.
constexpr int kSigW = 4;
__global__ void __launch_bounds__(128) k_sig_omega(const double2* __restrict__ U, const double2* __restrict__ W,
                                                   const double* __restrict__ theta, int M, int K,
                                                   const double* __restrict__ wt, int K_w, double eta_t,
                                                   double2* __restrict__ part) {
  const int k = blockIdx.x * 128 + threadIdx.x, w0 = blockIdx.y * kSigW, sgn = blockIdx.z;
  const double s = sgn == 0 ? 1.0 : -1.0;
  // retarded: z = e + w + i eta, g_n = -2i q^n / sqrt(1 - z^2), q = z - i sqrt(1 - z^2)
  // advanced: z = e - w - i eta, g_n = +2i q^n / sqrt(1 - z^2), q = z + i sqrt(1 - z^2)
  cplx q[kSigW], g0[kSigW], p[kSigW];
  const bool on = k < K;
  const double e = on ? cos(theta[k]) : 0.0;
#pragma unroll
  for (int i = 0; i < kSigW; ++i) {
    const cplx z = {e + s * wt[min(w0 + i, K_w - 1)], s * eta_t};
    // 1 - z^2, without the cancellation near the band edges
    const cplx r = csqrt_p({fma(1.0 - z.re, 1.0 + z.re, z.im * z.im), -2.0 * z.re * z.im});
    q[i] = {z.re + s * r.im, z.im - s * r.re};  // z - s i r
    g0[i] = cdiv({0.0, -2.0 * s}, r);
    p[i] = {0.0, 0.0};
  }
  if (on) {
    const double2* X = (sgn == 0 ? U : W) + k;
#pragma unroll 4
    for (int n = M - 1; n >= 0; --n) {
      const double2 x = X[(int64_t)n * K];
#pragma unroll
      for (int i = 0; i < kSigW; ++i)
        p[i] = {fma(p[i].re, q[i].re, fma(-p[i].im, q[i].im, x.x)), fma(p[i].re, q[i].im, fma(p[i].im, q[i].re, x.y))};
    }
  }
  __shared__ double2 red[128];
#pragma unroll
  for (int i = 0; i < kSigW; ++i) {
    const cplx v = cmul(g0[i], p[i]);
    __syncthreads();
    red[threadIdx.x] = on ? make_double2(v.re, v.im) : make_double2(0.0, 0.0);
    __syncthreads();
    for (int st = 64; st > 0; st >>= 1) {
      if ((int)threadIdx.x < st) {
        red[threadIdx.x].x += red[threadIdx.x + st].x;
        red[threadIdx.x].y += red[threadIdx.x + st].y;
      }
      __syncthreads();
    }
    if (threadIdx.x == 0 && w0 + i < K_w) part[((int64_t)(w0 + i) * 2 + sgn) * gridDim.x + blockIdx.x] = red[0];
  }
}

// sigma = -i factor / w * S, S the sum of a frequency's `n` partials in order
__global__ void k_sig_final(const double2* __restrict__ part, int n, const double* __restrict__ wt, int K_w,
                            double factor, double* __restrict__ sigma) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= K_w) return;
  double re = 0.0, im = 0.0;
  for (int b = 0; b < n; ++b) {
    re += part[(int64_t)i * n + b].x;
    im += part[(int64_t)i * n + b].y;
  }
  sigma[2 * i] = factor / wt[i] * im;
  sigma[2 * i + 1] = -factor / wt[i] * re;
}

// ---- DC conductivity (Kubo-Greenwood, T = 0) ---------------------------------------
// One block per energy (grid-stride): the kernel-damped delta coefficients
// c_n = w_n T_n(e) / (pi sqrt(1 - e^2)), w_n = (2 - delta_n0) g_n, in shared memory; each
// warp contracts whole rows, s = sum_n c_n sum_m Re(mu_nm) c_m, then a fixed-order sum
// over the warps.  sigma_k = pi ucf s (0 outside |e| < 1).  FP64 throughout.
__global__ void k_sigma_dc(const double* __restrict__ mu, int M_avail, int M, const double* __restrict__ w,
                           double de_plus, double de_minus, const double* __restrict__ E, int K, double ucf,
                           double* __restrict__ sigma) {
  extern __shared__ double c[];  // [M] + [blockDim/32]
  double* wsum = c + M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int k = blockIdx.x; k < K; k += gridDim.x) {
    const double e = (E[k] - de_plus) / de_minus;
    if (!(fabs(e) < 1.0)) {
      if (threadIdx.x == 0) sigma[k] = 0.0;
      continue;  // uniform across the block
    }
    const double th = acos(e), den = 3.141592653589793 * sqrt(1.0 - e * e);
    for (int n = threadIdx.x; n < M; n += blockDim.x) c[n] = w[n] * cos((double)n * th) / den;
    __syncthreads();
    double acc = 0.0;
    for (int n = warp; n < M; n += nwarp) {
      const double* row = mu + 2 * (size_t)n * M_avail;
      double r = 0.0;
      for (int m = lane; m < M; m += 32) r += row[2 * m] * c[m];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
      acc += c[n] * r;
    }
    if (lane == 0) wsum[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int q = 0; q < nwarp; ++q) sum += wsum[q];
      sigma[k] = 3.141592653589793 * ucf * sum;
    }
    __syncthreads();
  }
}

// w_n = (2 - delta_n0) g_n for the kernel built for M terms
__global__ void k_dc_weights(int M, int kernel, double param, double* __restrict__ w) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= M) return;
  double g = 1.0;
  if (kernel == KITE_KERNEL_JACKSON) {
    const double q = 3.141592653589793 / (double)(M + 1);
    g = ((double)(M - n + 1) * cos(q * n) + sin(q * n) * (cos(q) / sin(q))) / (double)(M + 1);
  } else if (kernel == KITE_KERNEL_LORENTZ) {
    g = sinh(param * (1.0 - (double)n / (double)M)) / sinh(param);
  }
  w[n] = (n == 0 ? 1.0 : 2.0) * g;
}

}  // namespace

namespace {

// Launches of the Gauss-Legendre rule: K nodes u = 1 + x and weights w, ab scratch of 2K doubles.
void gauss_rule(cudaStream_t st, int K, double* ab, double* u, double* w) {
  k_legendre_coef<<<std::min(1024, (K + 255) / 256), 256, 0, st>>>(K, reinterpret_cast<double2*>(ab));
  k_gauss_legendre<<<((K + 1) / 2 + kGaussBlock / 16 - 1) / (kGaussBlock / 16), kGaussBlock, 0, st>>>(
      K, reinterpret_cast<const double2*>(ab), u, w);
}

// The rule of few nodes on the host, in the kernel's form (four roots side by side), where the
// kernel's two launches and its serial chain cost more: Bastin's sum of eight nodes at M = 8
// takes 87 us so, 107 us with the kernel; of 64 nodes 88 and 107.
constexpr int kHostRule = 64;
void gauss_rule_host(int K, double* u, double* w) {
  double ca[kHostRule], cb[kHostRule];
  for (int j = 1; j <= K; ++j) ca[j - 1] = (2.0 * j - 1.0) / j, cb[j - 1] = (j - 1.0) / j;
  const int half = (K + 1) / 2;
  const double dK = (double)K;
  for (int i0 = 0; i0 < half; i0 += 4) {
    double d[4], wt[4];
    for (int q = 0; q < 4; ++q) {
      const double sh = sin(0.5 * kPi * (std::min(i0 + q, half - 1) + 0.75) / (dK + 0.5)), c0 = -2.0 * sh * sh;
      d[q] = c0 - (0.125 / (dK * dK) - 0.125 / (dK * dK * dK)) * (1.0 + c0);
    }
    bool done = false;
    for (int it = 0; it < 9 && !done; ++it) {
      double p[4] = {1.0, 1.0, 1.0, 1.0}, D[4] = {0.0, 0.0, 0.0, 0.0};
      for (int j = 0; j < K; ++j)
        for (int q = 0; q < 4; ++q) {
          D[q] = cb[j] * D[q] + (ca[j] * d[q]) * p[q];
          p[q] += D[q];
        }
      done = true;
      for (int q = 0; q < 4; ++q) {
        const double om = -d[q] * (2.0 + d[q]), dp = -dK * (d[q] * p[q] + D[q]) / om, dz = p[q] / dp;
        wt[q] = 2.0 / (om * dp * dp) * (1.0 + dz * (2.0 * (1.0 + d[q]) - dK * (dK + 1.0) * dz) / om);
        d[q] -= dz;
        done = done && !(fabs(dz) > 4e-9 * om);
      }
    }
    for (int q = 0; q < 4 && i0 + q < half; ++q) {
      const int i = i0 + q;
      u[K - 1 - i] = 2.0 + d[q];
      u[i] = -d[q];
      w[i] = w[K - 1 - i] = wt[q];
    }
  }
}

// The Fermi energy in theta (the lower end of the sea at T = 0).
double theta_fermi(double E_F, const Scale& sc) {
  return acos(fmin(1.0, fmax(-1.0, (E_F - sc.de_plus) / sc.de_minus)));
}

// Device buffers of the non-uniform transform for order M, in doubles, and its launches.
struct Nufft {
  int M, Nf, L, logN;
  double *inv, *tw, *grid;
  static bool fits(int M) { return M >= kNufftMinM && M <= kNufftMaxM; }  // (and enough nodes)
  explicit Nufft(int M_) : M(M_), Nf(nufft_grid(M_)), L(nufft_row(Nf)), logN(0) {
    while ((1 << logN) < Nf) ++logN;
  }
  size_t doubles(int rows) const {
    return (size_t)M + 1 + Nf + 2 * (size_t)rows * L;
  }
  void carve(double* b) {  // 16-byte aligned pieces
    inv = b;
    tw = b + ((size_t)M + 1) / 2 * 2;
    grid = tw + Nf;
  }
  // cosine sums of `rows` rows on the grid (see k_cos_fft)
  int rows_to_grid(kite_ctx* ctx, const double* mu, int M_avail, int kind, const double* w, int rows) const {
    cudaStream_t st = ctx->stream;
    k_nufft_tables<<<(std::max(32 * M, Nf / 2) + 127) / 128, 128, 0, st>>>(M, Nf, inv, reinterpret_cast<double2*>(tw));
    const int smem = Nf * 16;
    if (smem > 48 * 1024)
      KITE_CUDA_TRY(ctx, cudaFuncSetAttribute(k_cos_fft, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              nufft_grid(kNufftMaxM) * 16));
    k_cos_fft<<<rows, 256, smem, st>>>(mu, M_avail, M, kind, w, inv, reinterpret_cast<const double2*>(tw), Nf, logN,
                                       reinterpret_cast<double2*>(grid));
    return KITE_OK;
  }
};

}  // namespace

int reconstruct_sigma_impl(kite_ctx* ctx, const double* mu_dev, int M_avail, int M, int lattice,
                           int kernel, const Scale& sc, double E_F, double kT, double eta,
                           const double* omega_host, int K_w, int n_quad, double* sigma_dev) {
  const int K = n_quad > 0 ? n_quad : 2 * M + 64;
  const bool fast = Nufft::fits(M) && K >= kNufftMinNodes;
  Nufft nf(M);
  // rescaled frequencies, then the Fermi energy in E and theta, then few nodes and their weights
  const size_t Kp = ((size_t)K + 1) / 2 * 2, Wp = ((size_t)K_w + 3) / 2 * 2;
  std::vector<double> in(Wp + (K <= kHostRule ? 2 * Kp : 0));
  for (int i = 0; i < K_w; ++i) in[i] = omega_host[i] / sc.de_minus;
  in[K_w] = E_F;
  in[K_w + 1] = theta_fermi(E_F, sc);
  const bool on_host = K <= kHostRule;
  if (on_host) {
    double *th = in.data() + Wp, *wq = th + Kp;
    gauss_rule_host(K, th, wq);
    for (int k = 0; k < K; ++k)
      fermi_node(th[k], wq[k], E_F, in[K_w + 1], sc.de_plus, sc.de_minus, kT, &th[k], &wq[k]);
  }
  // all offsets even: 16-byte aligned complex values
  const size_t nU = 2 * (size_t)M * K, Mp = ((size_t)M + 1) / 2 * 2;
  const int blocks = (K + 127) / 128;
  const size_t nPart = 4 * (size_t)K_w * blocks;
  const size_t nDense = 2 * (size_t)M * M + (size_t)M * Kp;       // Gamma, D
  const size_t nFast = (nf.doubles(2 * M) + 2 + Kp + kTaps * Kp);  // transform, first taps, taps
  double* buf = nullptr;
  const size_t total = 2 * nU + 2 * Kp + 4 * Kp + Wp + Mp + nPart + (fast ? nFast : nDense);
  KITE_CUDA_TRY(ctx, cudaMallocAsync((void**)&buf, total * sizeof(double), ctx->stream));
  double* U = buf;
  double* W = U + nU;
  double* gab = W + nU;
  double* gx = gab + 2 * Kp;
  double* gw = gx + Kp;
  double* in_d = gw + Kp;
  double* th_d = in_d + Wp;
  double* wq_d = th_d + Kp;
  double* wk = wq_d + Kp;
  double* part = wk + Mp;
  double* rest = part + nPart;
  cudaStream_t st = ctx->stream;
  cudaError_t e = cudaMemcpyAsync(in_d, in.data(), in.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  int rc = e == cudaSuccess ? KITE_OK : cuda_fail(ctx, e, "sigma set-up");
  if (rc == KITE_OK) {
    if (!on_host) {
      gauss_rule(st, K, gab, gx, gw);
      k_fermi_nodes<<<(K + 255) / 256, 256, 0, st>>>(gx, gw, K, in_d + K_w, in_d + K_w + 1, 1, sc.de_plus, sc.de_minus,
                                                     kT, th_d, wq_d);
    }
    if (fast) {
      nf.carve(rest);
      double* taps = rest + (nf.doubles(2 * M) + 2) / 2 * 2;
      int* j0 = reinterpret_cast<int*>(taps + kTaps * Kp);
      k_dc_weights<<<(M + 63) / 64, 64, 0, st>>>(M, kernel, 0.0, wk);
      rc = nf.rows_to_grid(ctx, mu_dev, M_avail, 0, wk, 2 * M);
      k_nufft_taps<<<(K + 127) / 128, 128, 0, st>>>(th_d, wq_d, K, nf.Nf, j0, taps);
      dim3 grd((K + 127) / 128, (2 * M + kApplyRows - 1) / kApplyRows);
      k_nufft_apply<<<grd, 128, 0, st>>>(reinterpret_cast<const double2*>(nf.grid), nf.L, 2 * M, K, j0, taps,
                                         reinterpret_cast<double2*>(U));  // W follows U
    } else {
      double* G = rest;
      double* D = G + 2 * (size_t)M * M;
      k_sig_gamma<<<(int)(((int64_t)M * M + 255) / 256), 256, 0, st>>>(mu_dev, M_avail, M, kernel, G);
      k_sig_dmat<<<(int)(((int64_t)M * K + 255) / 256), 256, 0, st>>>(th_d, wq_d, M, K, D);
      dim3 blk(16, 16), grd((K + 15) / 16, (M + 15) / 16);
      k_zgemm_real<<<grd, blk, 0, st>>>(G, 0, D, M, K, U);
      k_zgemm_real<<<grd, blk, 0, st>>>(G, 1, D, M, K, W);
    }
    const double factor = lattice == KITE_HONEYCOMB ? 4.0 / sqrt(3.0) : 1.0;
    for (int i0 = 0; i0 < K_w; i0 += 65535 * kSigW) {  // (the grid's y extent)
      const int nw = std::min(K_w - i0, 65535 * kSigW);
      dim3 g3((unsigned)blocks, (unsigned)((nw + kSigW - 1) / kSigW), 2);
      k_sig_omega<<<g3, 128, 0, st>>>(reinterpret_cast<const double2*>(U), reinterpret_cast<const double2*>(W), th_d, M,
                                      K, in_d + i0, nw, eta / sc.de_minus,
                                      reinterpret_cast<double2*>(part) + 2 * (size_t)i0 * blocks);
    }
    k_sig_final<<<(K_w + 127) / 128, 128, 0, st>>>(reinterpret_cast<const double2*>(part), 2 * blocks, in_d, K_w, factor,
                                                   sigma_dev);
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(ctx, e, "sigma kernels");
  }
  cudaFreeAsync(buf, st);
  // (`in` is pageable: the copy above has taken its values before it returned)
  return rc;
}

}  // namespace kite

namespace kite {

// sigma_DC(E_k) for K energies from the leading M x M block of mu_nm (device pointers);
// w is device scratch of M doubles.
int reconstruct_sigma_dc_impl(kite_ctx* ctx, const double* mu_dev, int M_avail, int M, int kernel, double param,
                              int lattice, const Scale& sc, const double* E_dev, int K, double* sigma_dev,
                              double* w) {
  cudaStream_t st = ctx->stream;
  k_dc_weights<<<(M + 63) / 64, 64, 0, st>>>(M, kernel, param, w);
  // Few energies and long rows: wide blocks, so that each one's SM has enough warps in flight.
  // us per call with 256 / 512 / 1024 threads: M = 4096, 48 energies 6880 / 4413 / 4421, M = 2048
  // 1273 / 1207 / 1212, M = 1024 371 / 369 / 379, M = 64 50 / 53 / 60; more energies than SMs, M =
  // 2048 2365 / 2369 / 2383.
  const int block = K <= ctx->num_sms && M >= 1536 ? 512 : 256;
  const size_t smem = sizeof(double) * ((size_t)M + block / 32);
  if (smem > 48 * 1024)
    KITE_CUDA_TRY(ctx, cudaFuncSetAttribute(k_sigma_dc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int grid = std::max(1, std::min(K, ctx->num_sms * 4));
  const double ucf = lattice == KITE_HONEYCOMB ? 2.0 * 2.0 / sqrt(3.0) : 1.0;
  k_sigma_dc<<<grid, block, smem, st>>>(mu_dev, M_avail, M, w, sc.de_plus, sc.de_minus, E_dev, K, ucf,
                                         sigma_dev);
  KITE_CUDA_TRY(ctx, cudaGetLastError());
  return KITE_OK;
}

}  // namespace kite

// ====================================================================================
// DC conductivity tensor from the Kubo-Bastin formula, Fermi sea included (the Hall
// conductivity of the paper's quantum anomalous Hall example, Sec. 2b at omega -> 0):
//   sigma_ab(E_F) = Re{ i ucf int de f(e) sum_nm mu_nm [Delta_n(e) dG^R_m(e) - dG^A_n(e) Delta_m(e)] }
// with Delta_n(e) de = k_n (2 - d_n0)/pi cos(n theta) d theta (e = cos theta), the CPGF
// coefficients G^{R/A}_m(e) = k_m g^{+-}_m(e +- i eta)/(1 + d_m0) (Eq.
// green_function_cheb_expansionb) and their derivatives
//   d g_m/dz = g_m(z) [s i m / sqrt(1 - z^2) + z / (1 - z^2)]   (s = +1 retarded, -1 advanced).
// A_nm = mu_nm k_n k_m / ((1 + d_n0)(1 + d_m0)).  Each Fermi energy has its own
// Gauss-Legendre nodes theta_k on [theta_F, pi] (kT > 0: [0, pi] with Fermi weights).  Since
// G^A = conj(G^R) on the real axis' two sides and only the imaginary part of the sum counts,
// the second term folds into the first: with the Hermitian B_nm = A_nm + conj(A_mn),
//   Im F_k = Im sum_m dG^R_m(e_k) V[m][k],  V[m][k] = sum_n B_nm D[n][k],
// D[n][k] = (2/pi) cos(n theta_k) w_k: half the products, and V by the non-uniform transform
// (kite_nufft.cuh; a dense FP64 product outside its range of orders and nodes).  The CPGF terms are
// geometric, g_m = g_0 q^m with q = z - i sqrt(1 - z^2): S0 = sum_m q^m V_m and S1 = sum_m m
// q^m V_m by Horner's rule and its derivative, sum_m dg_m V_m = g_0 (i S1 / r + z S0 / r^2),
// r = sqrt(1 - z^2).  sigma = -ucf Im(sum_k F_k), each energy's node sum in a fixed order.
// M = 256, 48 energies of 576 nodes: 16.9 ms with two dense products per energy and host
// nodes, 0.88 ms so (0.59 ms of it the nodes' 40 multiply-adds per order, 0.45 ms at the FP64
// pipe's rate).
// ====================================================================================
namespace kite {
namespace {

// B_nm = A_nm + conj(A_mn) (dense path)
__global__ void k_bastin_gamma(const double* __restrict__ mu, int M_avail, int M, const double* __restrict__ w,
                               double* __restrict__ B) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)M * M) return;
  const int n = (int)(e / M), m = (int)(e - (e / M) * M);
  // w_n = (2 - d_n0) k_n, so w_n / 2 = k_n / (1 + d_n0)
  const double f = 0.25 * w[n] * w[m];
  const double* p = mu + 2 * ((int64_t)n * M_avail + m);
  const double* t = mu + 2 * ((int64_t)m * M_avail + n);
  B[2 * e] = f * (p[0] + t[0]);
  B[2 * e + 1] = f * (p[1] - t[1]);
}

// Im F_k per node from V (dense path: V[m][k]; else from the rows' grid values and the node's
// taps, sixteen multiply-adds per part on the way: V is never stored).
constexpr int kNodeBlock = 64;  // (small blocks: a few thousand nodes still fill the SMs evenly)
template <bool DENSE>
__global__ void __launch_bounds__(kNodeBlock) k_bastin_nodes(const double2* __restrict__ V, const double2* __restrict__ grid,
                                                      int L, const int* __restrict__ j0,
                                                      const double* __restrict__ taps,
                                                      const double* __restrict__ theta, int M, int64_t Kt,
                                                      double eta_t, double* __restrict__ F) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= Kt) return;
  cplx z = {0.0, eta_t};
  double sn;
  sincos(theta[k], &sn, &z.re);
  // 1 - z^2 from the sine: no cancellation near the band edges
  const cplx r = csqrt_p({fma(sn, sn, z.im * z.im), -2.0 * z.re * z.im});
  const cplx q = {z.re + r.im, z.im - r.re};  // z - i r
  const cplx g = cdiv({0.0, -2.0}, r);
  double t[kTaps];
  const double2* b = nullptr;
  if (!DENSE) {
#pragma unroll
    for (int i = 0; i < kTaps; ++i) t[i] = taps[(int64_t)i * Kt + k];
    b = grid + j0[k];
  }
  cplx P = {0.0, 0.0}, Q = {0.0, 0.0};  // sum_m q^m V_m and its derivative in q
#pragma unroll 1
  for (int m = M - 1; m >= 0; --m) {
    double2 v;
    if (DENSE) {
      v = V[(int64_t)m * Kt + k];
    } else {
      const double2* c = b + (int64_t)m * L;
      double re0 = 0.0, im0 = 0.0, re1 = 0.0, im1 = 0.0;
#pragma unroll
      for (int i = 0; i < kTaps; i += 2) {
        const double2 x = c[i], y = c[i + 1];
        re0 = fma(t[i], x.x, re0);
        im0 = fma(t[i], x.y, im0);
        re1 = fma(t[i + 1], y.x, re1);
        im1 = fma(t[i + 1], y.y, im1);
      }
      v = make_double2(re0 + re1, im0 + im1);
    }
    Q = {fma(Q.re, q.re, fma(-Q.im, q.im, P.re)), fma(Q.re, q.im, fma(Q.im, q.re, P.im))};
    P = {fma(P.re, q.re, fma(-P.im, q.im, v.x)), fma(P.re, q.im, fma(P.im, q.re, v.y))};
  }
  const cplx a = cdiv(cmul(q, Q), r), d = cdiv(cmul(z, P), cmul(r, r));
  F[k] = cmul(g, {-a.im + d.re, a.re + d.im}).im;  // g_0 (i S1 / r + z S0 / r^2)
}

// one block per energy: sigma = -ucf * sum_k Im F_k over that energy's K nodes
__global__ void k_bastin_sum(const double* __restrict__ F, int K, double ucf, double* __restrict__ sigma) {
  const double* f = F + (int64_t)blockIdx.x * K;
  double acc = 0.0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) acc += f[k];
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) sigma[blockIdx.x] = -ucf * red[0];
}

}  // namespace

int reconstruct_sigma_bastin_impl(kite_ctx* ctx, const double* mu_dev, int M_avail, int M, int lattice,
                                  int kernel, double param, const Scale& sc, double eta, double kT,
                                  const double* E_host, int K_E, int n_quad, double* sigma_dev) {
  const int K = n_quad > 0 ? n_quad : 2 * M + 64;
  const bool fast =
      Nufft::fits(M) && (K >= kNufftMinNodesBastin || (long long)K * K_E >= kNufftMinNodesBastinAll);
  Nufft nf(M);
  // nodes per batch of energies: theta, weight, F and the taps, or D and V (dense)
  const size_t per_energy = (size_t)K * (fast ? 3 + kTaps + 1 : 3 + 3 * (size_t)M);
  const size_t budget = (size_t)1 << 27;  // doubles (1 GiB)
  const int EB = (int)std::max<size_t>(1, std::min<size_t>((size_t)K_E, budget / per_energy));
  const size_t Kt_max = ((size_t)EB * K + 1) / 2 * 2, Kp = ((size_t)K + 1) / 2 * 2, Ep = ((size_t)K_E + 1) / 2 * 2,
               Mp = ((size_t)M + 1) / 2 * 2;
  const size_t fixed = Mp + 2 * Ep + 4 * Kp + (fast ? (nf.doubles(M) + 2) / 2 * 2 : 2 * (size_t)M * M);
  const size_t total = fixed + Kt_max * (fast ? 3 + kTaps + 1 : 3 + 3 * (size_t)M);
  double* buf = nullptr;
  KITE_CUDA_TRY(ctx, cudaMallocAsync((void**)&buf, total * sizeof(double), ctx->stream));
  double* wk = buf;
  double* E_d = wk + Mp;
  double* thF_d = E_d + Ep;
  double* gx = thF_d + Ep;
  double* gw = gx + Kp;
  double* gab = gw + Kp;
  double* mid = gab + 2 * Kp;  // the transform's buffers, or B
  double* th_d = buf + fixed;
  double* wq_d = th_d + Kt_max;
  double* F = wq_d + Kt_max;
  double* rest = F + Kt_max;  // taps and first taps, or V and D
  cudaStream_t st = ctx->stream;
  const double ucf = lattice == KITE_HONEYCOMB ? 4.0 / sqrt(3.0) : 1.0;
  k_dc_weights<<<(M + 63) / 64, 64, 0, st>>>(M, kernel, param, wk);
  // the Fermi energies in E and theta, then the rule of few nodes
  std::vector<double> in(2 * Ep + (K <= kHostRule ? 2 * Kp : 0));
  for (int i = 0; i < K_E; ++i) {
    in[i] = E_host[i];
    in[Ep + i] = theta_fermi(E_host[i], sc);
  }
  if (K <= kHostRule)
    gauss_rule_host(K, in.data() + 2 * Ep, in.data() + 2 * Ep + Kp);
  else
    gauss_rule(st, K, gab, gx, gw);
  cudaError_t e = cudaMemcpyAsync(E_d, in.data(), in.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  int rc = KITE_OK;
  if (fast) {
    nf.carve(mid);
    rc = nf.rows_to_grid(ctx, mu_dev, M_avail, 1, wk, M);
  } else {
    k_bastin_gamma<<<(int)(((int64_t)M * M + 255) / 256), 256, 0, st>>>(mu_dev, M_avail, M, wk, mid);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (rc == KITE_OK && e != cudaSuccess) rc = cuda_fail(ctx, e, "Bastin set-up");
  for (int b = 0; b < K_E && rc == KITE_OK; b += EB) {
    const int nb = std::min(EB, K_E - b);
    const int64_t Kt = (int64_t)nb * K;
    const int blocks = (int)std::min<int64_t>((Kt + 255) / 256, (int64_t)ctx->num_sms * 8);
    k_fermi_nodes<<<blocks, 256, 0, st>>>(gx, gw, K, E_d + b, thF_d + b, nb, sc.de_plus, sc.de_minus, kT, th_d, wq_d);
    const unsigned nblk = (unsigned)((Kt + kNodeBlock - 1) / kNodeBlock);
    if (fast) {
      double* taps = rest;
      int* j0 = reinterpret_cast<int*>(taps + kTaps * Kt_max);
      k_nufft_taps<<<blocks, 256, 0, st>>>(th_d, wq_d, Kt, nf.Nf, j0, taps);
      k_bastin_nodes<false><<<nblk, kNodeBlock, 0, st>>>(nullptr, reinterpret_cast<const double2*>(nf.grid), nf.L, j0, taps,
                                                  th_d, M, Kt, eta / sc.de_minus, F);
    } else {
      double* V = rest;
      double* D = V + 2 * (size_t)M * Kt_max;
      k_sig_dmat<<<(int)(((int64_t)M * Kt + 255) / 256), 256, 0, st>>>(th_d, wq_d, M, (int)Kt, D);
      dim3 blk(16, 16), grd((unsigned)((Kt + 15) / 16), (unsigned)((M + 15) / 16));
      k_zgemm_real<<<grd, blk, 0, st>>>(mid, 1, D, M, (int)Kt, V);  // V[m][k] = sum_n B_nm D[n][k]
      k_bastin_nodes<true><<<nblk, kNodeBlock, 0, st>>>(reinterpret_cast<const double2*>(V), nullptr, 0, nullptr, nullptr,
                                                 th_d, M, Kt, eta / sc.de_minus, F);
    }
    k_bastin_sum<<<nb, 256, 0, st>>>(F, K, ucf, sigma_dev + b);
    e = cudaGetLastError();
    if (e != cudaSuccess) rc = cuda_fail(ctx, e, "Bastin kernels");
  }
  cudaFreeAsync(buf, st);
  return rc;
}

}  // namespace kite
