// kite_nufft.cuh -- device kernels of the conductivity reconstructions' quadrature: the
// Gauss-Legendre rule, and cosine sums sum_n c_n cos(n theta_k) at many nodes theta_k.
//
// GB300's FP64 pipe does two multiply-adds per SM and cycle, so a dense product of M
// coefficients with cos(n theta_k) (2 M FP64 multiply-adds per complex row and node) is what
// the conductivities spent their time on.  Here a row costs one FFT and each node 16 taps:
// the non-uniform fast Fourier transform with the "exponential of semicircle" window of
// Barnett, Magland and af Klinteberg (SIAM J. Sci. Comput. 41, C479 (2019)),
//   phi(x) = exp(beta (sqrt(1 - (2x/w)^2) - 1)),  w = 16 taps, beta = 2.3 w, on a grid of Nf
// points: sum_n c_n cos(n theta) = sum_j b_j phi(theta/h - j), h = 2 pi/Nf, with
// b_j = sum_n (c_n / phihat_n) cos(n j h) and phihat_n the window's Fourier transform.  The
// sums are closer to extended-precision ones than FP64 sums of cos(n theta) are (see
// kNufftMinM).
#pragma once

#include <math.h>
#include <stdint.h>

namespace kite {
namespace {

constexpr int kTaps = 16;
constexpr double kBeta = 2.3 * kTaps;
constexpr double kPi = 3.141592653589793;
// Orders the transform is used for: below, its error is not smaller than the dense sum's (1.0
// to 1.8 of it at M = 32 .. 48, 0.9 at 64, 0.2 at 256, 0.1 at 512, against extended precision)
// and there is little to gain; above, a row no longer fits an SM's shared memory.
constexpr int kNufftMinM = 64, kNufftMaxM = 2048;
// Nodes the transform is used for.  It costs an FFT per row whatever the number of nodes, the
// dense product M multiply-adds per row and node.  GB300, us per call, dense / transform:
// optical sums (two products) at 64 nodes 164 / 195 (M = 64), 339 / 407 (256), 1245 / 1560
// (1024), 3439 / 4909 (2048), at 96 nodes 685 / 647 (M = 512), 1510 / 1569 (1024); Bastin's
// (one product) at 128 nodes of one energy 138 / 251 (M = 64), 424 / 1170 (512), 1013 / 2419
// (1024), at 32 nodes of eight energies 137 / 270, 568 / 1253, 1427 / 2699.  The dense side wins
// further at small M, but its errors are the larger ones there: the line stays below the
// default rule's 2 M + 64 nodes.
constexpr int kNufftMinNodes = 65, kNufftMinNodesBastin = 129, kNufftMinNodesBastinAll = 257;

// Coefficients ((2j-1)/j, (j-1)/j) of the Legendre recurrence
// P_j = (2j-1)/j z P_{j-1} - (j-1)/j P_{j-2}, j = 1..K.
__global__ void k_legendre_coef(int K, double2* __restrict__ ab) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x + 1; j <= K; j += gridDim.x * blockDim.x)
    ab[j - 1] = make_double2((2.0 * j - 1.0) / j, (j - 1.0) / j);
}

// Gauss-Legendre nodes and weights on [-1, 1], ascending, the nodes as u = 1 + x: Newton's
// iteration on P_K from Tricomi's estimate, sixteen lanes per root z = 1 + d, d in (-1, 0].
// The recurrence runs on P_j and D_j = P_j - P_{j-1},
//   D_j = (j-1)/j D_{j-1} + (2j-1)/j d P_{j-1},  P_j = P_{j-1} + D_j
// (Reinsch's form: no cancellation near z = 1, so d and the weights keep their relative
// accuracy, 1e-15 and 2e-14 at K = 1088, where the three-term form in z loses 1e-11 of the
// end weights; at T = 0 the integrand does not vanish at theta_F).  A lane takes a sixteenth
// of it as a 2 x 2 transfer matrix: the serial chain of K steps would be the whole cost (the
// host took 15 ms for K = 1088).
constexpr int kGaussBlock = 64;
__global__ void __launch_bounds__(kGaussBlock) k_gauss_legendre(int K, const double2* __restrict__ ab,
                                                                double* __restrict__ u, double* __restrict__ w) {
  const int lane = threadIdx.x & 31, part = lane & 15;
  const int root = blockIdx.x * (kGaussBlock / 16) + (int)(threadIdx.x >> 4);
  const int half = (K + 1) / 2;
  const int i = min(root, half - 1);  // surplus lanes repeat the last root
  const double dK = (double)K;
  const double sh = sin(0.5 * kPi * (i + 0.75) / (dK + 0.5)), c0 = -2.0 * sh * sh;
  double d = c0 - (0.125 / (dK * dK) - 0.125 / (dK * dK * dK)) * (1.0 + c0);
  const int j0 = (int)((long long)K * part / 16), j1 = (int)((long long)K * (part + 1) / 16);
  double wt = 0.0;
  for (int it = 0; it < 9; ++it) {
    // what (P, D) = (1, 0) and (0, 1) at j0 become at j1
    double a1 = 1.0, a0 = 0.0, b1 = 0.0, b0 = 1.0;
    for (int j = j0; j < j1; ++j) {
      const double2 c = ab[j];
      const double cd = c.x * d;
      a0 = fma(cd, a1, c.y * a0);
      a1 += a0;
      b0 = fma(cd, b1, c.y * b0);
      b1 += b0;
    }
    // product of the sixteen matrices, the later one on the left
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const double pa1 = __shfl_xor_sync(0xffffffffu, a1, o), pa0 = __shfl_xor_sync(0xffffffffu, a0, o);
      const double pb1 = __shfl_xor_sync(0xffffffffu, b1, o), pb0 = __shfl_xor_sync(0xffffffffu, b0, o);
      const bool later = (part & o) != 0;  // this lane's matrix is the later one
      const double la1 = later ? a1 : pa1, la0 = later ? a0 : pa0, lb1 = later ? b1 : pb1, lb0 = later ? b0 : pb0;
      const double ea1 = later ? pa1 : a1, ea0 = later ? pa0 : a0, eb1 = later ? pb1 : b1, eb0 = later ? pb0 : b0;
      a1 = fma(la1, ea1, lb1 * ea0);
      a0 = fma(la0, ea1, lb0 * ea0);
      b1 = fma(la1, eb1, lb1 * eb0);
      b0 = fma(la0, eb1, lb0 * eb0);
    }
    // (P_K, D_K): the image of (P_0, D_0) = (1, 0); (1 - z^2) P'_K = K (P_{K-1} - z P_K)
    const double om = -d * (2.0 + d);  // 1 - z^2
    const double dp = -dK * fma(d, a1, a0) / om, dz = a1 / dp;
    // the weight 2 / ((1 - z^2) P'^2) at the root, from its logarithmic derivative at z,
    // (-2 z + 2 K (K + 1) dz) / (1 - z^2) (Legendre's equation): without the second term the
    // last step, up to 4e-9, left every weight too large, by 6e-14 at most and 1 to 3e-15 in the
    // sum at K = 66 .. 192
    wt = 2.0 / (om * dp * dp) * (1.0 + dz * fma(-dK * (dK + 1.0), dz, 2.0 * (1.0 + d)) / om);
    d -= dz;
    // the next step would be below z / om * dz^2
    if (__all_sync(0xffffffffu, !(fabs(dz) > 4e-9 * om))) break;
  }
  if (root < half && part == 0) {
    u[K - 1 - i] = 2.0 + d;
    u[i] = -d;
    w[i] = w[K - 1 - i] = wt;
  }
}

// Quadrature nodes theta and weights of K_E Fermi energies: [theta_F, pi] (kT = 0) or
// [0, pi] weighted by the Fermi function (kT > 0).  theta_F comes from the host: the integral
// feels its last place, and the device's arc cosine is an ulp or two off.  The exponent is
// (E - E_F)/kT = de_minus (cos t - cos theta_F)/kT as a product of sines, whose relative error
// stays at the rounding for nodes next to the Fermi energy (a difference of cosines divided by
// a small kT does not); Fermi energies outside the band take the difference.
__host__ __device__ inline void fermi_node(double u, double w, double E_F, double theta_F, double de_plus,
                                           double de_minus, double kT, double* theta, double* wq) {
  const double thF = kT > 0.0 ? 0.0 : theta_F;
  const double t = thF + (kPi - thF) * 0.5 * u;
  double v = w * 0.5 * (kPi - thF);
  if (kT > 0.0) {
    const double eF = (E_F - de_plus) / de_minus;
    const double d = fabs(eF) < 1.0 ? -2.0 * sin(0.5 * (t + theta_F)) * sin(0.5 * (t - theta_F)) : cos(t) - eF;
    v /= (1.0 + exp(d * de_minus / kT));
  }
  *theta = t;
  *wq = v;
}
__global__ void k_fermi_nodes(const double* __restrict__ u, const double* __restrict__ w, int K,
                              const double* __restrict__ E_F, const double* __restrict__ theta_F, int K_E,
                              double de_plus, double de_minus, double kT,
                              double* __restrict__ theta, double* __restrict__ wq) {
  const int64_t n = (int64_t)K * K_E;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / K), k = (int)(e - (int64_t)i * K);
    fermi_node(u[k], w[k], E_F[i], theta_F[i], de_plus, de_minus, kT, &theta[e], &wq[e]);
  }
}

__device__ __forceinline__ double es_window(double x) {  // |x| <= kTaps/2
  const double u = x * (2.0 / kTaps);
  return exp(kBeta * (sqrt(fmax(0.0, 1.0 - u * u)) - 1.0));
}

// inv[n] = 1 / phihat_n, n < M: the window's transform by the trapezoidal rule at quarter grid
// steps (its aliases lie where the transform is below 1e-16), a warp per mode; tw[k] =
// exp(2 pi i k / Nf), k < Nf/2.
__global__ void __launch_bounds__(128) k_nufft_tables(int M, int Nf, double* __restrict__ inv,
                                                      double2* __restrict__ tw) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, n = t >> 5, lane = t & 31;
  if (n < M) {  // (warp-uniform)
    double v = es_window(0.25 * lane) * cospi(0.5 * (double)lane * n / Nf) * (lane ? 2.0 : 1.0);
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if (lane == 0) inv[n] = 1.0 / (0.25 * v);
  }
  if (t < Nf / 2) {
    double sn, cs;
    sincospi(2.0 * t / Nf, &sn, &cs);
    tw[t] = make_double2(cs, sn);
  }
}

// Per node: first grid index and the 16 taps (times the node's weight and 2/pi).
__global__ void k_nufft_taps(const double* __restrict__ theta, const double* __restrict__ wq, int64_t n, int Nf,
                             int* __restrict__ j0, double* __restrict__ taps) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    // theta/h with 1/(2 pi) in two parts: the position's rounding error, times up to M, would
    // otherwise be the largest error of the sum (as the rounding of n theta is in cos(n theta))
    const double hi = 0.15915494309189535 * Nf, lo = -9.839338337591243e-18 * Nf;
    const double xg = theta[k] * hi, err = fma(theta[k], hi, -xg) + theta[k] * lo;
    const int j = (int)ceil(xg - kTaps / 2);
    j0[k] = j + kTaps / 2;  // rows are stored from grid index -kTaps/2
    const double f = (2.0 / kPi) * wq[k];
    for (int t = 0; t < kTaps; ++t) taps[(int64_t)t * n + k] = f * es_window(((double)(j + t) - xg) - err);
  }
}

// Grid points: a power of two, at least four times the highest mode on either side of zero up
// to M = 256, twice above (the window's error is then below the rounding of the dense sum).
__host__ __device__ inline int nufft_grid(int M) {
  int n = 64;
  while (n < (M <= 256 ? 8 : 4) * M) n <<= 1;
  return n;
}
// Stored grid values of a row: indices -8 .. Nf/2 + 8 (even function: b_-j = b_j).
__host__ __device__ inline int nufft_row(int Nf) { return Nf / 2 + kTaps + 1; }

// Rows of the cosine sums on the grid, one block per row, an in-place radix-2 FFT in shared
// memory (bit-reversed load).  With the weights w_n = (2 - d_n0) g_n, row r < M:
//   kind 0: c_m = -w_r w_m mu_rm / 4 (rows of Gamma); rows r >= M: columns of it
//   kind 1: c_n = w_r w_n (conj(mu_rn) + mu_nr) / 4 (columns of the Hermitian fold)
__global__ void __launch_bounds__(256) k_cos_fft(const double* __restrict__ mu, int M_avail, int M, int kind,
                                                 const double* __restrict__ w, const double* __restrict__ inv,
                                                 const double2* __restrict__ tw, int Nf, int logN,
                                                 double2* __restrict__ out) {
  extern __shared__ __align__(16) double2 f[];
  const int r = blockIdx.x < (unsigned)M ? blockIdx.x : blockIdx.x - M;
  const bool col = blockIdx.x >= (unsigned)M;
  const double wr = 0.25 * w[r];
  for (int i = threadIdx.x; i < Nf; i += blockDim.x) f[i] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    const double2* p = reinterpret_cast<const double2*>(mu);
    double2 c;
    if (kind == 0) {
      c = col ? p[(int64_t)m * M_avail + r] : p[(int64_t)r * M_avail + m];
      c.x = -c.x;
      c.y = -c.y;
    } else {
      const double2 a = p[(int64_t)r * M_avail + m], b = p[(int64_t)m * M_avail + r];
      c = make_double2(a.x + b.x, b.y - a.y);
    }
    const double s = wr * w[m] * inv[m] * (m ? 0.5 : 1.0);
    c.x *= s;
    c.y *= s;
    f[__brev((unsigned)m) >> (32 - logN)] = c;
    if (m) f[__brev((unsigned)(Nf - m)) >> (32 - logN)] = c;
  }
  for (int len = 1; len < Nf; len <<= 1) {
    __syncthreads();
    const int step = Nf / (2 * len);
    for (int b = threadIdx.x; b < Nf / 2; b += blockDim.x) {
      const int k = b & (len - 1), i = ((b - k) << 1) + k;
      const double2 t = tw[k * step], u = f[i], v = f[i + len];
      const double vr = fma(v.x, t.x, -(v.y * t.y)), vi = fma(v.x, t.y, v.y * t.x);
      f[i] = make_double2(u.x + vr, u.y + vi);
      f[i + len] = make_double2(u.x - vr, u.y - vi);
    }
  }
  __syncthreads();
  const int L = nufft_row(Nf);
  double2* o = out + (int64_t)blockIdx.x * L;
  for (int i = threadIdx.x; i < L; i += blockDim.x) {
    const int j = i - kTaps / 2;
    o[i] = f[j < 0 ? -j : j];  // (j <= Nf/2 + 8 < Nf: the transform itself is even)
  }
}

// U[row][k] = sum_t taps[t][k] b_row[j0[k] + t] for eight rows per thread.
constexpr int kApplyRows = 8;
__global__ void __launch_bounds__(128) k_nufft_apply(const double2* __restrict__ grid, int L, int rows, int K,
                                                     const int* __restrict__ j0, const double* __restrict__ taps,
                                                     double2* __restrict__ U) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  double t[kTaps];
#pragma unroll
  for (int q = 0; q < kTaps; ++q) t[q] = taps[(int64_t)q * K + k];
  const int r0 = blockIdx.y * kApplyRows, r1 = min(rows, r0 + kApplyRows), j = j0[k];
  for (int r = r0; r < r1; ++r) {
    const double2* b = grid + (int64_t)r * L + j;
    double re0 = 0.0, im0 = 0.0, re1 = 0.0, im1 = 0.0;
#pragma unroll
    for (int q = 0; q < kTaps; q += 2) {
      const double2 u = b[q], v = b[q + 1];
      re0 = fma(t[q], u.x, re0);
      im0 = fma(t[q], u.y, im0);
      re1 = fma(t[q + 1], v.x, re1);
      im1 = fma(t[q + 1], v.y, im1);
    }
    U[(int64_t)r * K + k] = make_double2(re0 + re1, im0 + im1);
  }
}

}  // namespace
}  // namespace kite
