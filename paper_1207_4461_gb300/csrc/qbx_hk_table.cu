// qbx_hk_table.cu -- H0, H1 for complex k along the ray z = k rho.
//
// A call with complex k evaluates H_n(k rho) at every (centre, source) pair;
// the series / Miller / asymptotic evaluation (hankel01_cplx) costs far more
// than the real-axis fits.  But one call has one k, so every argument lies on
// the ray z = (k/|k|) |z|: the modulated amplitudes B_n = H_n(z) e^{-i(z -
// pi/4)} (DLMF 10.17.5: smooth in s = |z|^{-1/2}, no oscillation) are fitted
// once per k on the intervals of the real-axis table, by Chebyshev
// interpolation at QBX_HK_DEG + 1 nodes per interval, and the pair kernels
// evaluate them like the real-axis fits (KW<cplx>).  The values at the nodes
// are the integral
//   B_n(z) = (2/(pi z))^{1/2} e^{-i n pi/2} / Gamma(n + 1/2)
//            int_0^inf e^{-t} t^{n-1/2} (1 + i t/(2z))^{n-1/2} dt
// (DLMF 10.32.8 with K_n(-iz) = (pi i/2) e^{i n pi/2} H_n(z)), t = u^2, by the
// trapezoidal rule in u, whose error falls as e^{-2 pi |Im sqrt(2 i z)| / h}:
// step 0.2, 32 points, 7e-16 at |z| >= 1.9 for every angle in [0, pi/2]
// (against 90-digit values).  Nothing cancels, where the series and Miller
// sums J + iY lose e^{2 Im z} (k = 2 + 6i on the 48-panel starfish: S off by
// 1.4e-10 with those, 3e-15 with the integral; the table takes 56 us instead
// of 922).
#include <cuda_runtime.h>
#include "qbx_apply_impl.cuh"
#include "qbx_internal.h"

namespace qbx {
namespace {

constexpr int kN = QBX_HK_DEG + 1;   // nodes and coefficients per interval

constexpr int kPts = 32;             // quadrature points
constexpr double kStep = 0.2;
constexpr int kSplit = 4;            // threads per node
constexpr int kPerCta = 8;           // intervals per CTA

// One thread per (interval, node, quarter of the quadrature), then one per
// interval for the fit: about 60 complex square roots deep instead of 400.
// Interval i has width w = 2^-LOG2_PER_UNIT in s, [i w, (i+1) w].
__global__ void __launch_bounds__(kPerCta * kN * kSplit) k_hk_table(double kre, double kim, double* tab) {
  __shared__ cplx s_f[kPerCta][2][kN][kSplit];
  const double w = 1.0 / (double)(1 << QBX_HK_LOG2_PER_UNIT);
  const double half = 0.5 * w;
  {
    const int part = threadIdx.x % kSplit, j = threadIdx.x / kSplit % kN, q = threadIdx.x / (kSplit * kN);
    const int i = min((int)blockIdx.x * kPerCta + q, QBX_HK_NI - 1);
    const double ka = hypot(kre, kim);
    const double s = (i + 0.5) * w + half * cos(3.14159265358979323846 * (j + 0.5) / kN);
    const cplx iz{s * s * kre / ka, -s * s * kim / ka};   // 1/z, z = (k / |k|) / s^2
    cplx s0{0.0, 0.0}, s1{0.0, 0.0};
    for (int m = part; m < kPts; m += kSplit) {
      const double u2 = (m * kStep) * (m * kStep);
      const double wt = (m == 0 ? 1.0 : 2.0) * kStep * exp(-u2);
      const cplx r = csqrt_(cplx{1.0 - 0.5 * u2 * iz.im, 0.5 * u2 * iz.re});
      s0 = s0 + wt * cinv(r);
      s1 = s1 + (wt * u2) * r;
    }
    const cplx pre = 0.56418958354775628695 * csqrt_(0.63661977236758134308 * iz);   // (2/(pi z))^{1/2} / Gamma(1/2)
    const cplx b1 = pre * s1;
    s_f[q][0][j][part] = pre * s0;
    s_f[q][1][j][part] = cplx{2.0 * b1.im, -2.0 * b1.re};   // e^{-i pi/2} / (1/2)
  }
  __syncthreads();
  const int q = threadIdx.x, i = blockIdx.x * kPerCta + q;
  if (q >= kPerCta || i >= QBX_HK_NI) return;
  cplx f[2][kN];
  for (int n = 0; n < 2; ++n)
    for (int j = 0; j < kN; ++j) {
      f[n][j] = s_f[q][n][j][0];
      for (int c = 1; c < kSplit; ++c) f[n][j] = f[n][j] + s_f[q][n][j][c];
    }
  // monomial coefficients of T_0 .. T_{kN-1} in x (T_{m+1} = 2 x T_m - T_{m-1})
  double T[kN][kN];
  for (int m = 0; m < kN; ++m)
    for (int d = 0; d < kN; ++d) T[m][d] = 0.0;
  T[0][0] = 1.0;
  if (kN > 1) T[1][1] = 1.0;
  for (int m = 1; m + 1 < kN; ++m)
    for (int d = 0; d < kN; ++d) T[m + 1][d] = (d > 0 ? 2.0 * T[m][d - 1] : 0.0) - T[m - 1][d];
  double* out = tab + (size_t)i * kN * 4;
  for (int n = 0; n < 2; ++n) {
    // Chebyshev coefficients c_m = (2 - [m = 0]) / kN sum_j f_j T_m(x_j)
    cplx c[kN];
    for (int m = 0; m < kN; ++m) {
      cplx acc{0.0, 0.0};
      for (int j = 0; j < kN; ++j) acc = acc + cos(3.14159265358979323846 * m * (j + 0.5) / kN) * f[n][j];
      c[m] = ((m == 0 ? 1.0 : 2.0) / kN) * acc;
    }
    // p(x) = sum_m c_m T_m(x) in monomials of x, then of u = half x
    double scale = 1.0;
    for (int d = 0; d < kN; ++d) {
      cplx b{0.0, 0.0};
      for (int m = d; m < kN; ++m) b = b + T[m][d] * c[m];
      out[d * 4 + 2 * n] = b.re * scale;
      out[d * 4 + 2 * n + 1] = b.im * scale;
      scale /= half;
    }
  }
}

__global__ void k_debug_hankel_ray(double kre, double kim, const double* tab, const double* rho, int n, cplx* h0,
                                   cplx* h1) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  KW<cplx> kw;
  kw.init(kre, kim, tab);
  double inv, r, y;
  kw.geom(rho[t] * rho[t], inv, r, y);
  cplx a, b, tz;
  kw.hankel(r, inv, y, a, b, tz);
  h0[t] = a;
  h1[t] = b;
}

}  // namespace

int hk_table_doubles() { return QBX_HK_NI * kN * 4; }

cudaError_t launch_hk_table(double kre, double kim, double* tab, cudaStream_t st) {
  k_hk_table<<<(QBX_HK_NI + kPerCta - 1) / kPerCta, kPerCta * kN * kSplit, 0, st>>>(kre, kim, tab);
  return cudaGetLastError();
}

cudaError_t launch_debug_hankel_ray(double kre, double kim, const double* tab, const double* rho, int n, void* h0,
                                    void* h1, cudaStream_t st) {
  k_debug_hankel_ray<<<(n + 127) / 128, 128, 0, st>>>(kre, kim, tab, rho, n, (cplx*)h0, (cplx*)h1);
  return cudaGetLastError();
}

}  // namespace qbx
