// Coefficient tables of the Chebyshev series that replace the eigensolve of
// well-conditioned node and domain problems (host code).
//
// With A = alpha (I + G / alpha) and the spectrum of G / alpha in [0, r], the
// analysis applies (1 + g)^-1/2 and (1 + g)^-1 to vectors. In x = 2 g / r - 1,
// 1 + g = (r / 2)(chi + x), chi = (2 + r) / r, and
//   (chi + cos t)^-1/2 = (sqrt(2) / pi) sum_k eps_k (-1)^k Q_{k-1/2}(chi) cos(k t),
// eps_0 = 1, eps_k = 2 (Heine's expansion; Q: Legendre functions of the second
// kind). Q_{k-1/2} is the minimal solution of its three-term recurrence
//   (k + 1/2) Q_{k+1/2} = 2 k chi Q_{k-1/2} - (k - 1/2) Q_{k-3/2},
// so it is run downwards (Miller's algorithm) and scaled by the series' value at
// x = -1, where every term is positive and the sum is f = 1. For the inverse
//   (chi + cos t)^-1 = (chi^2 - 1)^-1/2 sum_k eps_k (-q)^k cos(k t),
//   q = chi - sqrt(chi^2 - 1),
// scaled the same way. The degree of a class is the first with both remainders
// below the tolerance (relative to the functions' maximum of 1).
#include <math.h>

#include <mutex>
#include <vector>

#include "letkf_common.cuh"

namespace {

// a[k], b[k], k = 0 .. degree; returns the degree.
int cheb_series(double r, double tol, std::vector<double> &a, std::vector<double> &b) {
  const double chi = (2.0 + r) / r, q = chi - sqrt(chi * chi - 1.0);
  // terms decay like q^k: far enough for the smallest tolerance
  const int n = (int)ceil(log(tol * 1e-3) / log(q)) + 16;
  a.assign(n + 2, 0.0);
  b.assign(n + 2, 0.0);
  a[n] = 1e-280;
  for (int k = n; k >= 1; --k) {
    a[k - 1] = (2.0 * k * chi * a[k] - (k + 0.5) * a[k + 1]) / (k - 0.5);
    if (a[k - 1] > 1e200)
      for (int j = k - 1; j <= n; ++j) a[j] *= 1e-250;
  }
  double sa = 0.0, sb = 0.0;
  for (int k = n; k >= 0; --k) {
    const double eps = k ? 2.0 : 1.0;
    a[k] *= eps;
    b[k] = eps * pow(q, k);
    sa += a[k];
    sb += b[k];
  }
  double ta = 0.0, tb = 0.0;
  int deg = n;
  for (int k = n; k >= 1; --k) {
    ta += a[k] / sa;
    tb += b[k] / sb;
    if (ta > tol || tb > tol) {
      deg = k;
      break;
    }
    deg = k - 1;
  }
  for (int k = 0; k <= n; ++k) {
    a[k] *= ((k & 1) ? -1.0 : 1.0) / sa;
    b[k] *= ((k & 1) ? -1.0 : 1.0) / sb;
  }
  return deg < 1 ? 1 : deg;
}

std::once_flag g_once;
std::vector<float2> g_table32;

void build_tables() {
  g_table32.assign((size_t)LK_CHEB_CLASSES32 * LK_CHEB_LD32, make_float2(0.f, 0.f));
  std::vector<double> a, b;
  for (int c = 0; c < LK_CHEB_CLASSES32; ++c) {
    const double r = LK_CHEB_R0 * pow(LK_CHEB_STEP, c);
    const int deg = cheb_series(r, 1e-8, a, b);
    float2 *row = g_table32.data() + (size_t)c * LK_CHEB_LD32;
    row[0] = make_float2((float)(2.0 / r), (float)deg);
    for (int k = 0; k <= deg && k + 1 < LK_CHEB_LD32; ++k)
      row[k + 1] = make_float2((float)a[k], (float)b[k]);
  }
}

}  // namespace

cudaError_t lk_setup_cheb(letkf_ctx *h) {
  std::call_once(g_once, build_tables);
  cudaError_t e = cudaMalloc((void **)&h->cheb32, g_table32.size() * sizeof(float2));
  if (e == cudaSuccess)
    e = cudaMemcpy(h->cheb32, g_table32.data(), g_table32.size() * sizeof(float2),
                   cudaMemcpyHostToDevice);
  return e;
}
