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
//   q = chi - sqrt(chi^2 - 1) = 1 / (chi + sqrt(chi^2 - 1)),
// scaled the same way. The degree of a class is the first with both remainders
// below the tolerance (relative to the functions' maximum of 1).
#include <math.h>

#include <mutex>
#include <vector>

#include "letkf_common.cuh"

namespace {

// a[k], b[k], k = 0 .. degree; returns the degree.
int cheb_series(double r, double tol, std::vector<double> &a, std::vector<double> &b) {
  // q without the difference's cancellation (chi >> 1 at small r: 8e-15 of q at r = 0.25)
  const double d = 2.0 / r, chi = 1.0 + d, q = 1.0 / (chi + sqrt(d * (d + 2.0)));
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

// Poles s_j and weights w_j of z^-1/2 ~ sum_j w_j / (z + s_j) on [1, M]: the
// midpoint rule in the elliptic substitution z = -sc^2(u, k'), which gives the best
// rational approximation (Hale, Higham & Trefethen 2008, method 3): with k^2 =
// 1 / M, u_j = (j - 1/2) K' / n, s_j = (sn / cn)^2 and w_j = 2 K' dn / (pi n cn^2) at
// modulus k'. K' and the functions by the arithmetic-geometric mean and descending Landen
// transformations (Abramowitz & Stegun 16.4, 17.6).
void lk_poles(double M, int n, double2 *out) {
  const double pi = 3.14159265358979323846, k = 1.0 / sqrt(M);
  double a[32], c[32], b = k;
  a[0] = 1.0;
  c[0] = sqrt(1.0 - k * k);
  int l = 0;
  while (fabs(c[l]) > 1e-17 && l < 30) {
    a[l + 1] = 0.5 * (a[l] + b);
    c[l + 1] = 0.5 * (a[l] - b);
    b = sqrt(a[l] * b);
    ++l;
  }
  const double K = pi / (2.0 * a[l]);
  for (int j = 0; j < n; ++j) {
    double phi = ldexp(a[l] * (j + 0.5) * K / n, l);
    for (int q = l; q > 0; --q) {
      phi = 0.5 * (phi + asin(c[q] * sin(phi) / a[q]));
    }
    const double sn = sin(phi), cn = cos(phi), dn = sqrt(1.0 - (1.0 - k * k) * sn * sn);
    out[j] = make_double2(sn * sn / (cn * cn), 2.0 * K * dn / (pi * n * cn * cn));
  }
}

std::once_flag g_once;
std::vector<double2> g_poles;
std::vector<float2> g_table32;
std::vector<float4> g_table64;   // pairs of floats: a_k high, low, b_k high, low

// The term up to which a series needs more than floats: from low + 1 on the coefficients,
// weighted by the growth of the recurrences' rounding (the number of steps since), add up
// to less than 2^-27, and so the rounding of these terms in FP32 to less than 2^-51.
int last_in_pairs(const std::vector<double> &a, const std::vector<double> &b, int deg) {
  double s = 0.0, tail = 0.0;
  int k = deg;
  for (; k > 1; --k) {
    s += fmax(fabs(a[k]), fabs(b[k]));
    tail += s;
    if (tail > ldexp(1.0, -27)) break;
  }
  return k;
}

template <typename V, typename F>
void fill_table(std::vector<V> &table, int classes, int ld, double tol, F pair) {
  table.assign((size_t)classes * ld, pair(0.0, 0.0));
  std::vector<double> a, b;
  for (int c = 0; c < classes; ++c) {
    const double r = LK_CHEB_R0 * pow(LK_CHEB_STEP, c);
    const int deg = cheb_series(r, tol, a, b);
    V *row = table.data() + (size_t)c * ld;
    row[0] = pair(2.0 / r, deg);
    if constexpr (sizeof(V) == sizeof(float4)) row[0].w = (float)last_in_pairs(a, b, deg);
    for (int k = 0; k <= deg && k + 1 < ld; ++k) row[k + 1] = pair(a[k], b[k]);
  }
}

void build_tables() {
  fill_table(g_table32, LK_CHEB_CLASSES32, LK_CHEB_LD32, 1e-8,
             [](double x, double y) { return make_float2((float)x, (float)y); });
  g_poles.assign(16, make_double2(0.0, 0.0));
  lk_poles(LK_TRI_MAX, 15, g_poles.data());
  fill_table(g_table64, LK_CHEB_CLASSES64, LK_CHEB_LD64, 1e-17,
             [](double x, double y) {
               const float xh = (float)x, yh = (float)y;
               return make_float4(xh, (float)(x - xh), yh, (float)(y - yh));
             });
}

template <typename V>
cudaError_t upload_table(V **dst, const std::vector<V> &table) {
  cudaError_t e = cudaMalloc((void **)dst, table.size() * sizeof(V));
  if (e == cudaSuccess)
    e = cudaMemcpy(*dst, table.data(), table.size() * sizeof(V), cudaMemcpyHostToDevice);
  return e;
}

}  // namespace

cudaError_t lk_setup_cheb(letkf_ctx *h) {
  std::call_once(g_once, build_tables);
  if (h->precision == 0) {
    const cudaError_t e = upload_table(&h->cheb32, g_table32);
    return e == cudaSuccess ? upload_table(&h->poles, g_poles) : e;
  }
  const cudaError_t e = upload_table(&h->cheb64, g_table64);
  return e == cudaSuccess ? lk_setup_series64(h) : e;
}

bool lk_series64(const letkf_ctx *h) {
  return h->precision == 1 && h->fp64_warm && h->cheb64 != nullptr;
}
