"""The Chebyshev coefficients of (1 + g)^-1/2 and (1 + g)^-1 (letkf_cheb.cu, host code) against
the same series in 60 decimal digits."""
import os
import subprocess
from decimal import Decimal as D, getcontext

import pytest

from paper_1408_7069_gb300 import build

MAIN = """
#include "letkf_cheb.cu"
#include <stdio.h>
cudaError_t lk_setup_series64(letkf_ctx *) { return cudaSuccess; }
int main() {
  std::vector<double> a, b;
  for (int c = 0; c < LK_CHEB_CLASSES64; ++c) {
    const double r = LK_CHEB_R0 * pow(LK_CHEB_STEP, c);
    const int deg = cheb_series(r, 1e-17, a, b);
    printf("%.17g %d", r, deg);
    for (int k = 0; k <= deg; ++k) printf(" %.17g %.17g", a[k], b[k]);
    printf("\\n");
  }
}
"""


@pytest.fixture(scope="module")
def series(tmp_path_factory):
    d = tmp_path_factory.mktemp("cheb")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    "--expt-relaxed-constexpr", str(d / "main.cu"), "-o", str(d / "main")],
                   check=True)
    rows = []
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    for line in subprocess.run([str(d / "main")], check=True, capture_output=True, text=True,
                               env=env).stdout.splitlines():
        v = line.split()
        rows.append((float(v[0]), int(v[1]), [float(x) for x in v[2::2]], [float(x) for x in v[3::2]]))
    assert len(rows) == 24
    return rows


def exact(r, deg):
    """a_k and b_k, k = 0 .. deg, by Miller's algorithm and in closed form."""
    getcontext().prec = 60
    chi = 1 + 2 / D(r)
    q = 1 / (chi + (chi * chi - 1).sqrt())
    n = deg + 200
    a = [D(0)] * (n + 2)
    a[n] = D("1e-200")
    for k in range(n, 0, -1):
        a[k - 1] = (2 * k * chi * a[k] - (k + D("0.5")) * a[k + 1]) / (k - D("0.5"))
    eps = [1] + [2] * n
    sa = sum(e * x for e, x in zip(eps, a))
    sign = [1 - 2 * (k & 1) for k in range(deg + 1)]
    return ([s * e * x / sa for s, e, x in zip(sign, eps, a)],
            [s * e * q ** k * (1 - q) / (1 + q) for k, (s, e) in enumerate(zip(sign, eps))], q)


def test_coefficients_to_fp64_rounding(series):
    """q, the ratio of successive b_k, to a few units of 2^-53 (chi's rounding enters it up to
    3.4 times at the largest class; a root, an addition and a division follow), and so each
    coefficient to that times its order; the functions' errors, the sums of these, likewise."""
    u = 2.0 ** -53
    for r, deg, a, b in series:
        ea, eb, q = exact(r, deg)
        assert abs(D(-b[1]) / D(b[0]) / 2 / q - 1) <= 10 * u, r
        for got, want in ((a, ea), (b, eb)):
            err = sum(abs(D(g) - w) for g, w in zip(got, want))
            assert err <= 10 * D(u) * sum((k + 1) * abs(w) for k, w in enumerate(want)), r


def test_the_series_are_the_functions(series):
    """At points of [0, r], to the truncation (1e-17 of the remainder) and the rounding."""
    u = 2.0 ** -53
    for r, deg, a, b in series:
        for i in range(9):
            g = D(r) * i / 8
            x = 2 * g / D(r) - 1
            t0, t1 = D(1), x
            sa, sb = D(a[0]) + D(a[1]) * x, D(b[0]) + D(b[1]) * x
            for k in range(2, deg + 1):
                t0, t1 = t1, 2 * x * t1 - t0
                sa, sb = sa + D(a[k]) * t1, sb + D(b[k]) * t1
            tol = D(3e-17) + 10 * D(u) * sum((k + 1) * abs(D(v)) for k, v in enumerate(b))
            assert abs(sa - 1 / (1 + g).sqrt()) <= tol and abs(sb - 1 / (1 + g)) <= tol, (r, i)
