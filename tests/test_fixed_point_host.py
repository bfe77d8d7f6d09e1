"""The fixed-point relaxation of FP64 nodes (csrc/fixed64.cuh), compiled for the host:
against the same formulas in extended precision, beside the double form it stands in for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <limits>
#include "fixed64.cuh"
#include "d3q19.cuh"
using namespace lbm;
typedef long double R;

static void reference(const double* h, double omega, const double* tf, R* out) {
  R rho = 0, j[3] = {0, 0, 0};
  for (int k = 0; k < 19; ++k) {
    rho += h[k];
    for (int a = 0; a < 3; ++a) j[a] += R(ca(k, a)) * h[k];
  }
  R u[3], uu = 0;
  for (int a = 0; a < 3; ++a) { u[a] = (j[a] + tf[a]) / rho; uu += u[a] * u[a]; }
  for (int k = 0; k < 19; ++k) {
    const R cu = cx(k) * u[0] + cy(k) * u[1] + cz(k) * u[2];
    const R eq = R(w36(k)) / 36 * rho * (1 + 3 * cu + R(4.5) * cu * cu - R(1.5) * uu);
    out[k] = h[k] + R(omega) * (eq - h[k]);
  }
}

// the double form of the sweep
static void in_double(const double* f, double omega, const double* tf, double* h) {
  double rho = 0, j[3] = {0, 0, 0}, v[3];
  for (int k = 0; k < 19; ++k) {
    rho += f[k];
    for (int a = 0; a < 3; ++a) j[a] += ca(k, a) * f[k];
  }
  double jv = 0;
  for (int a = 0; a < 3; ++a) { j[a] += tf[a]; v[a] = 1.5 * (j[a] / rho); jv += j[a] * v[a]; }
  const double b = rho - jv, keep = 1 - omega;
  for (int k = 0; k < 19; ++k) {
    const double ow = omega * (double(w36(k)) / 36);
    const double cj = cx(k) * j[0] + cy(k) * j[1] + cz(k) * j[2], cv = cx(k) * v[0] + cy(k) * v[1] + cz(k) * v[2];
    const double a = 3 * ow * cj;
    h[k] = keep * f[k] + (a * cv + ow * b + a);
  }
}

static int fail(const char* what, double a, double b) { std::printf("%s: %g %g\n", what, a, b); return 1; }

int main() {
  srand48(7);
  auto rnd = [] { return 2 * drand48() - 1; };
  const double none[3] = {0, 0, 0};
  for (double rho0 : {1.0, 1.9, 0.7, 1e-3, 5e10})
    for (double tau : {0.501, 0.6, 1.0, 2.0, 1e3})
      for (double umax : {0.0, 1e-3, 0.05, 0.18})
        for (int forced = 0; forced < 2; ++forced) {
          const double omega = 1 / tau;
          double tf[3] = {0, 0, 0};
          if (forced) for (double& t : tf) t = 1e-3 * rho0 * rnd();
          const FixedArgs fx = make_fixed(rho0, omega, tf);
          if (!fx.on) return fail("off", rho0, tau);
          double worst = 0, worst_double = 0, mass = 0;
          long taken = 0;
          for (int n = 0; n < 4000; ++n) {
            double u[3], h[19], d[19], g[19];
            for (double& x : u) x = umax * rnd();
            const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
            for (int k = 0; k < 19; ++k) {
              const double cu = cx(k) * u[0] + cy(k) * u[1] + cz(k) * u[2];
              h[k] = w36(k) / 36.0 * rho0 * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu) * (1 + 0.05 * rnd());
            }
            if (!fixed_in_range(h, fx)) continue;
            ++taken;
            R q[19];
            reference(h, omega, tf, q);
            in_double(h, omega, tf, d);
            int64_t f[19];
            for (int k = 0; k < 19; ++k) {
              f[k] = fixed_in(h[k], fx);
              if (double(f[k]) * fx.unit_in != h[k]) return fail("conversion", h[k], double(f[k]) * fx.unit_in);
            }
            FixedSums s = fixed_sums(f);
            s.x += fx.force[0];
            s.y += fx.force[1];
            s.z += fx.force[2];
            fixed_relax(f, s, fx, g);
            if (tau == 1.0) {  // the products with zero left out
              double t[19];
              fixed_relax_to<true>(f, s, fx, t);
              for (int k = 0; k < 19; ++k)
                if (t[k] != g[k]) return fail("tau = 1", t[k], g[k]);
            }
            for (int k = 0; k < 19; ++k) {
              const double e = double(std::fabs(R(g[k]) - q[k])) / rho0, ed = double(std::fabs(R(d[k]) - q[k])) / rho0;
              worst = e > worst ? e : worst;
              worst_double = ed > worst_double ? ed : worst_double;
              mass += double((R(g[k]) - h[k]) / rho0);
            }
          }
          if (taken < 3000) return fail("few nodes taken", double(taken), umax);
          // the last place of the rest population (rho0 / 3, up to 2^-53 rho0 for a density
          // scale just above a power of two) sets the largest error: half of it, and a
          // unit of S 2^-63 <= rho0 2^-60 for each of the up to 16 roundings of 12 o
          if (worst > 0x1p-54 * 1.1 + 0x1p-56) return fail("error", worst, worst_double);
          if (worst > 1.6 * worst_double) return fail("error beside double", worst, worst_double);
          if (std::fabs(mass / taken) > 0x1p-53) return fail("mass drift", mass / taken, tau);
        }
  // what the windows refuse: one population out of line at a time
  const FixedArgs fx = make_fixed(1.0, 1.25, none);
  double h[19];
  for (int k = 0; k < 19; ++k) {
    for (double bad : {0.0, -0.0, -0.02, 1e-300, 4.8e-4, 0.6, 1e300, std::numeric_limits<double>::infinity(),
                       -std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN()}) {
      for (int i = 0; i < 19; ++i) h[i] = w36(i) / 36.0;
      if (!fixed_in_range(h, fx)) return fail("rest refused", k, bad);
      h[k] = bad;
      if (fixed_in_range(h, fx)) return fail("taken", k, bad);
    }
    // the edges of the window of k
    const double lo = k == 18 ? 0x1p-4 : 0x1p-10, hi = k < 6 ? 0x1p-3 : k < 18 ? 0x1p-4 : 0x1p-1;
    for (int i = 0; i < 19; ++i) h[i] = w36(i) / 36.0;
    h[k] = lo;
    if (!fixed_in_range(h, fx)) return fail("low edge", k, lo);
    h[k] = std::nextafter(lo, 0.0);
    if (fixed_in_range(h, fx)) return fail("below the low edge", k, lo);
    h[k] = std::nextafter(hi, 0.0);
    if (!fixed_in_range(h, fx)) return fail("high edge", k, hi);
    h[k] = hi;
    if (fixed_in_range(h, fx)) return fail("above the high edge", k, hi);
  }
  // the corners of all windows at once: no intermediate may overflow
  for (double tau : {0.5000001, 1.0, 1e9})
    for (int n = 0; n < 20000; ++n) {
      const FixedArgs c = make_fixed(1.0, 1 / tau, none);
      double g[19];
      for (int k = 0; k < 19; ++k) {
        const double lo = k == 18 ? 0x1p-4 : 0x1p-10, hi = k < 6 ? 0x1p-3 : k < 18 ? 0x1p-4 : 0x1p-1;
        h[k] = drand48() < 0.5 ? lo : std::nextafter(hi, 0.0);
      }
      if (!fixed_in_range(h, c)) return fail("corner refused", n, tau);
      R q[19];
      reference(h, 1 / tau, none, q);
      int64_t f[19];
      for (int k = 0; k < 19; ++k) f[k] = fixed_in(h[k], c);
      fixed_relax(f, fixed_sums(f), c, g);
      for (int k = 0; k < 19; ++k)
        if (std::fabs(R(g[k]) - q[k]) > 0x1p-52L) return fail("corner", g[k], double(q[k]));
    }
  // scales and forces it does not take
  const double big[3] = {0.02, 0, 0};
  if (make_fixed(1e300, 1.0, none).on || make_fixed(1e-300, 1.0, none).on || make_fixed(1.0, 1e-20, none).on ||
      make_fixed(1.0, 1.0, big).on)
    return fail("should be off", 0, 0);
  std::printf("ok\n");
  return 0;
}
"""


def test_fixed_point_relaxation_on_the_host(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "fixed.cpp", tmp_path / "fixed"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", cuda, "-I",
                        os.path.join(ROOT, "paper_0811_4593_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout + out.stderr
