"""How far the fixed-point relaxation of FP64 nodes (csrc/fixed64.cuh, compiled for the host)
is from extended precision, population by population and over a whole node, beside the same
formulas in double. Up to tau = 3 errors by rms are no larger than double's for any kind and
size of population that a node may have; at longer relaxation times for those of at least
2^-8 S (rho0 / 64 to rho0 / 32), and the others lose three bits at most."""
import os
import shutil
import subprocess

import pytest

from test_fixed_point_host import PROGRAM as RELAXATION
from test_fixed_point_host import ROOT

# the reference and the double form of the relaxation test, with another main
PROGRAM = RELAXATION[:RELAXATION.index("int main()")] + r"""
int main() {
  srand48(11);
  auto rnd = [] { return 2 * drand48() - 1; };
  const double none[3] = {0, 0, 0};
  for (double rho0 : {1.0, 0.51, 1.9, 5e10})
    for (double tau : {0.501, 0.6, 1.0, 2.0, 3.0, 10.0, 50.0, 1e3})
      for (int wide = 0; wide < 2; ++wide) {
        const FixedArgs fx = make_fixed(rho0, 1 / tau, none);
        if (!fx.on) return fail("off", rho0, tau);
        int e = 0;
        e = std::frexp(rho0, &e) == 0.5 ? e + 1 : e + 2;  // S = 2^e
        double own[3][24] = {}, ref[3][24] = {}, worst = 0, worst_double = 0, mass = 0, square = 0;
        long count[3][24] = {}, taken = 0;
        for (long n = 0; n < 30000; ++n) {
          double h[19], d[19], g[19];
          for (int k = 0; k < 19; ++k) h[k] = w36(k) / 36.0 * rho0 * (1 + 0.1 * rnd());
          // some populations anywhere in their windows
          for (int i = wide ? lrand48() % 4 : 0; i > 0; --i) {
            const int k = lrand48() % 19;
            const double lo = k == 18 ? -6 : -12, hi = k < 6 ? -5 : k < 18 ? -6 : -3;
            h[k] = std::ldexp(std::exp2(lo + (hi - lo) * drand48()), e);
          }
          if (!fixed_in_range(h, fx)) continue;
          R q[19];
          reference(h, 1 / tau, none, q);
          in_double(h, 1 / tau, none, d);
          int64_t f[19];
          for (int k = 0; k < 19; ++k) f[k] = fixed_in(h[k], fx);
          fixed_relax(f, fixed_sums(f), fx, g);
          ++taken;
          for (int k = 0; k < 19; ++k) {
            const double v = double(q[k]), eo = double(R(g[k]) - q[k]), ed = double(R(d[k]) - q[k]);
            worst = std::fmax(worst, std::fabs(eo) / rho0);
            worst_double = std::fmax(worst_double, std::fabs(ed) / rho0);
            mass += double((R(g[k]) - h[k]) / rho0);
            square += (eo / rho0) * (eo / rho0);
            int at = 0;
            std::frexp(v, &at);
            const int bin = e - at;  // v in [S 2^-(bin + 1), S 2^-bin)
            if (v <= 0 || bin < 0 || bin >= 24) continue;
            const int c = k < 6 ? 0 : k < 18 ? 1 : 2;
            ++count[c][bin];
            own[c][bin] += (eo / v) * (eo / v);
            ref[c][bin] += (ed / v) * (ed / v);
          }
        }
        if (taken < 20000) return fail("few nodes taken", taken, tau);
        for (int c = 0; c < 3; ++c)
          for (int b = 0; b < 24; ++b) {  // (the rms of 1,000 values is known to 2 %)
            const double most = tau <= 3.0 || b + 1 <= 8 ? 1.0 : 8.0;
            if (count[c][b] >= 1000 && own[c][b] > most * most * ref[c][b]) {
              std::printf("rho0 %g tau %g kind %d size 2^-%d S: ", rho0, tau, c, b);
              return fail("rms beside double", std::sqrt(own[c][b] / count[c][b]), std::sqrt(ref[c][b] / count[c][b]));
            }
          }
        if (worst > worst_double) return fail("error beside double", worst, worst_double);
        // the rest population's last place is 2^-53 rho0 at most (rms 2^-54.8), and 12 times two
        // roundings of a unit of S 2^-63 <= 2^-60 rho0 go into it (rms 2^-57.7); the others'
        // errors add less than a tenth: over the node's 19 populations below 2^-56.7
        if (square / taken / 19 > 0x1p-113) return fail("rms", std::sqrt(square / taken / 19), tau);
        // a unit of S 2^-63 for each population, and a tenth for the sample
        if (std::fabs(mass / taken) > 1.1 * 19 * 0x1p-60) return fail("mass drift", mass / taken, tau);
      }
  std::printf("ok\n");
  return 0;
}
"""


def test_errors_of_the_fixed_point_relaxation(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "errors.cpp", tmp_path / "errors"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", cuda, "-I",
                        os.path.join(ROOT, "paper_0811_4593_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout + out.stderr
