"""The face closures of FP64 nodes in fixed point (csrc/fixed_close.cuh), compiled for the host
with a trap on signed overflow: against the closure in extended precision, and at the ends of
the windows, where a density that does not fit has to be noticed."""
import os
import shutil
import subprocess

import pytest

from test_fixed_point_host import ROOT

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <type_traits>
#include "fixed64.cuh"
#include "d3q19.cuh"
namespace lbm {
template <int K, int N, typename F>
void static_for(F&& f) {
  if constexpr (K < N) {
    f(std::integral_constant<int, K>{});
    static_for<K + 1, N>(f);
  }
}
}
#include "face.cuh"
using namespace lbm;
typedef long double R;

// closure of the plane with inward normal sg e_a, known populations f (S 2^-64) and the
// prescribed values r as the face's record holds them (rounded from doubles when it is made)
static R reference(int a, int sg, const int64_t* f, const int64_t* r, bool pressure, R* out) {
  R u[3], rho = R(r[2]), sum = 0;
  for (int t = 0, n = 0; t < 3; ++t)
    if (t != a) u[t] = R(r[n++]) * 3 / 2 / 0x1p62L;
  for (int k = 0; k < 19; ++k) {
    out[k] = R(f[k]);
    if (sg * ca(k, a) <= 0) sum += (ca(k, a) ? 2 : 1) * R(f[k]);
  }
  if (pressure) u[a] = sg * (1 - sum / rho);
  else rho = sum * (1 + R(r[2]) / 0x1p62L), u[a] = sg * (1 - sum / rho);
  for (int k = 0; k < 19; ++k) {
    if (sg * ca(k, a) <= 0) continue;
    R cu = 0, tn = 0;
    for (int t = 0; t < 3; ++t) {
      cu += ca(k, t) * u[t];
      if (t == a || !ca(k, t)) continue;
      R in_plane = 0;
      for (int i = 0; i < 19; ++i)
        if (ca(i, a) == 0) in_plane += ca(i, t) * R(f[i]);
      tn += ca(k, t) * (in_plane / 2 - rho * u[t] / 3);
    }
    out[k] = R(f[opp(k)]) + R(w36(k)) / 6 * rho * cu - tn;
  }
  return rho;
}

static int fail(const char* what, double a, double b) { std::printf("%s: %g %g\n", what, a, b); return 1; }

template <int A, int SG>
int face(const FixedArgs& fx) {
  auto rnd = [] { return 2 * drand48() - 1; };
  long wide = 0;
  for (int n = 0; n < 40000; ++n) {
    int64_t f[19], g[19];
    const int shape = n % 4;  // near rest, anywhere in the windows, at their ends, at their upper ends
    for (int k = 0; k < 19; ++k) {
      const int lo = k == 18 ? 58 : 52, hi = k < 6 ? 59 : k < 18 ? 58 : 61;
      const int64_t top = (int64_t(1) << hi) - 1;
      if (shape == 0) f[k] = int64_t(w36(k) / 36.0 / fx.unit_in * (1 + 0.1 * rnd()));
      else if (shape == 1) f[k] = int64_t(std::exp2(lo + (hi - lo) * drand48()));
      else f[k] = shape == 2 && drand48() < 0.5 ? int64_t(1) << lo : top;
      g[k] = f[k];
    }
    const bool pressure = n % 3 == 0;
    double u[3] = {0.2499 * rnd(), 0.2499 * rnd(), 0.2499 * rnd()};
    if (n % 5 == 0) u[A] = (rnd() < 0 ? -1 : 1) * 0.2499999;
    const double rho_p = std::exp2(-1.9 + 2.8 * drand48());
    int64_t r[4];
    if (pressure) u[A] = 0;
    make_fixed_face(fx, A, u, SG * u[A], pressure, rho_p, r);
    if (!r[3]) return fail("refused", u[A], rho_p);
    const bool fits = fixed_close_face<A, SG>(g, FixedFace{{r[0], r[1]}, r[2], true}, pressure);
    R want[19];
    const R rho = reference(A, SG, f, r, pressure, want);
    if (fits != (rho < R(0x1p63L))) return fail("fits", fits, double(rho));
    wide += !fits;
    // units of S 2^-64, errors of the rounded products: d 2 (and 1 for its factor), d / 3 1 more,
    // rho u_t three times 1 and 1 for its factor, halves; below 8
    for (int k = 0; fits && k < 19; ++k)
      if (std::fabs(R(g[k]) - want[k]) > 8) return fail("error", k, double(R(g[k]) - want[k]));
  }
  return wide ? 0 : fail("no density beyond the range", A, SG);
}

int main() {
  const double none[3] = {0, 0, 0};
  const FixedArgs fx = make_fixed(1.0, 1.25, none);
  if (face<0, 1>(fx) || face<0, -1>(fx) || face<1, 1>(fx) || face<1, -1>(fx) || face<2, 1>(fx) || face<2, -1>(fx)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def test_face_closures_in_fixed_point(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    csrc = os.path.join(ROOT, "paper_0811_4593_gb300", "csrc")
    with open(os.path.join(csrc, "fixed_close.cuh"), encoding="utf-8") as fh:
        text = fh.read()
    # the faces, without the rules that need the sweep's own headers
    (tmp_path / "face.cuh").write_text(text[:text.index("// As close_edge and close_corner")] + "}\n")
    src, exe = tmp_path / "faces.cpp", tmp_path / "faces"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fsanitize=signed-integer-overflow",
                        "-fsanitize-undefined-trap-on-error", "-I", cuda, "-I", csrc, "-I", str(tmp_path), str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout == "ok\n", (out.returncode, out.stdout, out.stderr)
