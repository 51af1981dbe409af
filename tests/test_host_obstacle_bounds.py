"""The box around an obstacle that lets links skip it (`obstacle_bounds`, csrc/prrtc_launch.h), on the CPU: a
sphere that touches the obstacle by the kernels' own test (boxes in the coordinates of the rows as given,
cylinders with the axis as given) reaches the box with its radius times kReachSlack.  Boxes with rotations that
are exact, rounded to a few decimals, scaled and sheared; cylinders with axes off unit length; spheres.  For each,
the farthest touching sphere in many directions, by bisection in 64 bits."""
import os
import subprocess

import numpy as np
import pytest

from paper_2503_06757_gb300 import build as B

PROGRAM = r'''
#include <cstdio>
#include <random>
#include "prrtc_launch.h"
using namespace prrtc;

static std::mt19937 gen(1);
static double uni(double lo, double hi) { return lo + (hi - lo) * std::uniform_real_distribution<double>()(gen); }
static void unit(double* v) {
  std::normal_distribution<double> n;
  double s = 0;
  for (int a = 0; a < 3; ++a) s += (v[a] = n(gen)) * v[a];
  for (int a = 0; a < 3; ++a) v[a] /= std::sqrt(s);
}

// squared distance of the kernels' test at c + v
static double dist2(int kind, const float4* e, const double* v) {
  double d[3] = {0, 0, 0};
  if (kind == 2) {
    const double z = e[1].x * v[0] + e[1].y * v[1] + e[1].z * v[2], ax[3] = {e[1].x, e[1].y, e[1].z};
    double rho = 0;
    for (int a = 0; a < 3; ++a) rho += (v[a] - z * ax[a]) * (v[a] - z * ax[a]);
    d[0] = std::max(std::sqrt(rho) - e[0].w, 0.0);
    d[1] = std::max(std::fabs(z) - e[1].w, 0.0);
  } else if (kind == 3) {
    d[0] = std::max(std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) - e[0].w, 0.0);
  } else {
    const double h[3] = {e[1].x, e[1].y, e[1].z};
    for (int j = 0; j < 3; ++j) {
      const double l = kind == 0 ? v[j] : e[2 + j].x * v[0] + e[2 + j].y * v[1] + e[2 + j].z * v[2];
      d[j] = std::max(std::fabs(l) - h[j], 0.0);
    }
  }
  return d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
}

int main() {
  // form: 0 aligned box; turned box with rows 1 exact, 2 / 3 / 4 rounded to 2 / 3 / 4 decimals, 5 scaled, 6 sheared;
  // 7 cylinder, 8 cylinder with its axis off, 9 sphere
  for (int form = 0; form < 10; ++form) {
    int misses = 0, unbounded = 0;
    double slack = 0;
    for (int k = 0; k < 150; ++k) {
      float4 e[5];
      const double size = std::pow(10.0, uni(-2, 0.5));
      double h[3], c[3];
      for (int a = 0; a < 3; ++a) h[a] = size * uni(0.02, 1), c[a] = uni(-3, 3);
      int kind = form == 0 ? 0 : form < 7 ? 1 : form < 9 ? 2 : 3;
      e[0] = make_float4(c[0], c[1], c[2], h[0]);
      e[1] = make_float4(h[0], h[1], h[2], 0);
      if (kind == 1) {
        double u[3], v[3], w[3];
        unit(u);
        unit(v);
        const double uv = u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
        double s = 0;
        for (int a = 0; a < 3; ++a) s += (v[a] - uv * u[a]) * (v[a] - uv * u[a]);
        for (int a = 0; a < 3; ++a) v[a] = (v[a] - uv * u[a]) / std::sqrt(s);
        for (int a = 0; a < 3; ++a) w[a] = u[(a + 1) % 3] * v[(a + 2) % 3] - u[(a + 2) % 3] * v[(a + 1) % 3];
        double* rows[3] = {u, v, w};
        const double step = std::pow(10.0, -form), scale = form == 5 ? uni(0.99, 1.05) : 1.0;
        for (int j = 0; j < 3; ++j) {
          for (int a = 0; a < 3; ++a) {
            if (form >= 2 && form <= 4) rows[j][a] = std::round(rows[j][a] / step) * step;
            if (form == 5) rows[j][a] *= scale;
            if (form == 6) rows[j][a] += uni(-2e-3, 2e-3);
          }
          e[2 + j] = make_float4(rows[j][0], rows[j][1], rows[j][2], 0);
        }
      } else if (kind == 2) {
        double u[3];
        unit(u);
        const double len = form == 8 ? uni(0.9991, 1.0009) : 1.0;
        e[1] = make_float4(u[0] * len, u[1] * len, u[2] * len, h[1]);
      }
      float lo[3], hi[3];
      obstacle_bounds(kind, e, lo, hi);
      if (hi[0] > 1e30f) { ++unbounded; continue; }
      double exact[3] = {0, 0, 0};  // farthest a small sphere touches along +x, +y, +z
      for (int t = 0; t < 300; ++t) {
        double dir[3];
        const double r = std::pow(10.0, uni(-3, 0));
        if (t < 3) for (int a = 0; a < 3; ++a) dir[a] = a == t;
        else unit(dir);
        // the farthest point of a ray from inside
        double a0 = 0, a1 = 100;
        for (int i = 0; i < 80; ++i) {
          const double m = 0.5 * (a0 + a1), v[3] = {m * dir[0], m * dir[1], m * dir[2]};
          (dist2(kind, e, v) < r * r ? a0 : a1) = m;
        }
        double d2 = 0;
        for (int a = 0; a < 3; ++a) {
          const double p = c[a] + a0 * dir[a], d = std::max(std::max(lo[a] - p, p - hi[a]), 0.0);
          d2 += d * d;
          exact[a] = std::max(exact[a], a0 * dir[a] - r);
        }
        misses += d2 > r * kReachSlack * r * kReachSlack;
      }
      // beyond the margin of 1e-4 and 1e-5 of the coordinates
      for (int a = 0; a < 3; ++a)
        slack = std::max(slack, hi[a] - c[a] - exact[a] - 1e-4 - 1e-5 * (std::fabs(c[a]) + exact[a]));
    }
    printf("%d %d %d %.3g\n", form, misses, unbounded, slack);
  }
  return 0;
}
'''


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    d = tmp_path_factory.mktemp("bounds")
    src, exe = os.path.join(d, "bounds.cu"), os.path.join(d, "bounds")
    with open(src, "w") as f:
        f.write(PROGRAM)
    cmd = [B.nvcc()] + B.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", B.INCLUDE, src, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return np.array([[float(x) for x in line.split()] for line in out.splitlines()])


def test_touching_spheres_reach_the_box(forms):
    assert len(forms) == 10
    assert not forms[:, 1].any(), forms


def test_usual_obstacles_are_bounded(forms):
    for form in (0, 1, 4, 7, 8, 9):
        assert forms[form, 2] == 0, forms[form]
    assert forms[2, 2] > 0 and forms[5, 2] > 0  # rows far from orthonormal are not
    # the margin and the rounding of the corners (coordinates below 8) and of the radius' own 1e-10
    assert forms[0, 3] < 2e-6 and forms[9, 3] < 2e-6
