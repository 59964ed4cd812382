"""The kernels' undistortion (several radii in step, with a shortcut out of a two-value cycle) against the
plain safeguarded Newton loop, bit for bit, for every number of steps.  Host build of the kernels' own
source."""
import os
import shutil
import subprocess

import pytest

from paper_2412_12507_gb300 import build

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "ut3d_device.cuh"
using namespace ut3d;

// One radius, one step after the other, to the last of the steps.
static float plain(const DevCam &c, float rd, int steps) {
  const bool radial = c.model == UT_CAM_PINHOLE_RADIAL;
  float lo = 0.f, hi = radial ? fminf(c.theta_max, fmaxf(2.f * rd, 1.f)) : c.theta_max;
  if (radial)
    for (int it = 0; it < 40 && std::isinf(c.theta_max) && rd > hi * radial_scale(c, hi * hi); ++it) hi *= 2.f;
  float x = fminf(rd, hi);
  for (int it = 0; it < steps; ++it) {
    const float f = radial ? fmaf(x, radial_scale(c, x * x), -rd) : theta_d_poly(c, x) - rd;
    if (f == 0.f) break;
    if (f > 0.f) hi = x; else lo = x;
    float nx = x - f / (radial ? radial_prime(c, x * x) : theta_d_prime(c, x));
    if (!(nx >= lo && nx <= hi)) nx = 0.5f * (lo + hi);
    if (nx == x) break;
    x = nx;
  }
  return x;
}

static bool same(float a, float b) { return std::memcmp(&a, &b, 4) == 0; }

int main() {
  std::mt19937 gen(7);
  std::uniform_real_distribution<float> u(0.f, 1.f), s(-1.f, 1.f);
  long bad = 0, odd = 0, n = 0;
  for (int t = 0; t < 60000; ++t) {
    DevCam c;
    std::memset(&c, 0, sizeof(c));
    c.model = t & 1 ? UT_CAM_FISHEYE : UT_CAM_PINHOLE_RADIAL;
    const float a = t % 3 ? 0.05f : 0.4f;
    c.k1 = a * s(gen); c.k2 = a * s(gen); c.k3 = a * s(gen); c.k4 = a * s(gen);
    c.theta_max = t & 1 ? 0.2f + 1.4f * u(gen) : (t & 2 ? INFINITY : 0.3f + 3.f * u(gen));
    float rd[3] = {2.f * u(gen), t % 7 ? u(gen) : (t % 5 ? 0.f : 1e-30f), c.theta_max < 10.f ? c.theta_max : 30.f * u(gen)};
    for (int steps = 1; steps <= 17; ++steps) {
      const int k = steps == 17 ? 64 : steps;
      float x1[1], x2[2], x3[3], p[3];
      const bool one[1] = {true}, some[2] = {(t & 8) != 0, true}, all[3] = {true, true, true};
      for (int j = 0; j < 3; ++j) {
        p[j] = plain(c, rd[j], k);
        const float r1[1] = {rd[j]};
        undistort<1>(c, r1, one, k, x1);
        bad += !same(x1[0], p[j]);
        if (k < 64) odd += !same(plain(c, rd[j], k + 1), p[j]);
        ++n;
      }
      const float r2[2] = {rd[0], rd[1]};
      undistort<2>(c, r2, some, k, x2);
      bad += !same(x2[0], some[0] ? p[0] : 0.f) + !same(x2[1], p[1]);
      undistort<3>(c, rd, all, k, x3);
      for (int j = 0; j < 3; ++j) bad += !same(x3[j], p[j]);
    }
  }
  // a number of steps that is off by one would show: many results change with the last step
  std::printf("%ld of %ld differ; %ld change with one more step\n", bad, n, odd);
  return bad == 0 && odd > n / 20 ? 0 : 1;
}
"""


def test_shortcut_gives_the_plain_loops_bits(tmp_path):
    nv = build._nvcc()
    if not shutil.which(nv):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "undistort.cu", tmp_path / "undistort"
    src.write_text(PROGRAM)
    # no contraction of the host's products and sums: both forms round alike
    cmd = [nv, *build.ARCH, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-Xcompiler", "-ffp-contract=off",
           "-I", os.fspath(build.CSRC), os.fspath(src), "-o", os.fspath(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([os.fspath(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    print(r.stdout)
