"""The mean gains that the resident, plane and line forms correct dtau for (reg_gain in
csrc/qf_fft_reg.cuh), computed again from the constants the kernels use.

The program restates each form's transform in double precision with the twiddles of the headers,
single precision as the kernels hold them, and takes the mean of the diagonal of inverse times
forward.  The table has two decimals of 1e-8: within 1e-10.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_10185_gb300", "csrc")
PROGRAM = r"""
#include <complex>
#include <cstdio>
#include <vector>
#include "qf_fft_reg.cuh"
using cd = std::complex<double>;
using V = std::vector<cd>;
static double f32(double x) { return (double)(float)x; }
// twiddle of the register forms, and a table's (rounded to nearest); forward
static cd tw(int k, int n, bool reg) {
  k %= n;
  const double c = qf::rc_cos(k, n), s = qf::rc_sin(k, n);
  if (4 * k % n == 0) return cd(std::round(c), -std::round(s));
  if (reg && 8 * k % n == 0) {
    const double h = 0.70710676908493042 + 1.2101617e-8;
    return cd(c > 0 ? h : -h, s > 0 ? -h : h);
  }
  if (!reg) return cd(f32(std::cos(2 * M_PI * k / n)), -f32(std::sin(2 * M_PI * k / n)));
  const qf::RcTwiddle t = qf::rc_twiddle(k, n);
  return cd(t.c, -t.s);
}
static V split(const V& x, int A, int B, bool reg, bool inv);
static V dft(const V& x, bool reg, bool inv) {
  const int n = (int)x.size();
  const cd i = inv ? cd(0, 1) : cd(0, -1);
  if (n == 1) return x;
  if (n == 2) return {x[0] + x[1], x[0] - x[1]};
  if (n == 3) {
    const double h = f32(0.86602540378443864676);
    const cd s = x[1] + x[2], d = x[1] - x[2], t = x[0] - 0.5 * s;
    return {x[0] + s, t + i * h * d, t - i * h * d};
  }
  if (n == 4) {
    const cd a0 = x[0] + x[2], a1 = x[0] - x[2], a2 = x[1] + x[3], d = x[1] - x[3];
    return {a0 + a2, a1 + i * d, a0 - a2, a1 - i * d};
  }
  const int A = n % 3 == 0 ? 3 : 4;
  return split(x, A, n / A, reg, inv);
}
static V split(const V& x, int A, int B, bool reg, bool inv) {
  const int n = A * B;
  std::vector<V> a(B);
  for (int n2 = 0; n2 < B; ++n2) {
    V u(A);
    for (int n1 = 0; n1 < A; ++n1) u[n1] = x[B * n1 + n2];
    a[n2] = dft(u, reg, inv);
  }
  V y(n);
  for (int k1 = 0; k1 < A; ++k1) {
    V z(B);
    for (int n2 = 0; n2 < B; ++n2) {
      const cd w = tw(n2 * k1, n, reg);
      z[n2] = a[n2][k1] * (inv ? std::conj(w) : w);
    }
    const V w = dft(z, reg, inv);
    for (int k2 = 0; k2 < B; ++k2) y[k1 + A * k2] = w[k2];
  }
  return y;
}
// the four-pass kernels' transform: twiddles of radix 8 and more are multiplied up from the table
static V stockham(V x, int n, int plan, bool inv) {
  for (int st = 0, ns = 1; st < qf::plan_stages(n, plan); ++st) {
    const int R = qf::plan_radix(n, st, plan);
    V y(n);
    for (int j = 0; j < n / R; ++j) {
      const int k = j % ns;
      V v(R);
      cd w1 = tw(k, ns * R, false), w = w1;
      for (int r = 0; r < R; ++r) {
        v[r] = x[j + r * n / R];
        if (r == 0 || ns == 1) continue;
        if (R < 8) w = tw(r * k, ns * R, false);
        else if (r == 8) w = tw(8 * k, ns * R, false);
        else if (r > 1) w = cd(f32((w * w1).real()), f32((w * w1).imag()));
        v[r] *= inv ? std::conj(w) : w;
      }
      const V o = dft(v, false, inv);
      for (int r = 0; r < R; ++r) y[(j / ns) * ns * R + k + r * ns] = o[r];
    }
    x = y;
    ns *= R;
  }
  return x;
}
template <typename F>
static double gain(int n, F f) {  // mean of diag(inverse o forward)/n - 1
  double g = 0;
  for (int e = 0; e < n; ++e) {
    V x(n);
    x[e] = 1;
    g += f(f(x, false), true)[e].real() / n - 1;
  }
  return g / n;
}
int main() {
  auto reg = [](int n) { return gain(n, [](const V& x, bool inv) { return dft(x, true, inv); }); };
  auto two = [](int n, int E) { return gain(n, [&](const V& x, bool inv) { return split(x, E, n / E, true, inv); }); };
  auto four = [](int n, int plan) { return gain(n, [&](const V& x, bool inv) { return stockham(x, n, plan, inv); }); };
  auto say = [](int n, int plan, double g) { printf("%d %d %.4e %.4e\n", n, plan, qf::reg_gain(n, plan), g); };
  for (int n : {8, 12, 16, 24}) say(n, 0, reg(n));
  for (int n : {32, 48, 64, 96}) say(n, 0, two(n, n / 4));
  say(192, 0, (2 * two(192, 24) + four(192, 0)) / 3);
  for (int plan : {0, 1}) say(512, plan, (two(512, 32) + 2 * four(512, plan)) / 3);
  return 0;
}
"""


def test_gains_are_those_of_the_constants(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "gain.cu", tmp_path / "gain"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    rows = [line.split() for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert [(int(n), int(plan)) for n, plan, _, _ in rows] == [(n, 0) for n in (8, 12, 16, 24, 32, 48, 64, 96, 192, 512)] + [(512, 1)]
    for n, plan, table, computed in rows:
        assert abs(float(table) - float(computed)) < 1e-10, (n, plan)
