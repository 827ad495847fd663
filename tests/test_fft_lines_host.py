"""The plan of the FFT passes' line transforms (csrc/fft_lines.h), compiled on the host: factors
multiply to L and divide the values per thread, and the exchanges' index arithmetic with the
twiddle table of either direction gives the DFT (FP64, every length, both value widths, forward
with the upper half zero and inverse with the upper half dropped)."""

import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1408_4495_gb300", "csrc")
LENGTHS = [16, 32, 48, 64, 96, 128, 256, 512, 1024, 2048, 4096]

# a line through its factors with every butterfly a plain DFT: value (k1, i) of the first exchange
# at k1 * (L / R1) + i, the second exchange in place, as in line_fft
PROG = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "fft_lines.h"
using cd = std::complex<double>;
using namespace ls;
static void dft(std::vector<cd>& v, int S) {
  const int R = v.size();
  std::vector<cd> w(R);
  for (int k = 0; k < R; ++k)
    for (int i = 0; i < R; ++i) w[k] += v[i] * std::polar(1.0, S * 2 * M_PI * ((k * i) % R) / R);
  v = w;
}
static std::vector<cd> table(int L, bool wide) {
  std::vector<cd> tw(line_tw_size(L, wide));
  for (int inv = 0; inv < 2; ++inv) {
    size_t t = inv ? line_tw_dir(L, wide, false) : 0;
    int N = L;
    for (int p = 0; line_radix(L, wide, inv, p + 1) > 1; ++p) {
      const int R = line_radix(L, wide, inv, p), J = N / R;
      for (int k = 0; k < R; ++k)
        for (int j = 0; j < J; ++j) tw.at(t + k * J + j) = std::polar(1.0, (inv ? 2 : -2) * M_PI * k * j / N);
      t += N;
      N = J;
    }
    if (t != (size_t)(inv ? line_tw_size(L, wide) : line_tw_dir(L, wide, false))) std::exit(3);
  }
  return tw;
}
static std::vector<cd> line(std::vector<cd> x, int L, bool wide, bool inv, const std::vector<cd>& tw) {
  const int S = inv ? 1 : -1, R1 = line_radix(L, wide, inv, 0), R2 = line_radix(L, wide, inv, 1), R3 = line_radix(L, wide, inv, 2);
  const int J1 = L / R1;
  const cd* t1 = tw.data() + (inv ? line_tw_dir(L, wide, false) : 0);
  std::vector<cd> s(L), y(L);
  for (int j = 0; j < J1; ++j) {
    std::vector<cd> v(R1);
    for (int r = 0; r < R1; ++r) v[r] = x[j + r * J1];
    dft(v, S);
    for (int k = 0; k < R1; ++k) s[k * J1 + j] = v[k] * t1[k * J1 + j];
  }
  for (int u = 0; u < L / R2; ++u) {
    const int k1 = u % R1, i3 = u / R1, o = k1 * J1 + i3;
    std::vector<cd> v(R2);
    for (int r = 0; r < R2; ++r) v[r] = s[o + r * R3];
    dft(v, S);
    for (int k = 0; k < R2; ++k) {
      if (R3 == 1) y[u + k * R1] = v[k];
      else s[o + k * R3] = v[k] * t1[L + k * R3 + i3];
    }
  }
  if (R3 > 1)
    for (int u = 0; u < L / R3; ++u) {
      std::vector<cd> v(R3);
      for (int r = 0; r < R3; ++r) v[r] = s[(u % R1) * J1 + (u / R1) * R3 + r];
      dft(v, S);
      for (int k = 0; k < R3; ++k) y[u + k * (L / R3)] = v[k];
    }
  return y;
}
int main() {
  for (int L; std::scanf("%d", &L) == 1;)
    for (int wide = 0; wide < 2; ++wide) {
      const LinePlan p = line_plan(L, wide);
      int prod = 1;
      bool div = p.nf >= 2 && L % p.e == 0;
      for (int q = 0; q < p.nf; ++q) { prod *= p.r[q]; div = div && p.e % p.r[q] == 0; }
      const std::vector<cd> tw = table(L, wide);
      double worst = 0;
      for (int inv = 0; inv < 2; ++inv) {
        std::vector<cd> x(L);
        for (int i = 0; i < L; ++i) x[i] = inv || i < L / 2 ? cd(std::sin(1.7 * i + 0.3), std::cos(0.9 * i * i)) : cd(0);
        const std::vector<cd> y = line(x, L, wide, inv, tw);
        double nx = 0;
        for (auto& v : x) nx += std::norm(v);
        for (int k = 0; k < (inv ? L / 2 : L); k += L > 512 ? 37 : 1) {
          cd s = 0;
          for (int i = 0; i < L; ++i) s += x[i] * std::polar(1.0, (inv ? 2 : -2) * M_PI * (double)((long)k * i % L) / L);
          worst = std::fmax(worst, std::abs(s - y[k]) / std::sqrt(nx));
        }
      }
      std::printf("%d %d %d %d %.3e\n", L, wide, prod, (int)div, worst);
    }
}
"""


def test_line_plans_transform(tmp_path):
    cxx = shutil.which(os.environ.get("CXX", "g++"))
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, input=" ".join(map(str, LENGTHS))).stdout
    rows = [line.split() for line in out.splitlines()]
    assert [(int(r[0]), int(r[1])) for r in rows] == [(L, w) for L in LENGTHS for w in (0, 1)]
    for L, _, prod, div, err in rows:
        assert prod == L and div == "1"
        # rounding of two sums of at most L terms of size |x| / sqrt(L) each
        assert float(err) < 1e-15 * np.sqrt(float(L)) * 8
