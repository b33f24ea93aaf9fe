"""Operator rows in split BF16 (csrc/split_bf16.hpp), compiled into a small host program: a row
rounded for smooth data holds the nearest value of every entry or the next one past it, and
its sums over the modes are far closer to the exact ones than with every low part to nearest.

The bound: the choices of n entries between two neighbours lie 2^n to a box, so that in m modes
the nearest of them to the exact sums is about 2^(-n/m) of the box away, the distance of the
nearest rows being of the order of the box. With m = 5 and n the nodes but node 0 (where every
mode vanishes), and twice that for a search that is not exhaustive: 0.57, 0.29 and 0.125 of
the nearest rows' rms at N = 3, 4 and 5.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1403_1661_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "split_bf16.hpp"
using namespace swe;
#define CHECK(x) do { if (!(x)) { std::printf("failed at line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
int main(int argc, char** argv) {
  const int N = std::atoi(argv[1]);
  std::mt19937 rng(11);
  std::normal_distribution<double> u;
  double near2 = 0.0, smooth2 = 0.0;
  for (int rep = 0; rep < 400; ++rep) {
    std::vector<std::vector<double>> modes(5);
    std::vector<double> w;
    for (int j = 0; j <= N; ++j)
      for (int i = 0; i <= N - j; ++i) {
        const double x = 2.0 * i / N, y = 2.0 * j / N;
        const double f[5] = {x, y, 0.1 * x * x, 0.1 * x * y, 0.1 * y * y};
        for (int q = 0; q < 5; ++q) modes[q].push_back(f[q]);
        w.push_back(rep % 7 == 0 && i == j ? 0.0 : u(rng) * (i % 2 ? -1.0 : 1.0));
      }
    const int n = (int)w.size();
    const std::vector<double> r = smooth_row(w.data(), n, modes);
    double a[5] = {}, b[5] = {};
    for (int j = 0; j < n; ++j) {
      uint16_t h, l, h2, l2;
      bf16_split(w[j], h, l);
      bf16_split(r[j], h2, l2);
      const double nearest = (double)bf16_value(h) + bf16_value(l);
      CHECK((double)bf16_value(h2) + bf16_value(l2) == r[j]);             // representable
      CHECK(w[j] != 0.0 || r[j] == 0.0);
      CHECK(r[j] == nearest || (r[j] - w[j]) * (nearest - w[j]) <= 0.0);    // else on the entry's other side
      for (int q = 0; q < 5; ++q) {
        a[q] += (nearest - w[j]) * modes[q][j];
        b[q] += (r[j] - w[j]) * modes[q][j];
      }
    }
    for (int q = 0; q < 5; ++q) {
      near2 += a[q] * a[q];
      smooth2 += b[q] * b[q];
    }
  }
  std::printf("rms of the sums: nearest %.3g, smooth %.3g\n", std::sqrt(near2), std::sqrt(smooth2));
  const int n = (N + 1) * (N + 2) / 2 - 1;
  CHECK(std::sqrt(smooth2 / near2) <= 2.0 * std::exp2(-n / 5.0));
}
"""


@pytest.mark.parametrize("N", [3, 4, 5])
def test_rows_are_rounded_for_smooth_data(N, tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", f"-I{CSRC}", str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t"), str(N)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
