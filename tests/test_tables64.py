"""The integer tables of the FP64 tensor-core apply (host code, no GPU): in exact
arithmetic every volume and jump column sums over the test functions to zero, every
flux column to one weight per face node for the three faces and both directions, and
no entry is further from the product in doubles than the rounding of either."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1801_00246_gb300", "csrc")
SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include "tables64.h"
using namespace dgx;
int main() {
  for (int N = 1; N <= kMaxN; ++N) {
    const RefElem R = build_reference(N);
    OutTable tables[2];
    build_out_tables(R, tables);
    for (int helm = 0; helm < 2; ++helm) {
      const OutTable& t = tables[helm];
      const int Np = R.Np, unit = *std::min_element(t.ea.begin(), t.ea.end());
      auto sum = [&](int k) {
        __int128 s = 0;
        for (int r = 0; r < Np; ++r) s += __int128(t.x[size_t(r) * t.cols + k]) << (t.ea[r] - unit);
        return s;
      };
      auto col = [&](int c, int g, int i) { return (g / 2 * 3 + c) * 16 + g % 2 * 8 + i; };
      int nonzero = 0, uneven = 0;
      for (int g = 0; g < t.gface; ++g)
        for (int i = 0; i < 8; ++i)
          for (int c = 0; c < (g < t.gvol ? 3 : 2); ++c) nonzero += sum(col(c, g, i)) != 0;
      auto weight = [&](int l) { return sum(col(2, t.gvol + l / 8, l % 8)); };
      for (int f = 0; f < 3; ++f)
        for (int j = 0; j <= N; ++j)
          uneven += weight(f * (N + 1) + j) != weight(j) || weight(j) != weight(N - j) || weight(j) <= 0;
      double off = 0.0, size = 0.0;
      for (int r = 0; r < Np; ++r)
        for (int n = 0; n < Np; ++n) {
          long double s[3] = {};
          for (int k = 0; k < Np; ++k) {
            const long double br = R.Br[size_t(r) * Np + k], bs = R.Bs[size_t(r) * Np + k];
            s[0] += br * R.Dr[size_t(k) * Np + n];
            s[1] += br * R.Ds[size_t(k) * Np + n] + bs * R.Dr[size_t(k) * Np + n];
            s[2] += bs * R.Ds[size_t(k) * Np + n];
          }
          for (int c = 0; c < 3; ++c) {
            const long double v = std::ldexp((long double)t.x[size_t(r) * t.cols + col(c, n / 8, n % 8)], t.ea[r] - 56);
            off = std::max(off, double(std::fabs(v - s[c])));
            size = std::max(size, double(std::fabs(s[c])));
          }
        }
      std::printf("%d %d %d %d %.3e\n", N, helm, nonzero, uneven, off / size);
    }
  }
}
"""


def test_columns_sum_to_what_the_basis_says(tmp_path):
    src, exe = tmp_path / "sums.cpp", tmp_path / "sums"
    src.write_text(SOURCE)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + cuda, "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, str(src),
                    os.path.join(CSRC, "tables64.cpp"), os.path.join(CSRC, "refelem.cpp"), "-o", str(exe)], check=True)
    lines = [ln.split() for ln in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(lines) == 20
    for N, helm, nonzero, uneven, off in lines:
        assert int(nonzero) == 0 and int(uneven) == 0, (N, helm)
        # the derivatives' row sums, taken out here, are below Np 2^-50; products of Np terms
        assert float(off) <= 66 * 2.0 ** -50, (N, helm)
