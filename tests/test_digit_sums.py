"""A sliced product's operator is refused on the host if the digit sums that carry a
result could leave the integers that FP32 holds exactly, whatever the data."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1801_00246_gb300")
# A row of n entries between 1/2 and 3/4: its exponent is that of its absolute sum less 6,
# 2 for 205 <= n <= 409, so leading digits average 40 and the others 64. Sum s is below
# 64 n (257 + 128 (s - 1)) + 128 40 n for s >= 1: at n = 400 sum 3 reaches 0.91 and sum 4
# 1.10 times 2^24, at n = 300 sum 4 0.82.
SOURCE = r"""
#include <cstdio>
#include "dg_internal.h"
int main(int, char** v) {
  const int n = std::stoi(v[1]);
  std::vector<double> A(n);
  unsigned long long s = 1;
  for (double& a : A) a = 0.5 + double((s = s * 6364136223846793005ull + 1442695040888963407ull) >> 11) * 0x1p-55;
  dgx::Tc64Op op;
  const cudaError_t e = dgx::tc64_op_create(A, 1, n, &op);
  std::printf("%d\n", e == cudaErrorInvalidValue);
  dgx::tc64_op_free(&op);
}
"""


def test_rows_too_long_for_exact_sums_are_refused(tmp_path):
    from paper_1801_00246_gb300 import build
    lib = build.build()
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    libs = [d for d in (os.path.join(cuda, "lib64"), os.path.join(cuda, "targets", "sbsa-linux", "lib")) if os.path.isdir(d)]
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + os.path.join(cuda, "include"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(PKG, "csrc"), str(src), lib, "-o", str(exe)] + ["-L" + d for d in libs] +
                   ["-lcudart", "-Wl,-rpath," + os.path.dirname(lib)] + ["-Wl,-rpath," + d for d in libs], check=True)
    refused = lambda n: subprocess.run([str(exe), str(n)], check=True, capture_output=True, text=True).stdout.strip()  # noqa: E731
    assert refused(300) == "0"
    assert refused(400) == "1"
