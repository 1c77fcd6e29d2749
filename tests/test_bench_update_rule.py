"""bench.py's account of the update pass (which kernel, how many digit products) follows the library's own rule:
the header's update_dig_fits and ud_orders over ranks and rows.  Host code only."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

PROGRAM = r"""
#include <cstdio>
#include "bigpass.cuh"
#include "update_dig.cuh"
template <typename T>
void show(const char* name, long rows, int r) {
  ttk::SrcStencil<T> s{};
  s.rcap = s.ldz = r;
  s.nterm = 4;
  s.nax = 2;
  const ttk::LivePattern lp{nullptr, r, 5, 0};
  const int ns = sizeof(T) == 4 ? 4 : 8, no = ttk::ud_orders(ns, ttk::ud_kp(r));
  int n = 0;
  for (int i = 0; i < ns; ++i)
    for (int j = 0; j < ns; ++j) n += i + j < no;
  std::printf("%s %ld %d %d\n", name, rows, r, ttk::update_dig_fits<T>(s, lp, rows, r) ? n : 0);
}
int main() {
  for (long rows : {256L, 1023L, 1024L, 100000L, 1L << 30, 1L << 31})
    for (int r = 1; r <= 80; ++r) {
      show<double>("fp64", rows, r);
      show<float>("mixed", rows, r);
    }
  return 0;
}
"""


def test_digit_products_follow_the_library(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    from paper_2602_00290_gb300 import _build
    lib = _build.build()
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc] + _build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", _build.CSRC, "-I",
                       os.path.join(ROOT, "include"), str(src), "-o", str(exe), lib, "-Xlinker",
                       "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lines = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(lines) == 960
    for line in lines:
        prec, rows, rank, n = line.split()
        assert (bench.update_digit_products(prec, int(rows), int(rank)) or 0) == int(n), line
    # where the precision asks for the split-TF32 kernel, it keeps the small passes of its ranks
    assert bench.update_digit_products("mixed_3xtf32", 4095, 32) is None
    assert bench.update_digit_products("mixed_3xtf32", 4096, 32) == bench.update_digit_products("mixed", 4096, 32)
    assert bench.update_digit_products("mixed_3xtf32", 4095, 24) == 13
