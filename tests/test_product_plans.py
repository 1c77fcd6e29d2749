"""Plans of the exact products of two matrices' columns, kept per shape on a host thread: every pair of column
counts is told apart, and pairs beyond 256 columns are refused whatever was planned before.  Host code only: a
small program over the library's own header, compiled here."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "xgram.cuh"
int main(int argc, char** argv) {
  double a = 0.0, b = 0.0;
  for (int i = 1; i + 1 < argc; i += 2) {
    const ttk::XgPair<double> p{&a, &b, std::atoi(argv[i]), std::atoi(argv[i + 1])};
    std::printf("%d ", ttk::xg_cross_fits(p) ? ttk::xg_cross_plan(p)->nraw : 0);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    from paper_2602_00290_gb300 import _build
    lib = _build.build()
    d = tmp_path_factory.mktemp("plans")
    src, exe = d / "plans.cu", d / "plans"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc] + _build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", _build.CSRC, "-I",
                       os.path.join(ROOT, "include"), str(src), "-o", str(exe), lib, "-Xlinker",
                       "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


def plans(program, pairs):
    out = subprocess.run([program] + [str(v) for p in pairs for v in p], capture_output=True, text=True, check=True)
    return [int(v) for v in out.stdout.split()]


@pytest.mark.parametrize("pairs", [
    [(2, 5), (1, 1005)], [(1, 1005), (2, 5)], [(3, 256), (2, 1256)], [(1, 1256), (2, 256)], [(256, 256), (255, 1256)],
    [(257, 3), (3, 257)], [(5, 2), (2, 5), (256, 1), (1, 256)],
])
def test_pairs_are_told_apart(program, pairs):
    # as in a process that plans nothing else: the columns of both (0: no plan)
    alone = [plans(program, [p])[0] for p in pairs]
    assert plans(program, pairs) == alone
    assert all(n in (0, a + b) for n, (a, b) in zip(alone, pairs))
    assert all(n == 0 for n, (a, b) in zip(alone, pairs) if max(a, b) > 256)
    assert all(n > 0 for n, (a, b) in zip(alone, pairs) if max(a, b) <= 64)
