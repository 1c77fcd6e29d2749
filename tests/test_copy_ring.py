"""The copies of the exact products' ring of stages that may be in flight when a CTA ends: the phase of each
stage's mbarrier that its last copies complete, against a replay of the ring.  Host code only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "xgram.cuh"
int main() {
  for (int nst = 2; nst <= ttk::kXgMaxStage; ++nst)
    for (int issued = 0; issued <= 40; ++issued) {
      std::printf("%d %d", nst, issued);
      for (int u = ttk::xg_last_first(issued, nst); u < issued; ++u)
        std::printf(" %d:%u", u % nst, ttk::xg_fill_parity(u, nst));
      std::printf("\n");
    }
  return 0;
}
"""


def test_last_fill_of_every_stage(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    from paper_2602_00290_gb300 import _build
    lib = _build.build()
    src, exe = tmp_path / "ring.cu", tmp_path / "ring"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc] + _build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", _build.CSRC, "-I",
                       os.path.join(ROOT, "include"), str(src), "-o", str(exe), lib, "-Xlinker",
                       "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines():
        nst, issued, *fills = line.split()
        last = {}
        for tile in range(int(issued)):  # a stage's k-th fill completes its mbarrier's phase k
            stage = tile % int(nst)
            last[stage] = last.get(stage, -1) + 1
        assert dict(tuple(map(int, f.split(":"))) for f in fills) == {s: k & 1 for s, k in last.items()}
        assert len(fills) == len(last)
