"""The entries a step makes of a work item that is a run (32 consecutive cells without walls)
equal those its table holds, for every place of a run in rows of 32 to 199 cells, a row of
exactly one run among them: checked on the CPU by compiling the same header code for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_02960_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <cstdint>
#include "lbm_device.cuh"
using namespace lbm;
int main() {
  long long checked = 0, bad = 0;
  for (uint32_t nx = 32; nx < 200; ++nx)
    for (uint32_t c0 = 0; c0 < 3 * nx; ++c0)
      for (uint32_t inner = 0; inner < 2; ++inner) {
        const uint32_t z = c0 | 1u << 31 | inner << 30, w = run_faces(c0 % nx, nx);
        for (uint32_t lane = 0; lane < 32; ++lane) {
          const uint32_t c = c0 + lane, x = c % nx;
          const uint32_t e = c | (x == 0 ? 1u << 28 : 0u) | (x == nx - 1 ? 1u << 29 : 0u) | inner << 30;
          ++checked;
          if (run_entry(z, w, lane) != e) ++bad;
        }
      }
  printf("%lld %lld\n", checked, bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc")
def test_run_entries_are_those_of_the_table(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "run.cu"
    src.write_text(SRC)
    exe = tmp_path / "run"
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    checked, bad = map(int, out.stdout.split())
    assert checked > 1_000_000
    assert bad == 0 and out.returncode == 0
