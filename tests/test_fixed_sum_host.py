"""The conversion of the integer sums to FP64 (csrc/fixed_sum.cuh): totals of both signs, small
ones exactly and larger ones to FP64's rounding, against exact integers, on the CPU by compiling
the same header code for the host."""
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1508_02960_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "fixed_sum.cuh"
int main() {
  long long x; int terms;
  while (scanf("%lld %d", &x, &terms) == 2) {  // the sum of `terms` terms x
    lbm::FixedSum s{0, 0ull};
    for (int i = 0; i < terms; ++i) s.add(x);
    printf("%a\n", lbm::to_double(((__int128)s.hi << 32) + (__int128)s.lo));
  }
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc")
def test_totals_of_both_signs(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "fs.cu"
    src.write_text(SRC)
    exe = tmp_path / "fs"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rng = random.Random(4)
    cases = [(x, 1) for x in (0, 1, 1000, 2 ** 32 - 1, 2 ** 32, 2 ** 40 + 513, 2 ** 53 - 1, 2 ** 62 + 12345)]
    cases += [(rng.getrandbits(rng.randint(1, 62)), rng.randint(1, 500)) for _ in range(300)]
    cases += [(-x, n) for x, n in cases]
    out = subprocess.run([str(exe)], input="".join("%d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True)
    got = [float.fromhex(v) for v in out.stdout.split()]
    assert len(got) == len(cases)
    for (x, n), v in zip(cases, got):
        # one rounding of the low word and one of the sum
        assert abs(int(v) - x * n) <= 2.0 ** -52 * abs(x * n), (x, n, v)
        if abs(x * n) < 2 ** 53:
            assert int(v) == x * n
    half = len(got) // 2
    assert [-v for v in got[:half]] == got[half:]
