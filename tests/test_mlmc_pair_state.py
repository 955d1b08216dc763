"""The word that the multilevel kernel keeps of a pair (mlmc_pair.cuh), compiled
for the host: steps and flags come back whole up to the largest step cap."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1705_03666_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "mlmc_pair.cuh"
int main() {
  const int units[] = {3, 4, 5, 7, 15, 16};
  long bad = 0, n = 0;
  for (int unit : units) {
    const long long last = (2147483647LL - 1) / unit * unit;  // the last unit start below the cap
    const long long at[] = {0, unit, 1 << 20, (1 << 30) - 1, 1 << 30, (1LL << 30) + unit, 3LL << 29, last};
    for (long long k : at) {
      const int steps = static_cast<int>(k / unit * unit);
      for (int f = 0; f < 2; ++f)
        for (int c = 0; c < 2; ++c, ++n) {
          const pdd::PairState p = pdd::pair_unpack(pdd::pair_pack(steps, unit, f, c), unit);
          bad += p.steps != steps || p.fine_done != (f != 0) || p.coarse_done != (c != 0);
        }
    }
  }
  std::printf("%ld of %ld\n", bad, n);
  return bad != 0;
}
"""


def test_steps_and_flags(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "pair.cu", tmp_path / "pair"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
