"""Mean and squared deviations of a node from its exact digit sums (fix_moments,
compiled for the host): each within half a unit in the last place of the exact
quotient, up to what the 63 leading bits of its numerator leave out."""
import os
import shutil
import subprocess
from fractions import Fraction
import math
import random
import struct

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1705_03666_gb300", "csrc")
SHIFT = 60

SOURCE = r"""
#include <cstdio>
#include "nodefix.cuh"
int main() {
  pdd::NodeFix F{};
  for (;;) {
    if (std::scanf("%lld", &F.n) != 1) return 0;
    for (auto *w : {F.s1, F.s2})
      for (int k = 0; k < 5; ++k)
        if (std::scanf("%lld", w + k) != 1) return 1;
    double m, m2;
    pdd::fix_moments(F, &m, &m2);
    std::printf("%a %a\n", m, m2);
  }
}
"""


def _digits(x):
    """x 2^60 truncated towards zero, as five digits of 24 bits with its sign."""
    v, sign = abs(x), -1 if x < 0 else 1
    t = int(v * (1 << SHIFT))
    return [sign * ((t >> (24 * k)) & 0xffffff) for k in range(5)]


def _sums(scores):
    s1, s2 = [0] * 5, [0] * 5
    for s in scores:
        f = Fraction(s)
        for k, d in enumerate(_digits(f)):
            s1[k] += d
        for k, d in enumerate(_digits(f * f)):
            s2[k] += d
    return s1, s2


def _ulp(x):
    return Fraction(math.ulp(float(x)))


def test_half_a_unit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "m.cu", tmp_path / "m"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    rng = random.Random(7)
    f32 = lambda v: struct.unpack("f", struct.pack("f", v))[0]
    cases = []
    for t in range(1500):
        n = rng.choice([1, 2, 3, 7, 50, 200])
        scale = 2.0 ** rng.randint(-20, 28)
        mid = rng.choice([0.0, 1.0, -3.0, 1000.0])
        s = [f32(mid + scale * rng.uniform(-1, 1)) for _ in range(n)]
        cases.append((n, *_sums(s)))
    for t in range(1500):   # large counts: any sums that scores could have
        n = rng.randint(2, 1 << 32)
        m = rng.uniform(-1000, 1000)
        s1 = [n * d + rng.randint(-n, n) // 2 for d in _digits(Fraction(m))]
        s2 = [n * abs(d) for d in _digits(Fraction(m) ** 2 * Fraction(rng.uniform(1.0000001, 3)))]
        cases.append((n, s1, s2))
    # numerators whose leading bits are all ones
    for n in (2, 3, 1 << 20):
        cases.append((n, [0, 0, 0, 0, 0], [(1 << 56) - 1] * 5))
        cases.append((n, [(1 << 24) * n - 1, n * 0xffffff, n * 0xffffff, 0, 0], [n] * 5))
    text = "\n".join(" ".join(map(str, [n, *s1, *s2])) for n, s1, s2 in cases)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
    worst = [0.0, 0.0]
    for (n, s1, s2), line in zip(cases, out.splitlines(), strict=True):
        mean, m2 = (Fraction(float.fromhex(v)) for v in line.split())
        S1 = Fraction(sum(d << (24 * k) for k, d in enumerate(s1)), 1 << SHIFT)
        S2 = Fraction(sum(d << (24 * k) for k, d in enumerate(s2)), 1 << SHIFT)
        em = S1 / n
        e2 = max(Fraction(0), S2 - S1 * S1 / n) if n > 1 else Fraction(0)
        for q, (got, exact) in enumerate(((mean, em), (m2, e2))):
            if exact == 0:
                assert got == 0
                continue
            worst[q] = max(worst[q], float(abs(got - exact) / _ulp(exact)))
    print(f"largest error: mean {worst[0]:.4f} ulp, M2 {worst[1]:.4f} ulp")
    # half an ulp, 2^-10 of one for the 63 bits, 2^-50 of one for the correction
    assert max(worst) <= 0.5 + 2.0 ** -9
