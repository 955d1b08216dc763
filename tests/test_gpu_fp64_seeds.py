"""FP64 square roots and quotients from hardware seeds (sqrt_r2, rcp_seed with
seeded_div, and the back substitution's quotient from a reciprocal) over exponents
and random mantissas, against extended precision: half a unit in the last place and
the little that the last correction leaves."""
import numpy as np
import pytest
import torch

from tests import device_harness

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "rbf.cu"
using namespace pdd;
__global__ void roots(const double *x, double *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = sqrt_r2(x[i]);
}
__global__ void quotients(const double *a, const double *b, double *q, double *p, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  q[i] = seeded_div(a[i], b[i], rcp_seed(b[i]));
  p[i] = back_quotient(a[i], b[i], 1.0 / b[i]);
}
extern "C" int root(const double *x, double *y, int n) {
  roots<<<(n + 255) / 256, 256>>>(x, y, n);
  return cudaDeviceSynchronize();
}
extern "C" int quotient(const double *a, const double *b, double *q, double *p, int n) {
  quotients<<<(n + 255) / 256, 256>>>(a, b, q, p, n);
  return cudaDeviceSynchronize();
}
"""
N = 1 << 21


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return device_harness.load(str(tmp_path_factory.mktemp("seeds")), SOURCE)


def _ulps(got, exact):
    """Error in units in the last place of the double nearest to exact."""
    e = np.abs(got.astype(np.longdouble) - exact)
    return float((e / np.spacing(np.abs(exact.astype(np.float64))).astype(np.longdouble)).max())


def _mantissas(rng):
    m = rng.uniform(1.0, 2.0, N)
    edge = np.concatenate([1.0 + np.arange(64) * 2.0 ** -52, 2.0 - np.arange(1, 65) * 2.0 ** -52,
                           1.0 + np.arange(1, 1024) / 1024])
    m[:len(edge)] = edge
    return m


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="no extended precision")
@pytest.mark.parametrize("exponents", [(-2, 2), (-30, 2), (-99, 99)])
def test_square_root(lib, exponents):
    rng = np.random.default_rng(exponents[1] - exponents[0])
    x = np.ldexp(_mantissas(rng), rng.integers(*exponents, N))
    x[0] = 0.0
    y = torch.empty(N, dtype=torch.float64, device="cuda")
    device_harness.call(lib.root, torch.from_numpy(x).cuda(), y, N)
    y = y.cpu().numpy()
    assert y[0] == 0.0
    worst = _ulps(y[1:], np.sqrt(x[1:].astype(np.longdouble)))
    print(f"square root, exponents {exponents}: {worst:.4f} ulp")
    assert worst <= 0.5 + 2.0 ** -5        # below 2^-58 before the rounding


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="no extended precision")
@pytest.mark.parametrize("exponents", [(-2, 2), (-200, 200)])
def test_quotient(lib, exponents):
    """|a| <= |b|, as the multipliers of a pivoted column are, and any a for the back
    substitution."""
    rng = np.random.default_rng(exponents[1])
    b = np.ldexp(_mantissas(rng), rng.integers(*exponents, N)) * rng.choice([-1.0, 1.0], N)
    a = b * rng.uniform(-1, 1, N) * rng.choice([1.0, 1.0, 2.0 ** -20, 2.0 ** -50], N)
    a[:4] = [0.0, b[1], -b[2], b[3] / 2]
    q, p = (torch.empty(N, dtype=torch.float64, device="cuda") for _ in range(2))
    device_harness.call(lib.quotient, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), q, p, N)
    exact = a.astype(np.longdouble) / b.astype(np.longdouble)
    for name, v in (("multiplier", q), ("back substitution", p)):
        v = v.cpu().numpy()
        assert v[0] == 0.0 and v[1] == 1.0 and v[2] == -1.0 and v[3] == 0.5
        worst = _ulps(v[1:], exact[1:])
        print(f"{name}, exponents {exponents}: {worst:.4f} ulp")
        assert worst <= 0.5 + 2.0 ** -6    # 2^-60 before the rounding
