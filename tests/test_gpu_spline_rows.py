"""Second derivatives of the interface spline (spline_kernel: cyclic reduction and
one refinement) against the rows' own solution in extended precision and against
the plain Thomas algorithm in one thread: on even knots, gaps of 3:1, and end gaps
far longer and far shorter than the rest.  And a value that is no number, anywhere,
reaches every row."""
import numpy as np
import pytest
import torch

from tests import device_harness

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "stencil.cu"
namespace pdd {  // (not called here)
size_t dst_scratch_bytes(int, int) { return 0; }
pdd_status dst_solve(pdd_ctx *, double *, int, int, double, double, char *, int64_t *, double *) { return PDD_OK; }
pdd_status subdomain_solve3d_impl(pdd_ctx *, const pdd_subdomain *, const double *, int64_t, double *,
                                  int64_t *, double *) { return PDD_OK; }
}
using namespace pdd;
__global__ void plain(const double *s, const double *y, int K, double *M, double *work) {
  double *a = work, *b = a + K + 1, *c = b + K + 1, *d = c + K + 1;
  const double h0 = s[1] - s[0], h1 = s[2] - s[1], hl = s[K] - s[K - 1], hm = s[K - 1] - s[K - 2];
  for (int i = 1; i < K; ++i) {
    const double g0 = s[i] - s[i - 1], g1 = s[i + 1] - s[i];
    a[i] = g0;
    b[i] = 2.0 * (g0 + g1);
    c[i] = g1;
    d[i] = 6.0 * ((y[i + 1] - y[i]) / g1 - (y[i] - y[i - 1]) / g0);
  }
  b[1] += a[1] * (h0 + h1) / h1;
  c[1] -= a[1] * h0 / h1;
  a[1] = 0.0;
  b[K - 1] += c[K - 1] * (hm + hl) / hm;
  a[K - 1] -= c[K - 1] * hl / hm;
  c[K - 1] = 0.0;
  for (int i = 2; i < K; ++i) {
    const double w = a[i] / b[i - 1];
    b[i] = b[i] - w * c[i - 1];
    d[i] = d[i] - w * d[i - 1];
  }
  M[K - 1] = d[K - 1] / b[K - 1];
  for (int i = K - 2; i >= 1; --i) M[i] = (d[i] - c[i] * M[i + 1]) / b[i];
  M[0] = ((h0 + h1) * M[1] - h0 * M[2]) / h1;
  M[K] = ((hm + hl) * M[K - 1] - hl * M[K - 2]) / hm;
}
extern "C" int run(const double *node_s, const double *vals, int K, double *s, double *y, double *M,
                   double *ref, double *work) {
  spline_kernel<<<1, std::min(1024, (K + 31) / 32 * 32)>>>(node_s, vals, 0.0, 1.0, 0.5, 1, s, y, K,
                                                                  M, work);
  plain<<<1, 1>>>(s, y, K, ref, work);
  return cudaDeviceSynchronize();
}
extern "C" int words() { return kSplineWork; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return device_harness.load(str(tmp_path_factory.mktemp("spline")), SOURCE)


def _run(lib, s, v):
    K = len(s) + 1
    out = [torch.zeros(K + 1, dtype=torch.float64, device="cuda") for _ in range(4)]
    work = torch.zeros(max(lib.words(), 4) * (K + 1), dtype=torch.float64, device="cuda")
    device_harness.call(lib.run, torch.from_numpy(s).cuda(), torch.from_numpy(v).cuda(), K, *out, work)
    return [t.cpu().numpy() for t in out]


def _knots(m, gaps, rng):
    g = np.ones(m + 1)
    if gaps == "3:1":
        g = rng.uniform(1, 3, m + 1)
    elif gaps != "even":
        g[0] = g[-1] = float(gaps)
    return np.cumsum(g)[:-1] / g.sum()


def _exact(s, y):
    """The rows as the kernel forms them, in double; their solution in extended
    precision (the plain algorithm: 2^-64 or better, times the rows' condition)."""
    K = len(s) - 1
    h = s[1:] - s[:-1]
    a, b, c, d = np.zeros((4, K + 1))
    a[1:K], b[1:K], c[1:K] = h[:-1], 2.0 * (h[:-1] + h[1:]), h[1:]
    d[1:K] = 6.0 * ((y[2:] - y[1:-1]) / h[1:] - (y[1:-1] - y[:-2]) / h[:-1])
    h0, h1, hl, hm = h[0], h[1], h[-1], h[-2]
    a1, ck = a[1], c[K - 1]
    b[1] += a1 * (h0 + h1) / h1
    c[1] -= a1 * h0 / h1
    b[K - 1] += ck * (hm + hl) / hm
    a[K - 1] -= ck * hl / hm
    a, b, c, d = (v.astype(np.longdouble) for v in (a, b, c, d))
    for i in range(2, K):
        w = a[i] / b[i - 1]
        b[i] -= w * c[i - 1]
        d[i] -= w * d[i - 1]
    M = np.zeros(K + 1, dtype=np.longdouble)
    M[K - 1] = d[K - 1] / b[K - 1]
    for i in range(K - 2, 0, -1):
        M[i] = (d[i] - c[i] * M[i + 1]) / b[i]
    return M[1:K]


@pytest.mark.parametrize("gaps", ["even", "3:1", "100", "0.01", "1e6"])
@pytest.mark.parametrize("m", [2, 3, 4, 16, 31, 32, 33, 63, 100, 128, 129, 1000, 1023, 1024, 3000])
def test_rows(lib, m, gaps):
    rng = np.random.default_rng(m)
    s = _knots(m, gaps, rng)
    v = np.exp(0.5) * np.cos(s) + 1e-3 * rng.standard_normal(m)
    sk, y, M, plain = _run(lib, s, v)
    want = _exact(sk, y)
    top = float(np.abs(want).max())
    err = np.abs(M[1:-1] - want).astype(float)
    err_plain = float(np.abs(plain[1:-1] - want).max())
    print(f"{m} nodes, gaps {gaps}: {err.max() / top:.2e} of the largest, plain {err_plain / top:.2e}")
    if gaps in ("even", "3:1"):
        # M's own rounding; the reduction's error, at most 100 u of the largest (4 a
        # round, twice the dominance), to the binary32 solution's 2^-17
        assert np.all(err <= 2.0 ** -53 * np.abs(want).astype(float) * 1.01 + 2.0 ** -63 * top)
    assert err.max() <= max(err_plain, 2.0 ** -53 * top)


@pytest.mark.parametrize("m", [3, 48, 200, 2000])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_no_number_reaches_every_row(lib, m, value):
    rng = np.random.default_rng(m)
    s = _knots(m, "3:1", rng)
    for at in (0, m // 2, m - 1):
        v = np.cos(s)
        v[at] = value
        _, _, M, plain = _run(lib, s, v)
        assert not np.isfinite(M).any() and not np.isfinite(plain).any()
