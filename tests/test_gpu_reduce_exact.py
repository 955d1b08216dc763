"""Per-node sums of scores of very different size (reduce_wave_kernel): threads'
sums that cancel each other many times over lose nothing to the merge of the
threads, in one block per node and in several."""
import ctypes
import math

import numpy as np
import pytest
import torch

from tests import device_harness

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "reduce.cuh"
using namespace pdd;
template <typename R, bool kNaN>
static int run(const void *s, uint64_t n_paths, int nodes, int parts, void *scratch, void *acc) {
  const ReduceParts rp = reduce_parts_at(static_cast<char *>(scratch), nodes, parts);
  reduce_wave_kernel<R, kNaN><<<nodes * parts, kReduceBlock>>>(
      static_cast<const R *>(s), 0, n_paths * nodes, n_paths, 0, static_cast<NodeAcc *>(acc), rp);
  return cudaDeviceSynchronize();
}
extern "C" int reduce(const void *s, uint64_t n_paths, int nodes, int parts, int fp64, int nan,
                      void *scratch, void *acc) {
  if (fp64) return nan ? run<double, true>(s, n_paths, nodes, parts, scratch, acc)
                       : run<double, false>(s, n_paths, nodes, parts, scratch, acc);
  return nan ? run<float, true>(s, n_paths, nodes, parts, scratch, acc)
             : run<float, false>(s, n_paths, nodes, parts, scratch, acc);
}
"""


@pytest.fixture(scope="module")
def reduce(tmp_path_factory):
    return device_harness.load(str(tmp_path_factory.mktemp("reduce")), SOURCE).reduce


def _run(reduce, scores, parts, nan):
    """(count, mean, M2) per node of scores [nodes][n]."""
    nodes, n = scores.shape
    s = torch.from_numpy(scores).cuda()
    scratch = torch.zeros(nodes * parts * 64 + nodes * 4 + 4096, dtype=torch.uint8, device="cuda")
    acc = torch.zeros(nodes, 3, dtype=torch.float64, device="cuda")
    device_harness.call(reduce, s, ctypes.c_uint64(n), nodes, parts, int(scores.dtype == np.float64),
                        int(nan), scratch, acc)
    return acc.cpu().numpy()


@pytest.mark.parametrize("nan", [False, True])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,parts", [(1024, 1), (1000, 1), (40, 1), (4096, 4), (32768, 32)])
def test_sums_that_cancel(reduce, n, parts, dtype, nan):
    """One score per thread and zeros (a thread's own sum is exact then), large
    ones in pairs of opposite sign: the mean is right to its last bits (the sum's
    and the quotient's rounding), although the partial sums are 2^30 times it."""
    rng = np.random.default_rng(n)
    nodes = 6
    s = np.zeros((nodes, n), dtype)
    step = 4 if dtype == np.float32 else 1     # binary32 scores are read four at a time
    at = np.arange(step, n - 3, step)          # (the first score, the shift, is zero)
    per = -(-n // parts)
    if dtype == np.float64:                    # one per thread of a block
        at = at[(at % per) < 256]
    for i in range(nodes):
        k = len(at) // 3
        big = (rng.uniform(1, 2, k) * 2.0 ** rng.integers(0, 30, k)).astype(dtype)
        v = np.concatenate([big, -big, rng.uniform(0.5, 1, len(at) - 2 * k).astype(dtype)])
        s[i, at] = v[rng.permutation(len(at))]
    if nan:
        s[:, 2] = np.nan
    r = _run(reduce, s, parts, nan)
    kept = n - int(nan)
    for i in range(nodes):
        v = s[i][~np.isnan(s[i])].astype(float)
        exact = math.fsum(v) / kept
        assert r[i, 0] == kept
        assert abs(r[i, 1] - exact) <= 3 * 2.0 ** -53 * abs(exact), (i, r[i, 1], exact)
        m2 = math.fsum((v - exact) ** 2)       # (the squares to 2^-48, as two floats)
        assert abs(r[i, 2] - m2) <= 2.0 ** -46 * m2


@pytest.mark.parametrize("n,parts", [(1, 1), (7, 1), (5000, 1), (40000, 8)])
def test_scores_of_one_size(reduce, n, parts):
    rng = np.random.default_rng(n)
    s = rng.uniform(0.3, 2.0, (5, n)).astype(np.float32)
    r = _run(reduce, s, parts, False)
    for i in range(5):
        v = s[i].astype(float)
        m = math.fsum(v) / n
        assert abs(r[i, 1] - m) <= 2.0 ** -46 * m
        m2 = math.fsum((v - m) ** 2)
        assert abs(r[i, 2] - m2) <= 2.0 ** -40 * max(m2, 1e-300)


def test_infinite_scores(reduce):
    s = np.ones((3, 300), np.float32)
    s[0, 7] = np.inf
    s[1, 7], s[1, 200] = np.inf, -np.inf
    r = _run(reduce, s, 1, False)
    assert not np.isfinite(r[:2, 1]).any() and r[2, 1] == 1.0 and r[2, 2] == 0.0
