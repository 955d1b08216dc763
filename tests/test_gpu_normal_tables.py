"""Binary64 Box-Muller normals from tables (box_muller_tables): every one of the
2^23 radius codes and of the 2^23 angle codes against log, sqrt, sin and cos."""
import numpy as np
import pytest
import torch

from tests import device_harness

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "normal_tables.cuh"
using namespace pdd;
__global__ void normals(const double2 *t, uint32_t fixed, int vary_angle, double2 *out) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  double z0, z1;
  box_muller_tables(NormalTables(t), (vary_angle ? fixed : k) << 9, (vary_angle ? k : fixed) << 9, z0, z1);
  out[k] = make_double2(z0, z1);
}
extern "C" int tables(void *t) {
  launch_normal_tables(static_cast<double2 *>(t), 0);
  return cudaDeviceSynchronize();
}
extern "C" unsigned long table_bytes() { return kNormalBytes; }
extern "C" int run(const void *t, unsigned fixed, int vary_angle, void *out) {
  normals<<<(1 << 23) / 256, 256>>>(static_cast<const double2 *>(t), fixed, vary_angle,
                                    static_cast<double2 *>(out));
  return cudaDeviceSynchronize();
}
"""

N = 1 << 23
# units in the last place of a normal: 4.5 for the rotation (half a unit each of the
# table's entries, one or two of the library's sine, beside an axis where the result
# is half the larger term), 1.5 for the root, half a unit for the product, 1.5 for
# the references below
TOL = 8.0 * 2.0 ** -52


@pytest.fixture(scope="module")
def normals(tmp_path_factory):
    lib = device_harness.load(str(tmp_path_factory.mktemp("normals")), SOURCE)
    t = torch.empty(lib.table_bytes(), dtype=torch.uint8, device="cuda")
    device_harness.call(lib.tables, t)

    def f(fixed, vary_angle):
        out = torch.empty(N, 2, dtype=torch.float64, device="cuda")
        device_harness.call(lib.run, t, fixed, int(vary_angle), out)
        return out.cpu().numpy()
    return f


def _radius(k):
    return np.sqrt(-2.0 * np.log((2 * k + 1) * 2.0 ** -24))


def _cos_sin(k):
    """cos and sin of 2 pi (2 k + 1) / 2^24, the octant taken in integers."""
    m = 2 * np.asarray(k, dtype=np.int64) + 1
    q, r = m >> 22, m & ((1 << 22) - 1)          # quarter turns and the rest
    swap = r > (1 << 21)
    x = 2.0 * np.pi * np.where(swap, (1 << 22) - r, r) * 2.0 ** -24
    c, s = np.cos(x), np.sin(x)
    c, s = np.where(swap, s, c), np.where(swap, c, s)
    return (np.choose(q, [c, -s, -c, s]), np.choose(q, [s, c, -s, -c]))


@pytest.mark.parametrize("fixed", [0, 4194304, 6291455, N - 1])
def test_every_angle(normals, fixed):
    z = normals(fixed, True)
    k = np.arange(N)
    c, s = _cos_sin(k)
    r = _radius(fixed)
    for got, ref in ((z[:, 0], r * c), (z[:, 1], r * s)):
        worst = np.max(np.abs(got - ref) / np.abs(ref))
        print(f"angles at radius code {fixed}: {worst / 2.0 ** -52:.2f} ulp")
        assert worst <= TOL


@pytest.mark.parametrize("fixed", [0, 2097151, 2097152, 5555555, N - 1])
def test_every_radius(normals, fixed):
    z = normals(fixed, False)
    r = _radius(np.arange(N))
    c, s = _cos_sin(fixed)
    for got, ref in ((z[:, 0], r * c), (z[:, 1], r * s)):
        worst = np.max(np.abs(got - ref) / np.abs(ref))
        print(f"radii at angle code {fixed}: {worst / 2.0 ** -52:.2f} ulp")
        assert worst <= TOL
