"""GPU check of the interface spline (parallel cyclic reduction) and the sine
transforms at the sizes where they can go wrong: two to a few thousand unevenly
spaced nodes (rounds around powers of two, more rows than threads), grids whose
interiors leave partial tiles, are smaller than one, or differ along the axes.
Against scipy's not-a-knot spline and the discrete system itself."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api as a
    assert torch.cuda.is_available()
    return a


@pytest.mark.parametrize("m", [2, 3, 4, 5, 8, 9, 16, 17, 33, 1022, 1023, 3000])
@pytest.mark.parametrize("grid", [(33, 129)])
def test_spline(api, m, grid):
    interpolate = pytest.importorskip("scipy.interpolate")
    rng = np.random.default_rng(m)
    gap = 0.5 + rng.random(m + 1)
    s = np.cumsum(gap)[:-1] / gap.sum()
    vals = np.exp(0.5) * np.cos(s) + 0.01 * np.sin(9 * s)
    with api.Context(W.laplace_expcos()) as ctx:
        u = ctx.subdomain_solve((0.0, 0.0), (0.5, 1.0), grid, iface_axis=0, iface_side=1,
                                iface_s=torch.from_numpy(s), iface_vals=torch.from_numpy(vals),
                                method="dst")["u"].cpu().numpy()
    x = np.concatenate([[0.0], s, [1.0]])
    y = np.concatenate([[np.exp(0.5)], vals, [np.exp(0.5) * np.cos(1.0)]])
    want = interpolate.CubicSpline(x, y, bc_type="not-a-knot")(np.linspace(0.0, 1.0, grid[1]))
    # |y| <= 1.65; the evaluation's four terms and the second derivatives' rounding
    # (12 u |y| / h^2, times h^2 / 8 and the gaps' ratio squared, at most 9) come to
    # about 30 u |y| on either side
    np.testing.assert_allclose(u[:, -1][1:-1], want[1:-1], rtol=0, atol=64 * 2.0 ** -53 * 1.65)


@pytest.mark.parametrize("grid", [(3, 3), (3, 40), (9, 10), (10, 11), (34, 35), (41, 18), (66, 130), (131, 131)])
def test_sine_transforms(api, grid):
    s = np.linspace(0.1, 0.9, 9)
    with api.Context(W.laplace_expcos()) as ctx:
        r = ctx.subdomain_solve((0.0, 0.0), (0.5, 1.0), grid, iface_axis=0, iface_side=1,
                                iface_s=torch.from_numpy(s),
                                iface_vals=torch.from_numpy(np.exp(0.5) * np.cos(s)), method="dst")
    u = r["u"].cpu().numpy()
    hx, hy = 0.5 / (grid[0] - 1), 1.0 / (grid[1] - 1)
    au = ((2 * u[1:-1, 1:-1] - u[1:-1, :-2] - u[1:-1, 2:]) / hx ** 2
          + (2 * u[1:-1, 1:-1] - u[:-2, 1:-1] - u[2:, 1:-1]) / hy ** 2)
    # rounding of the products: a few ulp of |u| <= e times the largest eigenvalue
    scale = 4 / hx ** 2 + 4 / hy ** 2
    assert np.abs(au).max() <= 64 * np.e * 2.0 ** -53 * scale * np.log2(max(grid))
    assert r["resid"] <= 1e-12
