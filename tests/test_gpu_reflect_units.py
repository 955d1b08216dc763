"""GPU checks of the reflecting kernel's units (four steps without a branch,
reflections queued per lane and weighted together, units that may hold an exit
parked and redone exactly) at their edges, path by path against the FP64 oracle:
path counts around a warp, caps around a unit, every number of reflecting faces
(one, two, any), time steps at which a unit reflects more often than a lane's
queue holds.  Per-path bounds and the flip fraction are those of the existing
comparison (one flip allowed in a small case)."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

NODES2 = np.array([[0.5, 0.5], [0.97, 0.03], [0.3, 0.0], [0.0, 0.6], [0.02, 0.98], [1.0, 0.5]])
NODES3 = np.array([[0.5, 0.5, 0.1], [0.03, 0.5, 0.02], [0.0, 0.4, 0.6], [0.9, 0.95, 0.97]])


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api as a
    assert torch.cuda.is_available()
    return a


def _compare(api, orc, prob, nodes, precision, **kw):
    o = orc.interface_solve(prob, nodes, dump_paths=True, **kw)
    with api.Context(prob) as ctx:
        t = torch.from_numpy(nodes)
        g = ctx.interface_solve(t, precision=precision, dump_paths=True, diag=True, **kw)
        plain = ctx.interface_solve(t, precision=precision, **kw)
    how = dict(prob=prob) if precision == "fp32" else dict(path_tol=1e-9)
    c = parity.compare_paths(g, o, geometry=prob["geometry"], **how)
    assert c["mismatch"] == 0, c["max_bound_ratio"]
    assert c["step_flips"] + c["face_flips"] <= max(1, 2e-4 * c["paths"]), c
    assert torch.equal(g["mean"], plain["mean"]) and torch.equal(g["se"], plain["se"])
    np.testing.assert_allclose(g["mean"].cpu().numpy(), g["score"].cpu().numpy().mean(1), rtol=1e-12,
                               atol=1e-15)
    return g, o


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("reflect,phi", [([2], 0.0), ([1, 2], -2.0), ([0, 1], -0.3), ([0, 1, 2], -0.5)])
@pytest.mark.parametrize("paths,dt,cap", [(1, 1e-3, 10 ** 6), (33, 1e-3, 10 ** 6), (600, 1e-3, 1),
                                          (600, 1e-3, 4), (600, 2e-3, 9), (1500, 0.02, 10 ** 6)])
def test_square(api, orc, precision, reflect, phi, paths, dt, cap):
    prob = W.laplace_expcos(reflect=reflect, phi=phi)
    _compare(api, orc, prob, NODES2, precision, seed=W.SEED_BASE + 81, dt=dt, n_paths=paths,
             max_steps=cap)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("reflect,phi", [([5], -1.0), ([0, 4], -1.0), ([0, 2, 3, 5], -0.4)])
@pytest.mark.parametrize("dt,cap", [(1e-3, 10 ** 6), (1e-3, 8), (0.02, 10 ** 6)])
def test_cube(api, orc, precision, reflect, phi, dt, cap):
    prob = W.elliptic_manufactured(reflect=reflect, phi=phi)
    _compare(api, orc, prob, NODES3, precision, seed=W.SEED_BASE + 82, dt=dt, n_paths=500,
             max_steps=cap)


def test_without_the_bridge(api, orc):
    prob = W.laplace_expcos(reflect=[1, 2], phi=-2.0)
    _compare(api, orc, prob, NODES2, "fp32", seed=W.SEED_BASE + 83, dt=1e-3, n_paths=700, bridge=False)
