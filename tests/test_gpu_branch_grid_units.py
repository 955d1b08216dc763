"""GPU checks of the grid-tree kernel's batching (lanes whose step may exit or
whose particle or tree is over wait and are served together, the exits' boundary
data and the scores one (lane, time) pair per lane) at its edges, tree by tree
against the FP64 oracle: time counts around the powers of two that the pairs are
laid out by, tree counts around a warp, steps longer than the grid spacing and
than the distance bound's two-face range, boundary nodes, offspring laws with
none and several children, pruned trees.  The tolerances are those of the
existing tree-by-tree comparison."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W
from test_gpu_branch_grid import FLIP_MAX, _parity, api  # noqa: F401  (api: fixture)

pytestmark = pytest.mark.gpu

SQ = np.array([[0.5, 0.5], [0.0, 0.4], [0.97, 0.96], [1.0, 1.0], [0.2, 0.02]])
LS = np.array([[0.25, 0.75], [0.5, 0.75], [0.49, 0.49], [0.75, 0.25]])


@pytest.mark.parametrize("m,trees,dt", [(1, 1, 1e-3), (2, 33, 1e-3), (3, 1000, 1e-3), (5, 700, 0.4),
                                        (16, 700, 2e-3), (17, 700, 0.03), (32, 700, 1e-2)])
@pytest.mark.parametrize("geometry,law", [("unit_square", None), ("unit_square", "mixed"),
                                          ("l_shape", None), ("interval", "mixed")])
def test_batches(api, orc, m, trees, dt, geometry, law):
    dim = 1 if geometry == "interval" else 2
    kw = {} if law is None else dict(q=(0.2, 0.3, 0.2, 0.3), alpha=(0.5, -0.2, 0.7, 0.4))
    prob = W.kpp("travelling", 1.1, 4.0, dim=dim, geometry=geometry, **kw)
    nodes = {"unit_square": SQ, "l_shape": LS, "interval": SQ[:, :1]}[geometry]
    times = np.cumsum(0.01 + 0.4 / m * (1.0 + 0.5 * np.sin(np.arange(m))))
    _parity(api, orc, prob, nodes, times, FLIP_MAX, seed=31 + m, n_trees=trees, dt=dt)


@pytest.mark.parametrize("cap", [2, 5])
def test_pruned_in_a_domain(api, orc, cap):
    prob = W.kpp("const", 0.5, 6.0, geometry="unit_square")
    g, o, _ = _parity(api, orc, prob, SQ[:1], np.array([0.3, 0.8]), FLIP_MAX, seed=8, n_trees=2000,
                      dt=2e-3, max_particles=cap, max_depth=4)
    assert o["discarded"][0] > 20
