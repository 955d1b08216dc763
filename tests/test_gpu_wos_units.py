"""GPU checks of the Walk on Spheres kernel's units (four jumps per Philox
block, starts and stopped walks staged 32 at a time, sums kept per warp while
the node repeats) at their edges, walk by walk against the FP64 oracle: counts
around a warp, many nodes of few walks (the node changes within a flush), caps
around a unit, nodes on the boundary and outside."""
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


@pytest.mark.parametrize("geometry", ["unit_square", "l_shape"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,walks,cap", [(1, 1, 10 ** 6), (1, 31, 10 ** 6), (1, 33, 10 ** 6),
                                         (200, 3, 10 ** 6), (7, 1031, 10 ** 6), (3, 100, 1),
                                         (3, 100, 4), (3, 100, 5)])
def test_counts_and_caps(api, orc, geometry, precision, n, walks, cap):
    prob = W.laplace_expcos(geometry)
    nodes = W.nodes_cfg1(n) if geometry == "unit_square" else W.nodes_lshape_interfaces(n)
    kw = dict(seed=W.SEED_BASE + 51, n_paths=walks, eps=1e-3, max_steps=cap)
    with api.Context(prob) as ctx:
        g = ctx.wos_solve(torch.from_numpy(nodes), precision=precision, dump_paths=True, **kw)
        plain = ctx.wos_solve(torch.from_numpy(nodes), precision=precision, **kw)
    o = orc.wos_solve(prob, nodes, dump_paths=True, **kw)
    # a walk is a flip when it stops at another jump (|d - eps| below rounding);
    # the scores themselves, whose rounding a walk amplifies from jump to jump,
    # are compared in test_gpu_wos.py
    st, so = g["steps"].cpu().numpy(), o["steps"]
    flips = int((st != so).sum())
    assert flips <= max(1, 1e-3 * st.size), flips
    s = g["score"].cpu().numpy()
    np.testing.assert_allclose(g["mean"].cpu().numpy(), s.mean(1), rtol=1e-13)
    if walks > 1:
        np.testing.assert_allclose(g["se"].cpu().numpy(), s.std(1, ddof=1) / np.sqrt(walks),
                                   rtol=1e-9, atol=1e-16)
    for k in ("mean", "se", "n"):
        assert torch.equal(g[k], plain[k])
    assert g["path_steps"] == int(np.abs(st).sum())


def test_boundary_and_outside_nodes(api):
    with api.Context(W.laplace_expcos()) as ctx:
        nodes = torch.tensor([[0.0, 0.3], [0.5, 0.5], [1.5, 0.5]], dtype=torch.float64)
        r = ctx.wos_solve(nodes, seed=3, n_paths=100, eps=1e-3)
    m, se, n = (r[k].cpu().numpy() for k in ("mean", "se", "n"))
    assert abs(m[0] - np.cos(0.3)) < 1e-6 and se[0] == 0.0
    assert np.isfinite(m[1]) and np.isnan(m[2]) and np.isnan(se[2])
    assert n.tolist() == [100, 100, 100]
