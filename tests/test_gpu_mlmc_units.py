"""GPU checks of the multilevel kernel's units (branch-free units of fine and
coarse steps, parked units rerun exactly, finished pairs summed 32 at a time)
at their edges, pair by pair against the FP64 oracle: pair counts around a
warp, caps around a unit, every unit length (refine 2, and 3, 4, 5, 16 as one
coarse step per unit), time steps where a coarse increment reaches far."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("geometry", ["unit_square", "l_shape"])
@pytest.mark.parametrize("level,refine,dt0,pairs,cap", [
    (0, 2, 4e-3, 1, 10 ** 6), (1, 2, 4e-3, 33, 10 ** 6), (0, 2, 4e-3, 700, 4), (1, 2, 4e-3, 700, 8),
    (1, 2, 4e-3, 700, 9), (1, 3, 0.02, 700, 10 ** 6), (2, 4, 4e-3, 700, 10 ** 6),
    (1, 5, 0.0277, 700, 10 ** 6), (1, 16, 0.02, 700, 10 ** 6), (1, 16, 0.02, 300, 40)])
def test_pairs(api, orc, precision, geometry, level, refine, dt0, pairs, cap):
    prob = W.laplace_expcos(geometry)
    nodes = W.nodes_cfg1(3) if geometry == "unit_square" else W.nodes_lshape_interfaces(3)
    kw = dict(seed=W.SEED_BASE + 71, dt0=dt0, level=level, refine=refine, n_paths=pairs,
              max_steps=cap)
    with api.Context(prob) as ctx:
        g = ctx.mlmc_level(torch.from_numpy(nodes), precision=precision, dump_paths=True, **kw)
        plain = ctx.mlmc_level(torch.from_numpy(nodes), precision=precision, **kw)
    o = orc.mlmc_level(prob, nodes, dump_paths=True, **kw)
    ag, ao = g["aux"].cpu().numpy(), np.asarray(o["aux"])
    # exit steps of both walks; a flipped walk is a binary32 event (the suite's
    # limit, and one pair of a small case)
    flip = (ag[..., 2:4] != ao[..., 2:4]).any(-1)
    assert flip.sum() <= max(1, 2e-4 * flip.size), flip.sum()
    # scores of the others: n steps of binary32 (or binary64) rounding of the
    # position, |grad g| <= e, twice for the exit point (grazing exits aside: the
    # exit points themselves must be as near)
    n = np.abs(ao[..., 2:4]).max() * 1.0
    u = 2.0 ** -23 if precision == "fp32" else 2.0 ** -52
    near = np.abs(ag[..., 4:8] - ao[..., 4:8]).max(-1) <= 4 * (n + 8) * u * 2
    d = np.abs(ag[..., :2] - ao[..., :2]).max(-1)
    assert (d[~flip & near] <= 8 * np.e * (n + 8) * u).all()
    assert (~flip & ~near).sum() <= max(1, 0.02 * flip.size)
    s = g["diff"].cpu().numpy()
    np.testing.assert_allclose(g["mean"].cpu().numpy(), s.mean(1), rtol=1e-12, atol=1e-16)
    if pairs > 1:
        np.testing.assert_allclose(g["var"].cpu().numpy(), s.var(1, ddof=1), rtol=1e-9, atol=1e-18)
    np.testing.assert_allclose(g["fine_mean"].cpu().numpy(), ag[..., 0].mean(1), rtol=1e-12)
    np.testing.assert_allclose(g["coarse_mean"].cpu().numpy(), ag[..., 1].mean(1), rtol=1e-12,
                               atol=1e-300)
    for k in ("mean", "var", "fine_mean", "coarse_mean"):
        assert torch.equal(g[k], plain[k])
