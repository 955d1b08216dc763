"""Range and resolution of the multilevel sums (pdd_mlmc_level): boundary data
of any magnitude, and scores and differences far below one, against the moments of
the same pairs' own scores in extended precision."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _moments(s):
    s = s.cpu().numpy().astype(np.longdouble)
    m = s.mean(1)
    return m.astype(float), (((s - m[:, None]) ** 2).sum(1) / (s.shape[1] - 1)).astype(float)


def _check(g, n):
    """Means to the rounding of a double; variances likewise (sums of squares of
    exact scores: n roundings of 2^-64 in the reference, one of 2^-53 here), where
    the mean does not cancel more than 2^10 of them."""
    assert g["status"] == 0 or g["capped"] > 0
    m, v = _moments(g["diff"])
    # (a mean is exact to its own last bits; the reference's to n 2^-64 max |s|)
    top = np.abs(g["diff"].cpu().numpy()).max(1)
    assert np.all(np.abs(g["mean"].cpu().numpy() - m) <= 4 * 2.0 ** -53 * np.abs(m) + n * 2.0 ** -64 * top)
    np.testing.assert_allclose(g["var"].cpu().numpy(), v, rtol=2.0 ** -40, atol=0)
    assert np.all(v > 0)


@pytest.mark.parametrize("level", [0, 2])
@pytest.mark.parametrize("precision,factor", [("fp32", 1.0), ("fp32", 2.0 ** 30), ("fp32", 1e15),
                                              ("fp32", 1e36), ("fp64", 2.0 ** 31), ("fp64", 1e140)])
def test_boundary_data_of_any_size(precision, factor, level):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    prob = W.poisson_fourier(5)
    prob["params"] = np.concatenate([prob["params"][:64] * factor, prob["params"][64:]])
    nodes = torch.from_numpy(W.nodes_cfg5(2))
    with api.Context(prob) as ctx:
        g = ctx.mlmc_level(nodes, seed=W.SEED_BASE + 81, dt0=4e-3, level=level, n_paths=1000,
                           precision=precision, dump_paths=True, diag=True)
    _check(g, 1000)


@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_scores_far_below_one(precision, level):
    """No boundary data, a source of one and steps of 10^-12 next to the boundary:
    scores of 10^-12 to 10^-10, squares below 10^-20."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    prob = W.poisson_fourier(5)
    prob["params"] = np.zeros(80)
    nodes = torch.tensor([[2e-6, 0.4], [0.3, 3e-6]], dtype=torch.float64)
    with api.Context(prob) as ctx:
        g = ctx.mlmc_level(nodes, seed=W.SEED_BASE + 82, dt0=1e-12, level=level, n_paths=1000,
                           max_steps=200, precision=precision, dump_paths=True, diag=True)
    _check(g, 1000)
