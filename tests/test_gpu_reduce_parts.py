"""GPU check of the per-node reduction with several blocks per node (few nodes,
many scores): means and standard errors against the dumped scores, at score
counts around the sizes where the number of blocks changes, over waves that cut
nodes, for trees (discarded ones left out) and reflecting paths (both
precisions), and the same bits with and without the dump."""
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


def _check(r, plain, count=None):
    s = r["score"].cpu().numpy().astype(np.float64)
    kept = (~np.isnan(s)).sum(1)
    mean = np.nansum(s, 1) / kept
    se = np.sqrt(np.nansum((s - mean[:, None]) ** 2, 1) / (kept - 1) / kept)
    # two-float sums hold 48 bits; the variance is a difference of sums of squares
    # of size s^2, so its error is that of the sums over the variance
    np.testing.assert_allclose(r["mean"].cpu().numpy(), mean, rtol=1e-11)
    big = np.nanmax(s ** 2, 1) / (se ** 2 * kept)
    assert (np.abs(r["se"].cpu().numpy() - se) <= se * (1e-9 + big * 2.0 ** -40)).all()
    assert np.array_equal(r["n"].cpu().numpy(), kept)
    for k in ("mean", "se", "n"):
        assert torch.equal(r[k], plain[k])


@pytest.mark.parametrize("nodes,trees,wave", [(1, 8191, 0), (1, 8192, 0), (3, 16385, 0), (2, 131072, 0),
                                              (3, 40001, 50000), (5, 20000, 31000)])
def test_trees(api, nodes, trees, wave):
    prob = W.kpp("travelling", 1.1, 2.0)
    xt = torch.from_numpy(W.nodes_kpp()[5:5 + 16 * nodes:16].copy())
    with api.Context(prob) as ctx:
        if wave:
            ctx.set_tuning(wave_max_paths=wave)
        kw = dict(seed=W.SEED_BASE + 95, n_trees=trees, max_particles=12)
        _check(ctx.branching_solve(xt, dump_trees=True, **kw), ctx.branching_solve(xt, **kw))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nodes,paths,wave", [(1, 8192, 0), (2, 33000, 0), (3, 12000, 17000)])
def test_reflecting_paths(api, precision, nodes, paths, wave):
    prob = W.laplace_expcos(reflect=[1, 2], phi=-2.0)
    x = torch.from_numpy(W.nodes_cfg1(nodes))
    with api.Context(prob) as ctx:
        if wave:
            ctx.set_tuning(wave_max_paths=wave)
        kw = dict(seed=W.SEED_BASE + 96, dt=2e-3, n_paths=paths, precision=precision)
        _check(ctx.interface_solve(x, dump_paths=True, **kw), ctx.interface_solve(x, **kw))
