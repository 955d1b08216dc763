"""The multilevel solve with more nodes times levels than its scratch holds side
by side (1 GiB: the levels then follow one another on one level's scratch): the
level calls' results, the counts, and no more memory than that."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,levels", [(250000, 13), (4, 13)])
def test_many_nodes(n, levels):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    rng = np.random.default_rng(n)
    nodes = rng.uniform(0.05, 0.95, (n, 2))
    nodes[:, 0] = rng.uniform(1e-4, 1e-3, n)
    nodes = torch.from_numpy(nodes).cuda()
    kw = dict(seed=W.SEED_BASE + 95, dt0=2e-2)
    counts = [3] + [1] * (levels - 1)
    with api.Context(W.laplace_expcos()) as ctx:
        free0 = torch.cuda.mem_get_info()[0]
        r = ctx.mlmc_solve(nodes, n_per_level=counts, **kw)
        torch.cuda.synchronize()
        used = free0 - torch.cuda.mem_get_info()[0]
        with_counts = ctx.mlmc_solve(nodes, n_per_level=counts, diag=True, **kw)
        steps = 0
        for l, N in enumerate(counts):
            one = ctx.mlmc_level(nodes, level=l, n_paths=N, diag=True, **kw)
            steps += one["path_steps"]
            for k in ("mean", "var"):
                assert torch.equal(r["levels"][l][k], one[k]), (l, k)
        outside = nodes.clone()
        outside[n // 2, 0] = -0.5
        with pytest.raises(api._lib.PDDError, match="1 pairs|3 pairs"):
            ctx.mlmc_solve(outside, n_per_level=counts, diag=True, **kw)
    assert torch.equal(r["mean"], with_counts["mean"]) and torch.equal(r["se"], with_counts["se"])
    assert with_counts["path_steps"] == steps and with_counts["capped"] == 0
    # the solve's outputs (2 + 2 levels doubles a node) and a GiB of scratch
    assert used <= (2 + 2 * levels) * 8 * n + (1 << 30) + (64 << 20)
