"""Kernel timing of the multilevel solve (pdd_profile): one timed launch per
level, as many as there are levels, and the same results as without."""
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [1, 2, 4, 5, 9])
def test_every_level_is_timed(levels):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    nodes = torch.from_numpy(W.nodes_cfg1(5))
    kw = dict(seed=W.SEED_BASE + 91, dt0=4e-3, n_per_level=[max(40, 4000 >> l) for l in range(levels)])
    with api.Context(W.laplace_expcos()) as ctx:
        plain = ctx.mlmc_solve(nodes, **kw)
        ctx.profile(True)
        timed = ctx.mlmc_solve(nodes, **kw)
        ms, launches = ctx.profile_read()
        one = [ctx.mlmc_level(nodes, level=l, n_paths=N, **{k: kw[k] for k in ("seed", "dt0")})
               for l, N in enumerate(kw["n_per_level"])]
        ms1, launches1 = ctx.profile_read()
        ctx.profile(False)
        after = ctx.mlmc_solve(nodes, **kw)
        assert ctx.profile_read()[1] == 0
    assert launches == launches1 == levels and ms > 0.0 and ms1 > 0.0
    for r in (timed, after):
        assert torch.equal(r["mean"], plain["mean"]) and torch.equal(r["se"], plain["se"])
    for l in range(levels):
        assert torch.equal(one[l]["mean"], plain["levels"][l]["mean"])
