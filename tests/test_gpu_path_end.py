"""GPU check of the forward path kernel's end, where a warp's last paths are run
with several lanes to each: the first paths of a solve, alone (so that they run
there from their start or after a few units), must be bit for bit those of a
solve in which they ran among thousands of others, at path counts around every
group size, with and without a step cap that ends some of them."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PROBS = {"square": (W.laplace_expcos(), W.nodes_cfg1(2)),
         "lshape": (W.laplace_expcos("l_shape"), W.nodes_lshape_interfaces(2)),
         "cube": (W.elliptic_manufactured(), W.nodes_cube_planes(2)),
         "fourier": (W.poisson_fourier(5), W.nodes_cfg5(1)[:2])}


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api as a
    assert torch.cuda.is_available()
    return a


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(PROBS))
@pytest.mark.parametrize("cap", [10 ** 6, 90])
def test_same_paths(api, name, precision, cap):
    prob, nodes = PROBS[name]
    kw = dict(seed=W.SEED_BASE + 91, dt=1e-3, precision=precision, max_steps=cap, dump_paths=True)
    with api.Context(prob) as ctx:
        t = torch.from_numpy(nodes)
        big = ctx.interface_solve(t, n_paths=4096, **kw)
        for count in (1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 40, 129):
            few = ctx.interface_solve(t, n_paths=count, **kw)
            for k in ("score", "steps", "exit"):
                assert torch.equal(few[k], big[k][:, :count]), (count, k)
            assert np.isclose(few["mean"].cpu().numpy(), few["score"].cpu().numpy().mean(1),
                              rtol=1e-12, atol=1e-15).all()
            assert few["capped"] == int((few["steps"] < 0).sum())
            assert few["path_steps"] == int(few["steps"].abs().sum())
