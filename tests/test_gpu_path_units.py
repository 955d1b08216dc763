"""GPU checks of the forward path kernel's unit scheme (branch-free units of
four steps, parked units rerun with the exact tests, the loop at the wave's
end) at the sizes where it can go wrong, path by path against the FP64 oracle:
path counts around a warp and a block, step caps around a unit, time steps on
both sides of the L-shape's two-face rule and the largest allowed one, with and
without the bridge test, both precisions."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu

PROBS = {"square": (W.laplace_expcos(), "unit_square", W.nodes_cfg1(5)),
         "lshape": (W.laplace_expcos("l_shape"), "l_shape", W.nodes_lshape_interfaces(5)),
         "cube": (W.elliptic_manufactured(), "unit_cube", W.nodes_cube_planes(5)),
         "fourier": (W.poisson_fourier(5), "unit_square", W.nodes_cfg5(2)[:5])}


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api as a
    assert torch.cuda.is_available()
    return a


def _compare(api, orc, name, precision, nodes=None, **kw):
    prob, geometry, all_nodes = PROBS[name]
    nodes = all_nodes if nodes is None else all_nodes[:nodes]
    with api.Context(prob) as ctx:
        g = ctx.interface_solve(torch.from_numpy(nodes), precision=precision, dump_paths=True, **kw)
        plain = ctx.interface_solve(torch.from_numpy(nodes), precision=precision, **kw)
    o = orc.interface_solve(prob, nodes, dump_paths=True, **kw)
    tol = {"path_tol": 1e-11} if precision == "fp64" else {"prob": prob}
    c = parity.compare_paths(g, o, geometry=geometry, **tol)
    parity.report(f"{name} {precision} {kw}", c)
    assert c["mismatch"] == 0, c
    # an exit flip is a binary32 (or, rarely, rounding-level binary64) event: the
    # suite's limit, and one path of a small case
    assert c["step_flips"] + c["face_flips"] <= max(1, 2e-4 * c["paths"]), c
    assert g["capped"] == int((g["steps"] < 0).sum())
    for k in ("mean", "se", "n"):
        assert torch.equal(g[k], plain[k])
    assert np.array_equal(g["n"].cpu().numpy(), o["n"])
    return g, o


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(PROBS))
@pytest.mark.parametrize("nodes,n_paths", [(1, 1), (1, 31), (1, 33), (3, 43), (5, 26), (5, 1031)])
def test_path_counts(api, orc, name, precision, nodes, n_paths):
    _compare(api, orc, name, precision, nodes=nodes, seed=W.SEED_BASE + 41, dt=1e-3,
             n_paths=n_paths)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", ["square", "cube", "lshape"])
@pytest.mark.parametrize("cap", [1, 3, 4, 5, 8, 41])
def test_step_caps(api, orc, name, precision, cap):
    g, o = _compare(api, orc, name, precision, seed=W.SEED_BASE + 42, dt=2e-3, n_paths=200,
                    max_steps=cap)
    assert g["capped"] == o["capped"] or abs(g["capped"] - o["capped"]) <= 1


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("bridge", [True, False])
@pytest.mark.parametrize("name,dt", [("lshape", 1.2e-3), ("lshape", 1.3e-3), ("lshape", 0.02),
                                     ("square", 0.0277), ("cube", 0.0277), ("fourier", 0.01)])
def test_time_steps(api, orc, name, dt, bridge, precision):
    _compare(api, orc, name, precision, seed=W.SEED_BASE + 43, dt=dt, n_paths=4000, bridge=bridge)
