"""Interpolation systems without a usable pivot (pdd_interface_interp): a node
with a NaN coordinate makes its row and column NaN, so that from its column on
no unused row has a number in it; coincident nodes make two rows equal.  Both are
reported as singular, and the call after works."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", ["first", "middle", "last", "twin"])
@pytest.mark.parametrize("sizes", [(9, 40), (40, 9), (17, 33), (120, 120, 120), (1700, 30)])
def test_reported_as_singular(sizes, bad):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    from paper_1705_03666_gb300._lib import PDDError
    rng = np.random.default_rng(sum(sizes))
    planes = []
    for p, m in enumerate(sizes):
        x = rng.uniform(0.02, 0.98, (m, 3))
        x[:, p % 3] = 0.5
        planes.append((p % 3, 0.5, x, rng.standard_normal(m)))
    q = [x[:5] for _, _, x, _ in planes]
    with api.Context(W.elliptic_manufactured()) as ctx:
        ref = [v.clone() for v in ctx.interface_interp(planes, q, n_bnd=2)]
        for p, (axis, pos, x, v) in enumerate(planes):
            y = x.copy()
            if bad == "twin":
                y[-1] = y[0]
            else:
                y[{"first": 0, "middle": len(y) // 2, "last": len(y) - 1}[bad], (axis + 1) % 3] = np.nan
            with pytest.raises(PDDError, match="singular"):
                ctx.interface_interp(planes[:p] + [(axis, pos, y, v)] + planes[p + 1:], q, n_bnd=2)
            got = ctx.interface_interp(planes, q, n_bnd=2)
            for a, b in zip(got, ref):
                assert torch.equal(a, b)
