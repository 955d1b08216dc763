"""Device memory of the interface interpolation: one copy of the systems (the
factored rows stay in them), and what grows with the number of unknowns."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unknowns", [(6000,), (3000, 5000, 3200)])
def test_one_copy_of_the_systems(unknowns):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    rng = np.random.default_rng(len(unknowns))
    planes, queries = [], []
    for p, M in enumerate(unknowns):
        x = rng.uniform(0.01, 0.99, (M - 7, 3))
        x[:, p] = 0.5
        planes.append((p, 0.5, x, rng.standard_normal(M - 7)))
        queries.append(x[:8])
    for _ in range(2):   # (the first loads the kernels)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        with api.Context(W.elliptic_manufactured()) as ctx:
            out = ctx.interface_interp(planes, queries, n_bnd=1)
            torch.cuda.synchronize()
            used = free - torch.cuda.mem_get_info()[0]
    assert all(torch.isfinite(o).all() for o in out)
    systems = sum(8 * M * (M + 1) for M in unknowns)
    # a row keeps its multipliers of two panels and what goes aside (16 columns each
    # at most), a few lists, points and values; the context asks for an eighth more
    # than it needs, and the driver hands it out in blocks
    assert used <= 1.125 * (systems + sum(unknowns) * (3 * 16 * 8 + 64)) + (16 << 20)
