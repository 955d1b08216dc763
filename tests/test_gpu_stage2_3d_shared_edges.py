"""Grid points that boxes of the split cube share (pdd_elliptic3d_stage2):
each is written by one box.  On an edge of the cube's boundary the value is g
at the box's own coordinate, and with these grids lo + h (m - 1) of one box is
not the next box's lo to the last bit."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

# (split, grid); the last is a control whose coordinates are exact
_GRIDS = [(2, 99), (4, 197), (5, 56), (4, 33)]


def _uneven(split, grid):
    """Interfaces whose coordinate differs between the two boxes beside it
    (the products and sums rounded once, as a fused multiply-add does)."""
    m = (grid - 1) // split + 1
    out = []
    for k in range(split - 1):
        lo, hi = k / split, (k + 1) / split
        h = (hi - lo) / (m - 1)
        if float(Fraction(lo) + Fraction(h) * (m - 1)) != hi:
            out.append(k + 1)
    return out


def test_grids_have_uneven_interfaces():
    for split, grid in _GRIDS[:-1]:
        assert _uneven(split, grid), (split, grid)
    assert not _uneven(*_GRIDS[-1])


@pytest.mark.gpu
@pytest.mark.parametrize("method", ["dst", "jacobi"])
@pytest.mark.parametrize("split,grid", _GRIDS)
def test_shared_edges(split, grid, method):
    """The bits of the boxes solved on their own and copied in order, the last
    along every axis over the others; and the same bits in every call."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    rng = np.random.default_rng(grid)
    n = 90
    axis = rng.integers(0, 3, n)
    nodes = rng.uniform(0.02, 0.98, (n, 3))
    nodes[np.arange(n), axis] = rng.integers(1, split, n) / split
    values = np.sin(np.pi * nodes[:, 0]) * np.sin(np.pi * nodes[:, 1]) * np.exp(nodes[:, 2])
    m = (grid - 1) // split + 1
    kw = dict(method=method, tol=1e-9 if method == "dst" else 0.0,
              max_iter=200 if method == "dst" else 17)   # (an odd count ends in the second buffer)
    with api.Context(W.elliptic_manufactured()) as ctx:
        r = api.elliptic3d_pdd_solve(ctx, nodes, values, axis, grid=grid, split=split, n_bnd=4, **kw)
        again = [api.elliptic3d_pdd_solve(ctx, nodes, values, axis, grid=grid, split=split, n_bnd=4,
                                          **kw)["u"] for _ in range(3)]
        pv = r["plane_values"]
        u = torch.empty_like(r["u"])
        for kk in np.ndindex(split, split, split):
            kk = kk[::-1]
            sl = [slice(c * (m - 1), c * (m - 1) + m) for c in kk]
            faces = {}
            for a in range(3):
                o = [b for b in range(3) if b != a]
                for side in (0, 1):
                    if 0 < kk[a] + side < split:
                        faces[2 * a + side] = pv[(a, kk[a] + side)][sl[o[1]], sl[o[0]]].contiguous()
            b = ctx.subdomain_solve3d([c / split for c in kk], [(c + 1) / split for c in kk],
                                      (m, m, m), faces, **kw)
            u[sl[2], sl[1], sl[0]] = b["u"]
    assert torch.equal(r["u"], u)
    for v in again:
        assert torch.equal(v, r["u"])
