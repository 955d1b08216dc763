"""Two contexts in two host threads: a solve of small systems beside one of
large systems (whose kernels need far more shared memory) changes nothing for
either."""
import threading

import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _boxes(api, ctx, n):
    return ctx.subdomain_solve3d((0.25, 0.5, 0.0), (0.5, 0.75, 0.25), n, {}, tol=0.0, max_iter=12)["u"]


def _planes(api, ctx, m):
    rng = np.random.default_rng(m)
    x = rng.uniform(0.02, 0.98, (m, 3))
    x[:, 0] = 0.5
    return ctx.interface_interp([(0, 0.5, x, rng.standard_normal(m))], [x[:64]], n_bnd=1)[0]


@pytest.mark.parametrize("solve,large,small", [(_boxes, (128, 128, 6), (5, 6, 7)),
                                               (_planes, 1500, 9)])
def test_small_solves_beside_large_ones(solve, large, small):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1705_03666_gb300 import api
    failed, done = [], threading.Event()

    def work(size, until, least):
        try:
            with torch.cuda.stream(torch.cuda.Stream()), api.Context(W.elliptic_manufactured()) as ctx:
                ref = solve(api, ctx, size).clone()
                k = 0
                while k < least or not until():
                    got = solve(api, ctx, size)
                    torch.cuda.current_stream().synchronize()
                    assert torch.equal(got, ref)
                    k += 1
        except BaseException as e:   # reported by the test's own thread
            failed.append(repr(e))
        finally:
            done.set()

    a = threading.Thread(target=work, args=(large, lambda: True, 60))
    b = threading.Thread(target=work, args=(small, done.is_set, 1))
    a.start()
    b.start()
    a.join(120)
    b.join(120)
    assert not a.is_alive() and not b.is_alive()
    assert not failed, failed
