"""Axes of the stage-two nodes (elliptic3d_pdd_solve's node_axis) in every
tensor type: an entry names axis a exactly when it equals a."""
import numpy as np
import pytest
import torch

from paper_1705_03666_gb300 import api, workloads as W

_WHOLE = [torch.bool, torch.uint8, torch.uint16, torch.uint32, torch.uint64, torch.int8,
          torch.int16, torch.int32, torch.int64]
_REAL = [torch.float16, torch.bfloat16, torch.float32, torch.float64, torch.complex64]


@pytest.mark.parametrize("dtype", _WHOLE + _REAL)
def test_axis_conversion(dtype):
    values = [0, 1, 1, 0] if dtype == torch.bool else [0, 1, 2, 1, 3, 100]
    if dtype in (torch.uint16, torch.uint32, torch.uint64):
        values += [(1 << (8 * dtype.itemsize)) - 1, (1 << (8 * dtype.itemsize - 1)) + 1]
    if dtype.is_signed:
        values += [-1, -100]
    if dtype in _REAL:
        values += [0.5, 1.5, float("nan"), float("inf"), -float("inf")]
    if dtype.is_complex:
        values += [1 + 1j, 2j]
    axis = torch.tensor(values, dtype=dtype)
    got = api._axis_i32(axis)
    assert got.dtype == torch.int32
    for a in range(3):
        assert torch.equal(got == a, axis == a), (a, got)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.uint8, torch.uint16, torch.float32])
def test_stage_two_by_axis_type(dtype):
    import __graft_entry__
    __graft_entry__.build()
    nodes = W.nodes_cube_planes(96)
    values = np.sin(np.pi * nodes[:, 0]) * np.sin(np.pi * nodes[:, 1]) * np.exp(nodes[:, 2])
    axis = torch.from_numpy(np.arange(96) % 3)
    kw = dict(grid=17, split=4, n_bnd=4)
    with api.Context(W.elliptic_manufactured()) as ctx:
        ref = api.elliptic3d_pdd_solve(ctx, nodes, values, axis, **kw)
        got = api.elliptic3d_pdd_solve(ctx, nodes, values, axis.to(dtype).cuda(), **kw)
    assert torch.equal(got["u"], ref["u"])
