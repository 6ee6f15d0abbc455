"""Calls on a grid other than the one the batch was created on. Every call takes
its own grid of the context: a coarser or a finer one, or one with further boxes.
The field lies between margins that hold a marker: what a call clears, adds and
writes ends with the grid of the call. Fields equal those of a batch created on
that grid: the same bits where the order of a value's terms is fixed, else
within the FP32 tolerance (relative L2 1e-5, of the spread of |F|)."""
import dataclasses

import numpy as np
import pytest

import ifem_workloads as W

pytestmark = pytest.mark.gpu

MARK, MARGIN = 12345.0, 1 << 16


def _workload(precision):
    w = W.make("C1")
    x = w.x_local_all().astype(np.float32 if precision == 0 else np.float64)
    return dataclasses.replace(w, instances=[dataclasses.replace(w.instances[0], x_local=x)])


def _calls(cp, grid, step, flags):
    """Spread (or a step) into a field of `grid` between margins; the field, its size and |F|'s."""
    import torch
    from paper_1807_08219_gb300 import ifem as I
    G = I.ifem_grid_values(grid)
    store = torch.full((G + 2 * MARGIN,), MARK, dtype=cp.dtype, device=cp.device)
    f = store[MARGIN:MARGIN + G]
    f.fill_(0.25)
    x = cp.nodes_to_device(cp.wl.x_local_all())
    g = torch.Generator(device=cp.device).manual_seed(3)
    F = torch.randn((3, cp.N), generator=g, device=cp.device, dtype=cp.dtype)
    if step:
        u = torch.randn(G, generator=g, device=cp.device, dtype=cp.dtype)
        F, v = torch.empty_like(F), torch.empty_like(F)
        I.ifem_step_coupling(cp.ctx, cp.batch, grid, x, u, F, f, v, None, flags)
    else:
        I.ifem_spread(cp.ctx, cp.batch, grid, x, F, f, flags)
    I.ifem_sync_status(cp.ctx)
    assert bool((store[:MARGIN] == MARK).all()) and bool((store[MARGIN + G:] == MARK).all())
    got = f.clone()
    I.ifem_spread(cp.ctx, cp.batch, grid, x, F.abs(), f, I.IFEM_SPREAD_OVERWRITE)
    return got, float(f.double().norm())


@pytest.mark.parametrize("step", [False, True])
@pytest.mark.parametrize("overwrite", [False, True])
@pytest.mark.parametrize("precision,kernel,scatter,first,call", [
    (1, 0, 0, [64], [40]), (1, 0, 0, [40], [64]), (1, 1, 0, [48], [33]), (1, 1, 0, [33], [48]),
    (0, 0, 0, [64], [40]), (0, 0, 1, [40], [64]), (0, 1, 0, [48], [33]),
    (0, 0, 0, [64], [64, 24]), (0, 0, 1, [64], [64, 24]), (0, 1, 0, [64], [64, 24]),
    (0, 0, 0, [64, 24], [64]), (0, 0, 1, [64, 24], [64]), (0, 1, 0, [64, 24], [64]),
    (0, 0, 0, [64, 160], [64]), (0, 0, 0, [64], [64, 160])])   # above 8 MB a step clears another way
def test_another_grid(precision, kernel, scatter, first, call, overwrite, step):
    from paper_1807_08219_gb300 import ifem as I
    flags = I.IFEM_SPREAD_OVERWRITE if overwrite else 0
    w = _workload(precision)
    got = []
    for create in (first, call):
        cp = I.Coupler(dataclasses.replace(w, boxes=[W.Box(n, 1.0) for n in create]), precision=precision,
                       kernel=kernel, scatter=scatter)
        try:
            grid = I.ifem_grid_create(cp.ctx, call, [1.0] * len(call))
            got.append(_calls(cp, grid, step, flags))
            I.ifem_grid_destroy(grid)
        finally:
            cp.close()
    if precision == 1 or scatter == 0 or kernel == 1:
        assert bool((got[0][0] == got[1][0]).all())
    else:
        assert float((got[0][0].double() - got[1][0].double()).norm()) < 1e-5 * got[1][1]


@pytest.mark.parametrize("precision", [0, 1])
def test_grid_at_the_address_of_a_destroyed_one(precision):
    """The batch's tiles follow the grid, not its handle's address."""
    from paper_1807_08219_gb300 import ifem as I
    w = _workload(precision)
    cp = I.Coupler(dataclasses.replace(w, boxes=[W.Box(64, 1.0)]), precision=precision)
    try:
        calls = [[48], [33]]
        first = I.ifem_grid_create(cp.ctx, calls[0], [1.0] * len(calls[0]))
        _calls(cp, first, False, 0)
        at = first.value
        I.ifem_grid_destroy(first)
        grids = []
        while len(grids) < 64 and (not grids or grids[-1].value != at):
            grids.append(I.ifem_grid_create(cp.ctx, calls[1], [1.0] * len(calls[1])))
        if grids[-1].value != at:
            pytest.skip("the allocator did not give the address back")
        got = _calls(cp, grids[-1], False, 0)[0]
        for g in grids[:-1]:
            I.ifem_grid_destroy(g)
        again = I.Coupler(dataclasses.replace(w, boxes=[W.Box(n, 1.0) for n in calls[1]]), precision=precision)
        try:
            assert bool((got == _calls(again, again.grid, False, 0)[0]).all())
        finally:
            again.close()
        I.ifem_grid_destroy(grids[-1])
    finally:
        cp.close()
