"""The position update of a step for nodes whose positions are not finite: they are
in no tile, so the transfer that writes the update beside each velocity does not
visit them. x_new still equals ifem_ab2_update on a copy of x with the v that the
call leaves (bit for bit, NaN where that gives NaN)."""
import numpy as np
import pytest

import ifem_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lost", [[], [0], [5, 6, 640], list(range(642))])
@pytest.mark.parametrize("precision,kernel,scatter", [(0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)])
def test_update_of_lost_nodes(precision, kernel, scatter, lost):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    w = W.make("C1")
    cp = I.Coupler(w, precision=precision, kernel=kernel, scatter=scatter)
    try:
        xl = w.x_local_all()
        for k, i in enumerate(lost):
            xl[i, k % 3] = (np.nan, np.inf, -np.inf)[k // 3 % 3]
        x, u, f = cp.nodes_to_device(xl), cp.grid_to_device(w.u), cp.zeros_grid()
        v, vp, F = (torch.full_like(x, q) for q in (0.5, 0.25, 0.0))
        xn = torch.full_like(x, 7.0)
        I.ifem_step_coupling_ab2(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, None, 0, vp, 0.01, xn)
        rc, st = I.ifem_sync_status(cp.ctx, raise_on_error=False)
        assert (st["domain_errors"] > 0) == bool(lost)
        want = x.clone()
        I.ifem_ab2_update(cp.ctx, cp.batch, want, v, vp, 0.01)
        torch.cuda.synchronize()
        assert torch.equal(xn.isnan(), want.isnan())
        assert torch.equal(xn.nan_to_num(nan=1.0), want.nan_to_num(nan=1.0))
        assert int((~xn.isfinite()).any(0).sum()) == len(lost)
    finally:
        cp.close()
