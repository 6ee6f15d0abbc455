"""The reproducible FP32 spread onto a field that is not cleared: every value that a
node reaches becomes, to the bit, the FP32 sum of what it was and what the same
spread gives a cleared field; the others keep their values (NaN among them). Tiles with even and odd edges, grids whose rows are
not pairs or quads, fields off 16 and 8 bytes, tiles without nodes, one tile or two
per axis."""
import dataclasses

import numpy as np
import pytest

from tests.test_gpu_transfer_tile import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("sizes,tile,shift", [
    ([64], 16, 0), ([64], 15, 0), ([33], 8, 0), ([34], 16, 1), ([34], 16, 2), ([48], 13, 0), ([49], 0, 3), ([8], 16, 0),
    ([13], 6, 1), ([24, 17, 40], 11, 0), ([21, 96], 16, 0)])
def test_adds_what_a_cleared_field_gets(sizes, tile, shift, kernel):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    w = _workload(sizes, 2, seed=tile + shift)
    if len(sizes) > 2:
        w = dataclasses.replace(w, instances=[i for i in w.instances if i.box != 1])
    cp = I.Coupler(w, precision=I.IFEM_FP32, kernel=kernel, tile=tile)
    try:
        g = torch.Generator(device=cp.device).manual_seed(5)
        x = cp.nodes_to_device(w.x_local_all())
        F = torch.randn((3, cp.N), generator=g, device=cp.device)
        store = torch.empty(cp.G + 16, device=cp.device)
        f = store[shift:cp.G + shift]
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F, f, I.IFEM_SPREAD_OVERWRITE)
        S = f.clone()
        base = torch.randn(cp.G, generator=g, device=cp.device) * S.abs().max()
        none = (S == 0).nonzero().flatten()
        assert len(none) > 16 or max(sizes) < 16
        base[none[::3]] = float("nan")
        F2, v, u = torch.empty_like(F), torch.empty_like(F), torch.randn(cp.G, generator=g, device=cp.device)
        for step in (False, True):
            if step:   # the forces of a step are its own
                I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F2, f, v, None, I.IFEM_SPREAD_OVERWRITE)
                S = f.clone()
            f.copy_(base)
            if step:
                I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F2, f, v, None, 0)
            else:
                I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F, f, 0)
            I.ifem_sync_status(cp.ctx)
            want = torch.where(S == 0, base, base + S)
            assert torch.equal(f.isnan(), want.isnan()) and torch.equal(f.nan_to_num(), want.nan_to_num())
    finally:
        cp.close()
