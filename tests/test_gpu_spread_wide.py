"""IFEM_SPREAD_ACC=64: the reproducible FP32 spread with 64-bit accumulators. One node's
force is 1e7 times the others'; away from its stencil the field still has FP32 accuracy
(relative L2 1e-5 of the spread of |F| there, against the FP64 spread of the same
forces; 32 bits leave 1e-3 to 1e-2). The same bits from run to run, fused into a step or
not, added or not; a step's velocities and update as without."""
import numpy as np
import pytest

from tests.test_gpu_transfer_tile import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("sizes,tile", [([32], 16), ([33], 12), ([24, 17, 40], 8), ([49], 11), ([8], 16)])
def test_small_forces_beside_a_large_one(sizes, tile, kernel, monkeypatch):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    w = _workload(sizes, 2, seed=tile)
    x32 = w.x_local_all().astype(np.float32)
    F32 = np.random.default_rng(2).standard_normal(x32.shape).astype(np.float32)
    F32[5] = 1e7
    large = np.zeros_like(F32)
    large[5] = 1.0

    def coupler(precision):
        return I.Coupler(w, precision=precision, kernel=kernel, tile=tile if precision == 0 else 6)

    def spread(cp, F, flags=I.IFEM_SPREAD_OVERWRITE, f=None):
        f = cp.zeros_grid() if f is None else f
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, cp.nodes_to_device(x32), cp.nodes_to_device(F), f, flags)
        I.ifem_sync_status(cp.ctx)
        return f

    ref = coupler(1)
    try:
        want, away = spread(ref, F32).cpu(), spread(ref, large).cpu() == 0
        size = float(spread(ref, np.abs(F32)).cpu()[away].norm())
    finally:
        ref.close()
    narrow = coupler(0)
    monkeypatch.setenv("IFEM_SPREAD_ACC", "64")
    wide = coupler(0)
    try:
        got = spread(wide, F32)
        assert float((got.double().cpu() - want)[away].norm()) < 1e-5 * size
        assert torch.equal(got, spread(wide, F32))
        base = torch.full_like(got, 0.25)
        assert torch.equal(spread(wide, F32, 0, base.clone()), torch.where(got == 0, base, base + got))
        x, u = wide.nodes_to_device(x32), wide.grid_to_device([q.astype(np.float32) for q in w.u])
        out = []
        for cp in (wide, narrow):
            F, v, xn, f = cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes(), cp.zeros_grid()
            red = torch.zeros(12 * len(w.instances) + 6 * len(w.boxes), dtype=torch.float64, device=cp.device)
            I.ifem_step_coupling_ab2(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, red, I.IFEM_SPREAD_OVERWRITE, x, 0.1, xn)
            I.ifem_sync_status(cp.ctx)
            out.append((F, v, xn, f, red))
        assert all(torch.equal(a, b) for a, b in zip(out[0][:3], out[1][:3]))
        assert torch.equal(out[0][3], spread(wide, out[0][0].cpu().numpy().T))
        # the boxes' sums are those of the field
        at = 12 * len(w.instances)
        for b, box in enumerate(w.boxes):
            mine = out[0][3][wide.box_off[b]:wide.box_off[b] + 3 * box.n ** 3].view(3, -1).double()
            h3 = (box.L / box.n) ** 3
            assert float((out[0][4][at + 6 * b:at + 6 * b + 3] - h3 * mine.sum(1)).abs().max()) < 1e-6 * h3 * float(mine.abs().sum())
    finally:
        wide.close()
        narrow.close()
