"""The reproducible FP32 spread (IFEM_SCATTER_DET, and the MLS kernel in both
scatter modes): the values that three or more tiles' boxes can reach are summed
from the stored boxes in a fixed order. At the sizes where that can go wrong: one tile or two
tiles per axis (a tile is its own neighbour), a remainder of one cell, grids
whose rows are not quads, fields off 16 bytes, tiles without nodes, a box
without nodes. Results within the FP32 tolerances of the FP64 path (relative L2
1e-6 on velocities, 1e-5 on the spread field, there of the spread of |F|), the
same bits from run to run and from a fused and a separate transfer, and
overwriting gives the bits of clearing first."""
import numpy as np
import pytest

from tests._helpers import rel_l2
from tests.test_gpu_transfer_tile import _workload

pytestmark = pytest.mark.gpu


def _run(w, precision, scatter, kernel, tile, F, shift=0):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    cp = I.Coupler(w, precision=precision, scatter=scatter, kernel=kernel, tile=tile)
    try:
        f32 = np.float32
        x = cp.nodes_to_device(w.x_local_all().astype(f32))
        Fd = cp.nodes_to_device(F)
        store = torch.empty(2 * cp.G + 16, dtype=cp.dtype, device=cp.device)
        f, u = store[shift:cp.G + shift], store[cp.G + 8 + shift:2 * cp.G + 8 + shift]
        u.copy_(cp.grid_to_device([q.astype(f32) for q in w.u]))
        v, Fs = cp.empty_nodes(), cp.empty_nodes()
        out = {}
        f.fill_(np.nan)
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, Fd, f, I.IFEM_SPREAD_OVERWRITE)
        out["spread"] = f.cpu().numpy().copy()
        f.zero_()
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, Fd, f, 0)
        assert (f.cpu().numpy() == out["spread"]).all()
        f.fill_(0.25)
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, Fd, f, 0)
        out["added"] = f.double().cpu().numpy() - 0.25
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, Fd.abs(), f, I.IFEM_SPREAD_OVERWRITE)
        size = float(f.double().norm())
        I.ifem_interpolate(cp.ctx, cp.batch, cp.grid, u, x, v)
        out["v"] = cp.nodes_to_host(v).copy()
        f.fill_(np.nan)
        I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, Fs, f, v, None, I.IFEM_SPREAD_OVERWRITE)
        out["f"], out["v step"] = f.cpu().numpy().copy(), cp.nodes_to_host(v).copy()
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, Fs, f, I.IFEM_SPREAD_OVERWRITE)
        assert (f.cpu().numpy() == out["f"]).all()
        I.ifem_sync_status(cp.ctx)
        return out, size
    finally:
        cp.close()


def _check(w, kernel, tile, shift=0):
    from paper_1807_08219_gb300 import ifem as I
    F = np.random.default_rng(7).standard_normal((w.x_local_all().shape[0], 3)).astype(np.float32)
    scatters = (I.IFEM_SCATTER_DET, I.IFEM_SCATTER_ATOMIC if kernel else I.IFEM_SCATTER_DET)
    got, again = (_run(w, I.IFEM_FP32, s, kernel, tile, F, shift)[0] for s in scatters)
    ref, size = _run(w, I.IFEM_FP64, I.IFEM_SCATTER_DET, kernel, 6, F)
    for k in got:
        assert (got[k] == again[k]).all(), k
    for k in ("spread", "added"):
        assert np.linalg.norm(got[k].astype(np.float64) - ref[k]) < 1e-5 * size, k
    for k in ("v", "v step"):
        assert rel_l2(got[k], ref[k]) < 1e-6, k


@pytest.mark.parametrize("n", [8, 9, 12, 13, 16, 17, 18, 24, 25, 32, 33, 49])
@pytest.mark.parametrize("tile", [6, 8, 12, 16])
def test_box_sizes(n, tile):
    _check(_workload([n], 3, seed=n), 0, tile)


@pytest.mark.parametrize("tile", [7, 9, 10, 11, 13, 14, 15])
@pytest.mark.parametrize("kernel", [0, 1])
def test_odd_tiles(tile, kernel):
    _check(_workload([32, 27], 4, seed=tile), kernel, tile)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("tile", [8, 12, 16])
@pytest.mark.parametrize("kernel", [0, 1])
def test_fields_off_16_bytes(shift, tile, kernel):
    w = _workload([32, 17, 24], 3, seed=shift)
    w.instances[:] = [i for i in w.instances if i.box != 1]   # the middle box stays empty
    _check(w, kernel, tile, shift=shift)


@pytest.mark.parametrize("n", [8, 9, 16, 17, 21])
@pytest.mark.parametrize("tile", [6, 8, 12, 16])
def test_mls_box_sizes(n, tile):
    _check(_workload([n], 2, seed=n), 1, tile)
