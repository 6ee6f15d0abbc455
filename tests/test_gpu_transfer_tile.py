"""FP32 tile transfer (own nodes, staged boxes, bank-ordered stencils) at the
sizes where its layout can go wrong: boxes smaller than a tile's halo box, tile
edges that leave every remainder, grids whose rows are not quads, fields that do
not start on 16 bytes, more nodes per tile than threads, one node, every tile
edge's box width, with and without the fused interpolation and position update.
Compared with the FP64 path on the same rounded inputs (positions, velocities
and the forces that are spread: a step's own FP32 forces), within the FP32
tolerances (relative L2 1e-6 on velocities, 1e-5 on the spread field, there of
the spread of |F|: the forces of closed membranes cancel within a cell, the
rounding of the weights, a few 1e-7 cells of position, does not)."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from tests._helpers import rel_l2

pytestmark = pytest.mark.gpu


def _workload(ns, parts, seed=0):
    """Boxes of ns cells with `parts` particles each, some across the periodic faces."""
    rng = np.random.default_rng(seed)
    boxes = [W.Box(n, n / 32.0) for n in ns]
    h = 1.0 / 32
    sizes = [(0, 1.3), (2, 3.2), (3, 2.6)]   # icosphere level, radius in cells: sparse, usual and crowded tiles
    tms = [C.Template("membrane", r * h * M.icosphere(lv)[0], M.icosphere(lv)[1], "nh") for lv, r in sizes]
    inst = []
    for b, box in enumerate(boxes):
        for k in range(parts):
            t = int(rng.integers(0, 3))
            inst.append(C.Instance(t, b, rng.uniform(-0.2, 1.2, 3) * box.L, tms[t].X + 0.05 * h * rng.standard_normal(tms[t].X.shape)))
    u = [rng.standard_normal((3, n, n, n)) for n in ns]
    return W.Workload("tiles", tms, inst, boxes, u, seed)


def _run(w, precision, scatter, tile, shift, flags, ab2, forces=None):
    """forces: spread these after the step instead of the step's own."""
    import torch
    from paper_1807_08219_gb300 import ifem as I
    cp = I.Coupler(w, precision=precision, scatter=scatter, tile=tile)
    try:
        f32 = np.float32
        x = cp.nodes_to_device(w.x_local_all().astype(f32))
        rng = np.random.default_rng(7)
        F0 = cp.nodes_to_device(rng.standard_normal((cp.N, 3)).astype(f32))
        vp = cp.nodes_to_device(rng.standard_normal((cp.N, 3)).astype(f32))
        store = torch.empty(2 * cp.G + 16, dtype=cp.dtype, device=cp.device)
        f, u = store[shift:cp.G + shift], store[cp.G + 8 + shift:2 * cp.G + 8 + shift]   # shift floats off 16 bytes
        u.copy_(cp.grid_to_device([q.astype(f32) for q in w.u]))
        f.fill_(0.25)
        F, v, xn = cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes()
        out = {}
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F0, f, flags)
        out["spread"] = f.double().cpu().numpy().copy()
        I.ifem_interpolate(cp.ctx, cp.batch, cp.grid, u, x, v)
        out["interp"] = cp.nodes_to_host(v)
        f.fill_(0.25)
        v.zero_()
        if ab2:
            I.ifem_step_coupling_ab2(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, None, flags, vp, 1e-3, xn)
            out["x"] = cp.nodes_to_host(xn)
        else:
            I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, None, flags)
        out["F"] = cp.nodes_to_host(F)
        if forces is not None:
            f.fill_(0.25)
            I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, cp.nodes_to_device(forces), f, flags)
            size = cp.zeros_grid()
            for k, G in (("spread", F0), ("f", cp.nodes_to_device(forces))):
                I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, G.abs(), size, flags | I.IFEM_SPREAD_OVERWRITE)
                out["size " + k] = float(size.norm())
        out["f"], out["v"] = f.double().cpu().numpy().copy(), cp.nodes_to_host(v)
        I.ifem_sync_status(cp.ctx)
        return out
    finally:
        cp.close()


def _check(w, tile, shift=0, flags=0, ab2=False):
    from paper_1807_08219_gb300 import ifem as I
    got = _run(w, I.IFEM_FP32, I.IFEM_SCATTER_ATOMIC, tile, shift, flags, ab2)
    ref = _run(w, I.IFEM_FP64, I.IFEM_SCATTER_DET, 6, 0, flags, ab2, forces=got.pop("F"))
    for k in got:
        if k in ("spread", "f"):
            assert np.linalg.norm(got[k] - ref[k]) < 1e-5 * ref["size " + k], k
        else:
            assert rel_l2(got[k], ref[k]) < 1e-6, k


@pytest.mark.parametrize("n", [8, 9, 11, 12, 16, 17, 18, 19, 20, 21, 23, 24, 33, 36, 44])
@pytest.mark.parametrize("tile", [6, 8, 12, 16])
def test_box_sizes(n, tile):
    _check(_workload([n], 3, seed=n), tile)


@pytest.mark.parametrize("tile", [7, 9, 10, 11, 13, 14, 15])
def test_odd_tiles(tile):
    _check(_workload([32, 27], 4, seed=tile), tile)


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("tile", [8, 12, 16])
def test_fields_off_16_bytes(shift, tile):
    _check(_workload([32, 17, 24], 3, seed=shift), tile, shift=shift, ab2=True)


@pytest.mark.parametrize("flags", [0, 1, 2, 3])
@pytest.mark.parametrize("ab2", [False, True])
def test_flags_and_update(flags, ab2):
    _check(_workload([40, 13], 5, seed=flags), 16, flags=flags, ab2=ab2)


@pytest.mark.parametrize("tile", [8, 12, 16])
def test_crowded_tiles(tile):
    """More own nodes in a tile than the kernel has node threads (several rounds of its node loop)."""
    _check(_workload([16], 16, seed=3), tile, ab2=True)
