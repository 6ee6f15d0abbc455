"""FP32 transfers far from a particle's origin: a node's place within its cell keeps its
digits although the coordinate it comes from is tens or thousands of cells. Velocities
interpolated from a field without smoothness, against the FP64 path on the same rounded
positions: relative L2 3e-7 (place, weights and sums are each within 1e-7; the rounding
of the coordinate itself, in cells, was added to that before) and, at 3000 cells,
where positions still resolve the cell to 1e-4, the same. Nodes at and just below
cell faces, and coordinates beyond 2^24 cells, stay finite."""
import dataclasses

import numpy as np
import pytest

import ifem_workloads as W

pytestmark = pytest.mark.gpu


def _velocities(x, n, kernel, precision, u, origin):
    from paper_1807_08219_gb300 import ifem as I
    w = W.make("C1")
    w = dataclasses.replace(w, boxes=[W.Box(n, 1.0)], u=[u],
                            instances=[dataclasses.replace(w.instances[0], origin=origin, x_local=x)])
    cp = I.Coupler(w, precision=precision, kernel=kernel)
    try:
        v = cp.empty_nodes()
        I.ifem_interpolate(cp.ctx, cp.batch, cp.grid, cp.grid_to_device(w.u), cp.nodes_to_device(x), v)
        I.ifem_sync_status(cp.ctx)
        return cp.nodes_to_host(v)
    finally:
        cp.close()


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("n,cells", [(64, 5), (96, 30), (57, 50), (101, 3000)])
def test_place_within_the_cell(n, cells, kernel):
    rng = np.random.default_rng(n)
    N = W.make("C1").n_nodes
    x = rng.uniform(-cells / n, cells / n, (N, 3)).astype(np.float32).astype(np.float64)
    u = rng.standard_normal((3, n, n, n)).astype(np.float32).astype(np.float64)
    origin = np.array([0.25, 0.5, 0.75])   # whole numbers of 1/64 cells: exact in FP32
    origin = np.round(origin * n * 64) / (n * 64)
    got, ref = (_velocities(x, n, kernel, p, u, origin) for p in (0, 1))
    assert np.linalg.norm(got - ref) < 3e-7 * np.linalg.norm(ref)


@pytest.mark.parametrize("kernel", [0, 1])
def test_faces_and_far_cells(kernel):
    n, N = 48, W.make("C1").n_nodes
    rng = np.random.default_rng(1)
    u = np.ones((3, n, n, n))
    for scale in (1.0, 1e6, 1e9):
        x = rng.integers(-n, n, (N, 3)) / n * scale
        x[::3] = np.nextafter(x[::3].astype(np.float32), np.float32(-np.inf))
        x[1::3] = np.nextafter(x[1::3].astype(np.float32), np.float32(np.inf))
        v = _velocities(x, n, kernel, 0, u, np.zeros(3))
        assert np.abs(v - 1.0).max() < 1e-5


@pytest.mark.parametrize("case", ["C1", "C2"])
def test_smooth_fields(case):
    """Velocities from a smooth field: relative L2 5.5e-8 against FP64 (the rounding of v
    itself is 2.5e-8, of its sums about 4e-8; weights that do not sum to 1 to the last
    bit would add 4e-8)."""
    from paper_1807_08219_gb300 import ifem as I
    w = W.make(case)
    xl = w.x_local_all(np.float32).astype(np.float64)
    got = []
    for precision in (0, 1):
        cp = I.Coupler(w, precision=precision)
        try:
            u = cp.grid_to_device([q.astype(np.float32).astype(np.float64) for q in w.u])
            v = cp.empty_nodes()
            I.ifem_interpolate(cp.ctx, cp.batch, cp.grid, u, cp.nodes_to_device(xl), v)
            got.append(cp.nodes_to_host(v))
        finally:
            cp.close()
    assert np.linalg.norm(got[0] - got[1]) < 5.5e-8 * np.linalg.norm(got[1])
