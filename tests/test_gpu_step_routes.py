"""The routes of a step that its sizes choose, on both sides of each line: with host
arrays one launch per lattice (v of 2.5 MB and more, the rows of v going back beside the
later lattices) or one in all, and a field to be cleared with the counters (up to 8 MB)
or on a stream of its own. Eagerly and replayed from a CUDA graph, with and without
IFEM_SPREAD_OVERWRITE, against the device-array step or the separate calls: forces,
velocities and the particles' sums bit for bit, the field to 1e-5 of the spread of |F|
(tiles' halos combine in any order with IFEM_SCATTER_ATOMIC) and the boxes' sums to 1e-6
of the summed magnitudes."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import meshes

pytestmark = pytest.mark.gpu


def _workload(count, n):
    X, f = meshes.icosphere(4)
    k = int(np.ceil(count ** (1 / 3)))
    rng = np.random.default_rng(count)
    X = 0.35 / k * X
    inst = [W.Instance(0, 0, (np.array([i % k, i // k % k, i // k ** 2]) + rng.random(3)) / k,
                       X * rng.uniform(0.9, 1.1, 3)) for i in range(count)]
    return W.Workload("routes", [W.Template("membrane", X, f, "nh")], inst, [W.Box(n, 1.0)], [], count)


def _replayed(call, replay):
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call(s)
        s.synchronize()
        if replay:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                call(s)
            replay()   # the outputs of the eager call go
            torch.cuda.synchronize()
            g.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("overwrite", [False, True])
@pytest.mark.parametrize("count", [85, 86])   # 217770 nodes: 2.49 MB of v, 220332: 2.52 MB
def test_host_rows(count, overwrite, graph):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    flags = I.IFEM_SPREAD_OVERWRITE if overwrite else 0
    w = _workload(count, 96)
    cp = I.Coupler(w, precision=I.IFEM_FP32, scatter=I.IFEM_SCATTER_ATOMIC, tile=16)
    try:
        assert (12 * cp.N >= 5 << 19) == (count == 86)
        g = torch.Generator(device=cp.device).manual_seed(1)
        u = torch.randn(cp.G, generator=g, device=cp.device)
        x = cp.nodes_to_device(w.x_local_all())
        n_red = 12 * count + 6
        F, v, f = cp.empty_nodes(), cp.empty_nodes(), torch.full((cp.G,), 0.5, device=cp.device)
        red = torch.zeros(n_red, dtype=torch.float64, device=cp.device)
        I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, red, flags)
        I.ifem_sync_status(cp.ctx)
        xh = x.cpu().pin_memory()
        vh, rh = torch.empty_like(xh).pin_memory(), torch.empty(n_red, dtype=torch.float64).pin_memory()
        xd, F2, v2, f2, red2 = torch.empty_like(x), torch.empty_like(F), torch.empty_like(v), torch.empty_like(f), torch.empty_like(red)

        def forget():
            for t in (xd, F2, v2, red2, vh, rh):
                t.fill_(-7.0)
            f2.fill_(0.5)

        forget()
        torch.cuda.synchronize()
        _replayed(lambda s: I.ifem_step_coupling_host(cp.ctx, cp.batch, cp.grid, xh, xd, u, F2, f2, v2, vh, red2, rh, flags, s),
                  forget if graph else None)
        I.ifem_sync_status(cp.ctx)
        assert torch.equal(F, F2) and torch.equal(v, v2) and torch.equal(vh, v.cpu()) and torch.equal(rh, red2.cpu())
        assert torch.equal(red[:-6], red2[:-6])
        size = torch.zeros_like(f)
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F.abs(), size, 0)
        assert float((f.double() - f2.double()).norm()) < 1e-5 * float(size.double().norm())
        assert float((red[-6:] - red2[-6:]).abs().max()) < 1e-6 * float(size.double().sum()) / 96 ** 3
    finally:
        cp.close()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("precision,n", [(0, 88), (0, 89), (1, 70), (1, 71)])   # 7.8 and 8.07 MB, 7.85 and 8.19 MB
def test_small_and_large_fields(precision, n, graph):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    w = _workload(2, n)
    cp = I.Coupler(w, precision=precision)
    try:
        assert (cp.G * (8 if precision else 4) <= 8 << 20) == (n in (88, 70))
        x, u = cp.nodes_to_device(w.x_local_all()), cp.zeros_grid()
        F, v, f, ref = cp.empty_nodes(), cp.empty_nodes(), cp.zeros_grid(), cp.zeros_grid()
        f.fill_(np.nan)
        torch.cuda.synchronize()
        _replayed(lambda s: I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, None, I.IFEM_SPREAD_OVERWRITE, s),
                  (lambda: f.fill_(np.nan)) if graph else None)
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F, ref, 0)
        I.ifem_sync_status(cp.ctx)
        assert torch.equal(f, ref)
    finally:
        cp.close()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("count", [3, 4])   # 7686 and 10248 nodes
def test_fp64_mls_order(count, graph):
    """Spread beside the interpolation and after it: the bits of the separate calls."""
    import torch
    from paper_1807_08219_gb300 import ifem as I
    w = _workload(count, 48)
    cp = I.Coupler(w, precision=I.IFEM_FP64, kernel=I.IFEM_KERNEL_MLS27, tile=6)
    try:
        g = torch.Generator(device=cp.device).manual_seed(1)
        u = torch.randn(cp.G, generator=g, device=cp.device, dtype=cp.dtype)
        x, f = cp.nodes_to_device(w.x_local_all()), cp.zeros_grid()
        F, v, F2, v2, f2 = cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes(), cp.zeros_grid()
        torch.cuda.synchronize()
        _replayed(lambda s: I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F, f, v, None, I.IFEM_SPREAD_OVERWRITE, s),
                  (lambda: [t.fill_(np.nan) for t in (F, v, f)]) if graph else None)
        I.ifem_compute_forces(cp.ctx, cp.batch, x, F2)
        I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, F2, f2, 0)
        I.ifem_interpolate(cp.ctx, cp.batch, cp.grid, u, x, v2)
        I.ifem_sync_status(cp.ctx)
        assert torch.equal(F, F2) and torch.equal(v, v2) and torch.equal(f, f2)
    finally:
        cp.close()
