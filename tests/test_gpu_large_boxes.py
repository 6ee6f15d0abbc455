"""The reproducible spread whose tiles' boxes take more memory than the three
lattices are given at once: it takes the lattices one after the other. The same
bits as two batches of half the particles each (which are small enough for all
three), the second added to what the first wrote; the halves share no value."""
import dataclasses

import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
def test_lattices_in_turn(kernel):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    n, k = 330, 4   # 55^3 tiles of 6 cells; 164 k nodes: 4.5 GB of boxes, halves 2.3
    X, f = meshes.icosphere(4)
    X = X * (12.3 / n)
    inst = [W.Instance(0, 0, (np.array([i % k, i // k % k, i // k ** 2]) + 0.43) / k, X) for i in range(k ** 3)]
    w = W.Workload("large", [W.Template("membrane", X, f, "nh")], inst, [W.Box(n, 1.0)], [], 0)
    out = []
    for groups in ([inst], [inst[::2], inst[1::2]]):
        field, v = None, []
        for group in groups:
            cp = I.Coupler(dataclasses.replace(w, instances=group), precision=I.IFEM_FP32, kernel=kernel, tile=6)
            try:
                g = torch.Generator(device=cp.device).manual_seed(9)
                u = torch.randn(cp.G, generator=g, device=cp.device)
                x = cp.nodes_to_device(cp.wl.x_local_all() * 1.07)
                F, vg = cp.empty_nodes(), cp.empty_nodes()
                first = field is None
                field = torch.full((cp.G,), 3.0, device=cp.device) if first else field
                I.ifem_step_coupling(cp.ctx, cp.batch, cp.grid, x, u, F, field, vg, None, I.IFEM_SPREAD_OVERWRITE if first else 0)
                I.ifem_sync_status(cp.ctx)
                v.append(vg.cpu())
            finally:
                cp.close()
        out.append((field, v))
    assert bool((out[0][0] == out[1][0]).all()) and int((out[0][0] != 0).sum()) > 1_000_000
    whole, halves = out[0][1][0].view(3, k ** 3, -1), out[1][1]
    assert torch.equal(whole[:, ::2].reshape(3, -1), halves[0]) and torch.equal(whole[:, 1::2].reshape(3, -1), halves[1])
