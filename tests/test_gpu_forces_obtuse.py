"""FP32 membrane forces of meshes with obtuse triangles (up to 167 degrees, here by
stretching a sphere's reference shape: the nodal kernel's plain form, its form for
obtuse triangles, one particle to a cluster or to a block, and beyond it the general
path) and of strongly deformed ones: relative L2 against the oracle within 1.5 times
that of ifem_compute_forces_noalloc, which works in the reference triangle's plane."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from oracle import oracle as O
from tests._helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("law", ["nh", "skalak"])
@pytest.mark.parametrize("stretch,amp,copies", [(1.0, 0.1, 4), (1.0, 0.35, 4), (3.0, 0.1, 4), (6.0, 0.1, 4), (6.0, 0.3, 4),
                                                (12.0, 0.1, 4), (2.0, 0.1, 240), (6.0, 0.1, 240)])
def test_obtuse_triangles(law, stretch, amp, copies):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    rng = np.random.default_rng(4)
    X, f = M.icosphere(3 if copies < 9 else 2)
    t = C.Template("membrane", 0.1 * X * np.array([stretch, 1.0, 1.0]), f, law, mu=1.0, C=10.0)
    inst, ref = [], []
    for _ in range(copies):
        q = np.linalg.qr(rng.standard_normal((3, 3)))[0]
        x = (t.X @ (q @ (np.eye(3) + amp * rng.uniform(-1, 1, (3, 3)))).T).astype(np.float32).astype(np.float64)
        inst.append(C.Instance(0, 0, np.full(3, 0.5), x))
        ref.append(O.template_forces(t, x))
    cp = I.Coupler(W.Workload("obtuse", [t], inst, [W.Box(32, 1.0)], [], 0), precision=I.IFEM_FP32)
    try:
        x = cp.nodes_to_device(cp.wl.x_local_all())
        F, general = cp.empty_nodes(), cp.empty_nodes()
        I.ifem_compute_forces(cp.ctx, cp.batch, x, F)
        I.ifem_compute_forces_noalloc(cp.ctx, cp.batch, x, general)
        torch.cuda.synchronize()
        ref = np.concatenate(ref)
        assert rel_l2(cp.nodes_to_host(F), ref) < 1.5 * rel_l2(cp.nodes_to_host(general), ref)
    finally:
        cp.close()
