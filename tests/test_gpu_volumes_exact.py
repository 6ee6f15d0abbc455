"""FP32 contexts' volumes against the exact volume of the same FP32 positions (whole
numbers): within two units in the last place of an FP64 value (4.5e-16), where an FP64
evaluation of every element, summed in a fixed tree, leaves up to 2.5e-16 and float
pairs summed as pairs 3 to 15e-16. Meshes on both sides of the size from which the
elements are evaluated as float pairs, several deformations each, one batch."""
from fractions import Fraction

import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import meshes

pytestmark = pytest.mark.gpu


def _exact(x, el):
    """Volume of FP32 positions as a fraction."""
    m, e = np.frexp(x.astype(np.float64))
    low = int((e[x != 0] - 24).min())
    X = np.array([[int(v * 2.0 ** 24) << int(k - 24 - low) if v else 0 for v, k in zip(r, q)] for r, q in zip(m, e)], dtype=object)
    p = [X[el[:, c]] for c in range(el.shape[1])]
    if el.shape[1] == 4:
        p = [q - p[0] for q in p[1:]]
    t = [p[1][:, (a + 1) % 3] * p[2][:, (a + 2) % 3] - p[1][:, (a + 2) % 3] * p[2][:, (a + 1) % 3] for a in range(3)]
    return Fraction(int(sum((p[0][:, a] * t[a]).sum() for a in range(3)))) * Fraction(2) ** (3 * low) / 6


@pytest.mark.parametrize("size", [0.1, 3e-6])
def test_volumes_to_two_units(size):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    rng = np.random.default_rng(21)
    made = [meshes.icosphere(k) for k in (1, 2, 3, 4)] + [meshes.rbc_surface(4, 2.0)]
    made += [meshes.kuhn_ball(m, 1.0) for m in (3, 6, 9, 11, 13)]
    tms = [W.Template("membrane" if f.shape[1] == 3 else "solid", size * X, f, "nh", lam=1.0) for X, f in made]
    inst = []
    for k, t in enumerate(tms):
        for _ in range(5):
            q = np.linalg.qr(rng.standard_normal((3, 3)))[0] @ (np.eye(3) + 0.1 * np.diag(rng.standard_normal(3)))
            noise = 1e-3 * size * rng.standard_normal(t.X.shape) if t.kind == "membrane" else 0.0
            inst.append(W.Instance(k, 0, np.full(3, 0.5), (t.X @ q.T + noise).astype(np.float32).astype(np.float64)))
    cp = I.Coupler(W.Workload("volumes", tms, inst, [W.Box(32, 1.0)], [], 0), precision=I.IFEM_FP32)
    try:
        x = cp.nodes_to_device(cp.wl.x_local_all())
        vol = torch.empty(len(inst), dtype=torch.float64, device=cp.device)
        I.ifem_volumes(cp.ctx, cp.batch, x, vol)
        for i, got in zip(inst, vol.tolist()):
            want = _exact(i.x_local.astype(np.float32), tms[i.tmpl].elems)
            assert abs(float((Fraction(got) - want) / want)) < 4.5e-16, (tms[i.tmpl].n_elems, got)
    finally:
        cp.close()
