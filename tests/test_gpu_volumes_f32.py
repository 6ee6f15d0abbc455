"""Volumes and the volume correction of FP32 positions in float pairs, where they
can lose what FP64 keeps: particles far from their local origin, tiny and huge
units, a few nodes, open meshes, templates beyond shared memory (general path).
Volumes against the FP64 oracle on the same rounded positions: an FP64
evaluation of the same sums is allowed 8 ulp of the summed magnitudes; 1e-12 of
the volume where that is larger (the tolerance of the existing volume test)."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _run(tms, xs, V0=None):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    inst = [C.Instance(k, 0, np.full(3, 0.5), x) for k, x in enumerate(xs)]
    w = W.Workload("volumes", list(tms), inst, [W.Box(32, 1.0)], [], 0)
    cp = I.Coupler(w, precision=I.IFEM_FP32)
    try:
        x = cp.nodes_to_device(w.x_local_all())
        vol = torch.empty(len(xs), dtype=torch.float64, device=cp.device)
        I.ifem_volumes(cp.ctx, cp.batch, x, vol)
        if V0 is None:
            return vol.cpu().numpy()
        I.ifem_volume_correct(cp.ctx, cp.batch, x, torch.as_tensor(V0, dtype=torch.float64, device=cp.device))
        I.ifem_sync_status(cp.ctx)
        return cp.nodes_to_host(x)
    finally:
        cp.close()


def _membrane(level, size, open_=False):
    X, f = M.rbc_surface(level, 2.0 * size)
    if open_:
        f = f[: len(f) // 2]
    return C.Template("membrane", X, f, "nh")


def _magnitude(el, x):
    a, b, c = (np.linalg.norm(x[el[:, k]], axis=1) for k in range(3))
    return float((a * b * c).sum()) / 6.0


@pytest.mark.parametrize("size", [1e-9, 0.06, 1e7])
@pytest.mark.parametrize("shift", [0.0, 3.0, 40.0])
def test_volumes(size, shift):
    rng = np.random.default_rng(1)
    tms = [_membrane(0, size), _membrane(2, size), _membrane(4, size), _membrane(3, size, open_=True),
           C.ball_template(2, size), C.ball_template(9, size)]
    xs = []
    for t in tms:
        x = t.X @ (np.eye(3) + 0.1 * rng.uniform(-1, 1, (3, 3))).T + shift * size * rng.uniform(-1, 1, 3)
        xs.append(x.astype(np.float32).astype(np.float64))
    got = _run(tms, xs)
    for t, x, g in zip(tms, xs, got):
        ref = O.volume(t.elems, x) if t.kind == "membrane" else O.tet_volume(t.elems, x)
        mag = _magnitude(t.elems, x) if t.kind == "membrane" else abs(ref)
        assert abs(g - ref) <= max(1e-12 * abs(ref), 8 * 2.0 ** -53 * mag), (t.kind, t.n_nodes)


@pytest.mark.parametrize("level", [1, 4, 5])   # 10242 nodes: the correction's general path
@pytest.mark.parametrize("size", [1e-9, 0.06])
def test_correction_meets_the_volume(level, size):
    t = _membrane(level, size)
    x = (t.X * 1.01).astype(np.float32).astype(np.float64)
    V0 = O.volume(t.elems, t.X)
    y = _run([t], [x], [V0])
    ref, _, _ = O.volume_correction(t.elems, x, V0)
    # positions to 2e-7 of the extent, the FP32 tolerance of the existing correction test
    assert np.abs(y - ref).max() <= 2e-7 * np.abs(ref).max()
    assert O.volume(t.elems, y) == pytest.approx(V0, rel=2e-6)
