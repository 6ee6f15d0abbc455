"""FP32 forces gathered per node, at the sizes where the kernel's layout can go
wrong: fewer nodes than a warp, chunks of a cluster that end early or hold
nothing, templates at and beyond the shared-memory limit, shuffled node orders,
open and non-manifold surfaces, batches on every side of the cluster rule.
Compared with the FP64 oracle on the same rounded positions: relative L2 1e-5
(the FP32 force tolerance) or, where the forces themselves are ill-conditioned
in FP32 (bending of a fine smooth mesh: kH^2 - kG cancels), 1.5 times the error
of the general path (element buffer and nodal sum, ifem_compute_forces_noalloc);
and required to be identical from run to run."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from oracle import oracle as O
from tests._helpers import rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-5


def _shuffled(X, el, seed):
    p = np.random.default_rng(seed).permutation(len(X))
    inv = np.empty_like(p)
    inv[p] = np.arange(len(p))
    return X[p], inv[el].astype(np.int32)


def _membrane(kind, law):
    level = {"icosa": 0, "level1": 1, "level4": 4, "level5": 5, "level6": 6}.get(kind, 3)
    X, f = M.icosphere(level)
    if kind == "open":        # a patch: rings that do not close
        f = f[X[f].mean(1)[:, 2] > 0.2]
    if kind == "touching":    # two spheres sharing node 0: two fans at one node
        f2 = f + len(X)
        f2[f == 0] = 0
        X, f = np.concatenate([X, 2 * X[:1] - X]), np.concatenate([f, f2[:, [0, 2, 1]]]).astype(np.int32)
    X, f = _shuffled(0.1 * X, f, level + 3)
    kb = 0.0 if kind in ("open", "touching") else 2e-3
    return C.Template("membrane", X, f, law, mu=1.0, C=5.0, kb=kb)


def _solid(m):
    t = C.ball_template(m, 0.1)
    t.X, t.elems = _shuffled(t.X, t.elems, m)
    return t


def _check(templates, seed=0):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    rng = np.random.default_rng(seed)
    inst, ref = [], []
    for k, t in enumerate(templates):
        # a homogeneous stretch and a smooth wave: no element inverts
        x = t.X @ (np.eye(3) + 0.1 * rng.uniform(-1, 1, (3, 3))).T
        x = (x + 2e-3 * np.sin(20.0 * t.X @ rng.standard_normal(3))[:, None]).astype(np.float32).astype(np.float64)
        inst.append(C.Instance(k, 0, np.full(3, 0.5), x))
        ref.append(O.template_forces(t, x))
    w = W.Workload("nodal", list(templates), inst, [W.Box(32, 1.0)], [], seed)
    cp = I.Coupler(w, precision=I.IFEM_FP32)
    try:
        x = cp.nodes_to_device(w.x_local_all())
        F, again, general = cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes()
        I.ifem_compute_forces(cp.ctx, cp.batch, x, F)
        I.ifem_compute_forces(cp.ctx, cp.batch, x, again)
        I.ifem_compute_forces_noalloc(cp.ctx, cp.batch, x, general)
        I.ifem_sync_status(cp.ctx)
        assert torch.equal(F, again)
        g, gen, at = cp.nodes_to_host(F), cp.nodes_to_host(general), 0
        for t, r in zip(templates, ref):
            mine = slice(at, at + t.n_nodes)
            assert rel_l2(g[mine], r) < max(TOL, 1.5 * rel_l2(gen[mine], r)), (t.kind, t.n_nodes)
            at += t.n_nodes
    finally:
        cp.close()


@pytest.mark.parametrize("law", ["nh", "skalak"])
@pytest.mark.parametrize("kind", ["icosa", "level1", "level3", "level4", "open", "touching"])
def test_membranes(kind, law):
    _check([_membrane(kind, law)])


@pytest.mark.parametrize("kind", ["level5", "level6"])   # 10242 nodes fit shared memory, 40962 take the general path
def test_large_membranes(kind):
    _check([_membrane(kind, "skalak")])


@pytest.mark.parametrize("m", [2, 3, 5, 16, 26])   # 26: 17576 nodes, the general path
def test_solids(m):
    _check([_solid(m)])


@pytest.mark.parametrize("count", [9, 10, 76, 77, 228, 229])   # both sides of the cluster rule of a 152-SM GPU
def test_mixed_batches(count):
    kinds = [_membrane("level1", "nh"), _solid(3), _membrane("level3", "skalak"), _solid(5), _membrane("icosa", "nh")]
    _check([kinds[k % 5] for k in range(count)])


def test_inverted_tets_are_counted_once():
    import torch
    from paper_1807_08219_gb300 import ifem as I
    t = _solid(5)
    w = W.Workload("inverted", [t], [C.Instance(0, 0, np.full(3, 0.5), t.X)], [W.Box(32, 1.0)], [], 0)
    cp = I.Coupler(w, precision=I.IFEM_FP32)
    try:
        x = cp.nodes_to_device(t.X * np.array([1.0, 1.0, -1.0]))   # mirrored: every tet inverted
        I.ifem_compute_forces(cp.ctx, cp.batch, x, cp.empty_nodes())
        rc, st = I.ifem_sync_status(cp.ctx, raise_on_error=False)
        assert st["inverted_elements"] == t.n_elems
    finally:
        cp.close()
