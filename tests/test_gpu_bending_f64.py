"""FP64 bending from values kept per triangle: valences up to 96 (the product of
(cot + i) over a vertex's corners is rescaled), obtuse corners at every place of a
triangle, meshes far from unit size, several templates of one launch with and
without bending. Forces against the oracle, relative L2: 1e-12, from up to 96
factors with cotangents up to 31, each with a few roundings."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from tests._helpers import oracle_step, rel_l2, run_gpu_step

pytestmark = pytest.mark.gpu


def _bipyramid(m, height):
    """Two apexes over a ring of m vertices: valence m; flat (obtuse corners) or tall (slivers)."""
    a = 2 * np.pi * np.arange(m) / m
    X = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, height], [0, 0, -height]]])
    k, n = np.arange(m), (np.arange(m) + 1) % m
    el = np.concatenate([np.stack([k, n, 0 * k + m], 1), np.stack([n, k, 0 * k + m + 1], 1)])
    return X, np.stack([np.roll(t, i % 3) for i, t in enumerate(el)]).astype(np.int32)   # every corner first in turn


@pytest.mark.parametrize("size", [1e-4, 0.1, 0.4])
@pytest.mark.parametrize("m,height", [(4, 1.0), (7, 0.2), (32, 0.5), (96, 1.0)])
def test_bending_forces(m, height, size):
    X, el = _bipyramid(m, height)
    rng = np.random.default_rng(m)
    tms = [C.Template("membrane", size * X, el, "nh", kb=1e-3, name="fan"),
           C.Template("membrane", size * M.icosphere(2)[0], M.icosphere(2)[1], "nh", name="no bending"),
           C.Template("membrane", size * M.icosphere(1)[0], M.icosphere(1)[1], "skalak", kb=1e-2, name="sphere")]
    box = W.Box(16, 1.0)
    inst = [C.Instance(t, 0, rng.uniform(0, 1, 3), tms[t].X * (1 + 0.02 * rng.standard_normal(tms[t].X.shape)))
            for t in (0, 1, 2, 0)]
    w = W.Workload("bend", tms, inst, [box], [np.zeros((3, 16, 16, 16))], m)
    g, o = run_gpu_step(w, 1, tile=8), oracle_step(w)
    at = 0
    for i in inst:   # each particle by itself: their forces differ in size
        k = len(tms[i.tmpl].X)
        assert rel_l2(g["F"][at:at + k], o["F"][at:at + k]) < 1e-12, tms[i.tmpl].name
        at += k
