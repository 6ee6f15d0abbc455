"""The FP64 spread's units: tiles with short candidate lists walked by one warp,
long ones by eight (an octant each), candidates that miss a unit left out, points
dealt to lanes; boxes of one tile, where a stencil comes back through the opposite
face; remainders. F, f and v are the oracle's bit for bit, as in the other FP64
tests, and so are two runs' sums; a box's sum of what it received agrees with the
field's to rounding (1e-12 of the sum of its terms' sizes)."""
import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import configs as C
from ifem_workloads import meshes as M
from tests._helpers import oracle_step, random_grid, run_gpu_step

pytestmark = pytest.mark.gpu


def _workload(ns, level, radius, parts, seed):
    """Boxes of ns cells, `parts` icospheres of `radius` cells in each: every list of a small box is long at level 4."""
    rng = np.random.default_rng(seed)
    boxes = [W.Box(n, n / 32.0) for n in ns]
    X, f = M.icosphere(level)
    tm = C.Template("membrane", radius / 32 * X, f, "nh")
    inst = [C.Instance(0, b, rng.uniform(-0.2, 1.2, 3) * box.L, tm.X + 0.01 / 32 * rng.standard_normal(tm.X.shape))
            for b, box in enumerate(boxes) for _ in range(parts)]
    return W.Workload("dense", [tm], inst, boxes, [rng.standard_normal((3, n, n, n)) for n in ns], seed)


@pytest.mark.parametrize("tile", [6, 8, 11, 12, 16])
@pytest.mark.parametrize("level,parts", [(0, 1), (2, 3), (4, 1)])
@pytest.mark.parametrize("ns", [(8,), (9, 13), (16,), (18, 33)])
def test_spread_bit_exact(ns, level, parts, tile):
    w = _workload(ns, level, 3.0, parts, seed=sum(ns) + tile)
    f0 = random_grid(w, seed=3)
    g, again = (run_gpu_step(w, 1, tile=tile, f0=f0) for _ in range(2))
    o = oracle_step(w, f0=f0)
    assert g["rc"] == 0, g["stats"]
    assert np.array_equal(g["F"], o["F"]) and np.array_equal(g["v"], o["v"])
    assert np.array_equal(g["red"], again["red"])
    red = g["red"][12 * len(w.instances):].reshape(-1, 6)
    for b, (got, want, start) in enumerate(zip(g["f"], o["f"], f0)):
        assert np.array_equal(got, want), np.abs(got - want).max()
        h3 = (w.boxes[b].L / w.boxes[b].n) ** 3
        d = (got - start).reshape(3, -1)
        assert (np.abs(red[b, :3] - h3 * d.sum(1)) <= 1e-12 * h3 * (np.abs(d) + np.abs(start.reshape(3, -1))).sum(1)).all()
