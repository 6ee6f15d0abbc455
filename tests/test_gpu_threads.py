"""Two contexts used from two threads at once, with batches of different sizes:
the dynamic shared memory a kernel may take belongs to the function, which the
contexts share, so no launch may lower it for another's (a launch that needs more
than is allowed is refused by the runtime). Each thread's results are those of the
same calls made alone, bit for bit."""
import threading

import numpy as np
import pytest

import ifem_workloads as W
from ifem_workloads import meshes

pytestmark = pytest.mark.gpu

CALLS = 4000


def _workload(m, copies):
    """Balls of m^3 nodes (18: 93 KB of positions, above the 48 KB a kernel may take unasked)."""
    X, t = meshes.kuhn_ball(m, 0.2)
    x = 1.02 * X
    return W.Workload("threads", [W.Template("solid", X, t, "nh", mu=1.0, lam=9.0)],
                      [W.Instance(0, 0, np.full(3, 0.3 + 0.2 * i), x) for i in range(copies)], [W.Box(40, 1.0)], [], m)


def _volumes(cp, stream):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    x = cp.nodes_to_device(cp.wl.x_local_all())
    vol = torch.zeros(len(cp.wl.instances), dtype=torch.float64, device=cp.device)
    return vol, lambda: I.ifem_volumes(cp.ctx, cp.batch, x, vol, stream)


def _spread(cp, stream):
    from paper_1807_08219_gb300 import ifem as I
    x, f = cp.nodes_to_device(cp.wl.x_local_all()), cp.zeros_grid()
    return f, lambda: I.ifem_spread(cp.ctx, cp.batch, cp.grid, x, x, f, I.IFEM_SPREAD_OVERWRITE, stream)


@pytest.mark.parametrize("call,precision,tiles", [(_volumes, 0, (16, 16)), (_spread, 1, (6, 12))])
def test_two_threads(call, precision, tiles):
    import torch
    from paper_1807_08219_gb300 import ifem as I
    cps = [I.Coupler(_workload(m, c), precision=precision, tile=t) for m, c, t in zip((8, 18), (2, 1), tiles)]
    try:
        streams = [torch.cuda.Stream() for _ in cps]
        made = [call(cp, s) for cp, s in zip(cps, streams)]
        ref = []
        torch.cuda.synchronize()
        for out, go in made:
            go()
            torch.cuda.synchronize()
            ref.append(out.clone())
        torch.cuda.synchronize()
        errors = []

        def work(i):
            try:
                for k in range(CALLS):
                    made[i][1]()
                    if k % 256 == 255:   # bounded queue
                        streams[i].synchronize()
            except Exception as e:   # reported in the test's own thread
                errors.append(e)

        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert not errors, errors
        for (out, _), r in zip(made, ref):
            assert bool((out == r).all())
    finally:
        for cp in cps:
            cp.close()
