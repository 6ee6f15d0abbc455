"""Measured cases of the coupling library: what a program built on it calls, through the public
entry points of ``paper_1807_08219_gb300`` (the C ABI's Python binding and the autograd operators).

A case is a dict of plain values:
  path       step       one coupling step (forces, spread, interpolation), device arrays
             step_ab2   the step with the position update in the same call
             step_host  the step for a caller whose node arrays live in pinned host memory
             transfer   spread and interpolation with their gradients (torch.autograd)
             elastic    elastic forces with their gradient (torch.autograd)
             fluid      solids in a viscoelastic fluid: velocity and conformation at the nodes,
                        elastic + fluid-stress forces, spread
             update     the Lagrangian end of a time step: position update, membrane volume
                        correction, volumes, indicator source
  mix        particle types: capsule642, capsule2562, rbc, blood (red cells and platelets 5:1),
             solid (tetrahedral balls), mixed (all of them)
  n, boxes   cells per side of the box; boxes > 1: that many boxes of 32 .. n cells
  particles  particles in all (boxes > 1: at most, over all boxes)
  d          particle diameter in cells
  precision  fp32 | fp64;  kernel: peskin4 | mls27;  scatter: det | atomic (ignored in fp64)
  sums       whether the step also returns the conservation sums

Particle shapes, material constants and velocity modes are those of the seeded workloads in
``ifem_workloads``; particles sit on a jittered lattice in random orientations, so that making a
suspension takes milliseconds.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import ifem_workloads.configs as W
import ifem_workloads.meshes as M
from paper_1807_08219_gb300 import autograd as AG
from paper_1807_08219_gb300 import ifem as I

ETA, BETA, RELAX = 1.0, 0.5, 0.5   # fluid viscosity, viscosity ratio, polymer relaxation time
N_MODES, AMPLITUDE = 8, 0.1        # velocity modes


def _case(path, mix, n, particles, d, precision="fp32", kernel="peskin4", scatter="det", sums=False, boxes=1, name=None):
    c = {"path": path, "mix": mix, "n": n, "boxes": boxes, "particles": particles, "d": float(d),
         "precision": precision, "kernel": kernel, "scatter": scatter, "sums": sums}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one capsule in a small box, time-stepped: the smallest call, all launches and latency
        _case("step_ab2", "capsule642", 64, 1, 20, name="capsule_step_ab2"),
        # one red cell in shear, the usual validation run, the fast scatter
        _case("step", "rbc", 128, 1, 20, scatter="atomic", name="one_rbc_step"),
        # a small suspension with the library's default configuration (reproducible FP32)
        _case("step", "blood", 128, 72, 26, name="blood72_step_default"),
        # the headline workload: 500 red cells and 100 platelets in production
        _case("step", "blood", 256, 600, 32.28, scatter="atomic", name="blood600_step"),
        # the same suspension driven by a flow solver on the host
        _case("step_host", "blood", 256, 600, 32.28, scatter="atomic", name="blood600_step_host"),
        # a parameter study: many independent boxes of uneven size in one call
        _case("step", "mixed", 96, 630, 20, scatter="atomic", boxes=64, name="boxes64_step"),
        # the FP64 reference run of a suspension, bit-reproducible and monitored by its conservation sums
        _case("step", "blood", 120, 60, 24, precision="fp64", sums=True, name="blood60_step_fp64"),
        # the paper's own kernel (linear moving least squares), odd box
        _case("step", "blood", 101, 48, 20, kernel="mls27", name="blood48_step_mls"),
        # differentiable coupling (control, parameter fitting): both transfers and their transposes
        _case("transfer", "rbc", 150, 120, 24, scatter="atomic", name="rbc120_transfer_grad"),
        # parameter fitting of solids: elastic forces and the Hessian-vector product behind their gradient
        _case("elastic", "solid", 96, 16, 24, name="solid16_elastic_grad"),
        # deformable solids in a viscoelastic fluid
        _case("fluid", "solid", 160, 64, 24, name="solid64_fluid"),
        # end of a time step of large capsules: update, volume correction, volumes, indicator source
        _case("update", "capsule2562", 192, 200, 28, scatter="atomic", name="capsule200_update"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    path = rng.choice(["step", "step", "step", "step_ab2", "step_host", "transfer", "elastic", "fluid", "update"])
    precision = "fp64" if rng.random() < 0.2 else "fp32"
    kernel = "mls27" if path in ("step", "step_ab2") and rng.random() < 0.25 else "peskin4"
    scatter = rng.choice(["det", "atomic"])
    slow = precision == "fp64" or kernel == "mls27"   # costlier paths: smaller suspensions
    n = round(_log(rng, 32, 128 if slow else 256))
    sums = path in ("step", "step_host") and precision == "fp64" and rng.random() < 0.6   # monitored reference runs
    if path in ("step", "step_ab2") and rng.random() < 0.2:
        boxes = rng.randint(2, 4 if slow else 64)
        return _case(path, "mixed", min(max(n, 40), 64 if slow else 96), 8 * boxes, 20, precision, kernel, scatter, sums, boxes)
    d = round(rng.uniform(16.0, min(33.0, n / 1.6)), 2)
    mix = {"elastic": rng.choice(["solid", "capsule2562"]), "fluid": "solid",
           "update": rng.choice(["capsule642", "capsule2562", "rbc"])}.get(
        path, rng.choice(["capsule642", "capsule2562", "rbc", "blood", "blood", "solid"]))
    most = (8 if precision == "fp64" and kernel == "mls27" else 60) if slow else {"blood": 600, "solid": 64}.get(mix, 480)
    if path in ("elastic", "fluid", "update"):
        most = min(most, 64 if mix == "solid" else 200)
    particles = round(_log(rng, 1, max(1, min(most, _sites(n, d) ** 3))))
    return _case(path, mix, n, particles, d, precision, kernel, scatter, sums)


# ---------------------------------------------------------------- inputs
def _sites(n, d):
    """Lattice sites per axis for particles of d cells in n cells."""
    return max(1, int(n / (0.88 * d)))


@functools.lru_cache(maxsize=None)
def _templates(mix, d, h, bending):
    D, R = d * h, 0.48 * d * h
    m = min(16, max(8, round(0.65 * d)))

    def capsule(level):
        X, f = M.icosphere(level)
        kb = W.KAPPA_B_HAT * R if level == 4 and bending else 0.0
        return W.Template("membrane", R * X, f, "nh", mu=1.0, kb=kb)

    if mix == "capsule642":
        return (capsule(3),)
    if mix == "capsule2562":
        return (capsule(4),)
    if mix == "rbc":
        return (W.rbc_template(D),)
    if mix == "solid":
        return (W.ball_template(m, 0.5 * D),)
    if mix == "blood":
        a = 0.1875 * D
        mu = 1.0 / (W.CA_PLT_OVER_CA_RBC * a)
        return (W.rbc_template(D), W.ball_template(8, a, mu=mu, semi_axes=np.array([a, a, 0.5 * a]),
                                                   lam=W.PLT_LAMBDA_OVER_MU * mu))
    return (capsule(3), capsule(4), W.rbc_template(D)) + tuple(W.ball_template(k, 0.5 * (k - 1) * h) for k in range(8, 16))


def _layout(case):
    """Boxes and (template, box, site) of every particle: fixed by the case, the same for every seed."""
    rng = np.random.default_rng([case["n"], case["boxes"], case["particles"]])
    if case["boxes"] == 1:
        boxes = [W.Box(case["n"], 1.0)]
        k = _sites(case["n"], case["d"])
        p = min(case["particles"], k ** 3)
        sites = rng.choice(k ** 3, size=p, replace=False)
        tm = [0] * p
        if case["mix"] == "blood":
            tm = [0] * (p - p // 6) + [1] * (p // 6)
        return boxes, [(t, 0, s, k) for t, s in zip(tm, sites)]
    h = 1.0 / 64
    boxes = [W.Box(int(n), int(n) * h) for n in rng.integers(32, case["n"] + 1, size=case["boxes"])]
    parts = []
    for b, box in enumerate(boxes):
        k = _sites(box.n, case["d"] * 1.25)
        count = min(int(rng.integers(1, 21)), k ** 3, max(1, case["particles"] - len(parts)))
        for s in rng.choice(k ** 3, size=count, replace=False):
            typ = int(rng.integers(0, 4))
            parts.append((typ if typ < 3 else int(rng.integers(3, 11)), b, s, k))
    return boxes, parts


def _rotations(rng, count):
    q, r = np.linalg.qr(rng.standard_normal((count, 3, 3)))
    q = q * np.sign(np.diagonal(r, axis1=1, axis2=2))[:, None, :]
    q[np.linalg.det(q) < 0, :, 0] *= -1.0
    return q


def _modes(rng):
    k = rng.integers(-4, 5, size=(N_MODES, 3)).astype(float)
    k[~k.any(axis=1), 0] = 1.0
    e = rng.standard_normal((N_MODES, 3))
    e -= (e * k).sum(1, keepdims=True) * k / (k * k).sum(1, keepdims=True)
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    return k, AMPLITUDE * e, rng.uniform(0.0, 2.0 * np.pi, N_MODES)


def _sample(k, amp, ph, n, o, dev):
    """sum_m amp_m cos(2 pi k_m.(i + o)/n + ph_m) on an n^3 lattice, FP64."""
    t = torch.arange(n, dtype=torch.float64, device=dev)
    ax = [2.0 * math.pi * torch.as_tensor(k[:, a], device=dev)[:, None] * (t + o[a])[None, :] / n for a in range(3)]
    zy = (ax[2][:, :, None] + ax[1][:, None, :] + torch.as_tensor(ph, device=dev)[:, None, None]).reshape(len(k), -1)
    w = torch.as_tensor(amp, device=dev)[:, None]
    left = torch.cat([w * torch.cos(zy), -w * torch.sin(zy)]).T
    return (left @ torch.cat([torch.cos(ax[0]), torch.sin(ax[0])])).reshape(-1)


def _at_nodes(modes, p, L):
    """The velocity modes at points p (3, N) of boxes of side L (N)."""
    k, e, ph = (torch.as_tensor(q, device=p.device) for q in modes)
    return (e.T[:, :, None] * torch.cos(2.0 * math.pi * (k @ (p / L)) + ph[:, None])[None]).sum(1)


class _Inputs:
    """Everything a program has in hand for a case: the same for the library and for exact()."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([seed, 17])
        self.dev = dev = torch.device("cuda", torch.cuda.current_device())
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(rng.integers(1 << 40)))
        self.dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        boxes, parts = _layout(case)
        h = boxes[0].h
        path = case["path"]
        tms = _templates(case["mix"], case["d"], h, path != "elastic")
        parts.sort(key=lambda q: q[0])
        nn = np.array([tms[q[0]].n_nodes for q in parts])
        self.off = np.concatenate([[0], np.cumsum(nn)])
        N = int(self.off[-1])
        rot = _rotations(rng, len(parts))
        site = np.array([[q[2] % q[3], q[2] // q[3] % q[3], q[2] // q[3] ** 2] for q in parts], dtype=float)
        Ls, ks = np.array([boxes[q[1]].L for q in parts]), np.array([q[3] for q in parts])
        origin = (site + 0.5 + 0.1 * rng.uniform(-1, 1, site.shape)) * (Ls / ks)[:, None]
        # membranes: stretch along the body axes and positional noise; solids: a small affine map
        # and a smooth wave, which keep their thin tets upright
        S = np.eye(3) + np.stack([np.diag(0.1 * rng.standard_normal(3)) if tms[q[0]].kind == "membrane"
                                  else 0.05 * rng.uniform(-1, 1, (3, 3)) for q in parts])
        A = torch.as_tensor(rot @ S, device=dev)
        wave = rng.standard_normal((len(parts), 3))
        wave = torch.as_tensor(wave / np.linalg.norm(wave, axis=1, keepdims=True), device=dev)
        x = torch.empty((3, N), dtype=torch.float64, device=dev)
        for t, tm in enumerate(tms):
            mine = [i for i, q in enumerate(parts) if q[0] == t]
            if not mine:
                continue
            X = torch.as_tensor(tm.X, device=dev)
            y = A[mine] @ X.T   # (instances, 3, nodes)
            if tm.kind == "membrane":
                noise = torch.randn(y.shape, dtype=y.dtype, device=dev, generator=gen)
                y += 1e-3 * case["d"] * h * (0.1 if boxes[1:] else 1.0) * noise
            else:
                phase = (X @ wave[mine][:, :, None]).mT * (math.pi / (0.5 * case["d"] * h))   # (instances, 1, nodes)
                y += 0.2 * h * wave[mine][:, :, None] * torch.sin(phase)
            a, b = int(self.off[mine[0]]), int(self.off[mine[-1] + 1])
            x[:, a:b] = y.permute(1, 0, 2).reshape(3, -1)
        self.x = x.to(self.dtype).contiguous()
        self.wl = W.Workload("case", list(tms), [W.Instance(q[0], q[1], origin[i], None) for i, q in enumerate(parts)], boxes, [], seed)
        self.N, self.origin = N, origin
        per_node = np.repeat(np.arange(len(parts)), nn)
        self.inst = torch.as_tensor(per_node, device=dev)
        L = torch.as_tensor(Ls, device=dev)[self.inst]
        p = torch.as_tensor(origin, device=dev).T[:, self.inst] + self.x.double()
        modes = _modes(rng)
        if path not in ("elastic", "update"):
            self.u = self._grid(boxes, modes)
        if path in ("step_ab2", "update"):
            self.dt = 0.3 * h / AMPLITUDE
            self.v = _at_nodes(modes, p, L).to(self.dtype)
            self.vp = _at_nodes((modes[0], modes[1], modes[2] + 0.05), p, L).to(self.dtype)
        if path == "update":
            self.V0 = _volumes(self, self.x.double())
        if path == "transfer":
            scale = 1.0 + torch.rand((3, N), dtype=torch.float64, device=dev, generator=gen)
            self.F = (scale * _at_nodes((modes[0], modes[1], modes[2] + 1.0), p, L)).to(self.dtype)
            self.gf = self._grid(boxes, _modes(rng))
            self.gv = _at_nodes(_modes(rng), p, L).to(self.dtype)
        if path == "elastic":
            self.gF = _at_nodes(modes, p, L).to(self.dtype)
        if path == "fluid":
            k, ph = modes[0], modes[2]
            w = 0.05 * rng.standard_normal((6, N_MODES))
            out = []
            for bx in boxes:
                for q in range(6):
                    out.append((q < 3) + _sample(k, w[q], ph, bx.n, (0.5, 0.5, 0.5), dev))
            self.C = torch.cat(out).to(self.dtype)

    def _grid(self, boxes, modes):
        k, e, ph = modes
        out = []
        for bx in boxes:
            for d in range(3):
                o = [0.0 if a == d else 0.5 for a in range(3)]
                out.append(_sample(k, e[:, d], ph, bx.n, o, self.dev).to(self.dtype))
        return torch.cat(out)


class _State:
    pass


def prepare(case, seed):
    q = _Inputs(case, seed)
    s = _State()
    s.path, s.q = case["path"], q
    s.cp = cp = I.Coupler(q.wl, precision=I.IFEM_FP64 if case["precision"] == "fp64" else I.IFEM_FP32,
                          kernel=I.IFEM_KERNEL_MLS27 if case["kernel"] == "mls27" else I.IFEM_KERNEL_PESKIN4,
                          scatter=I.IFEM_SCATTER_ATOMIC if case["scatter"] == "atomic" else I.IFEM_SCATTER_DET,
                          device=q.dev.index)
    I.ifem_prepare(cp.ctx, cp.batch, q.x)
    s.F, s.v, s.xn = cp.empty_nodes(), cp.empty_nodes(), cp.empty_nodes()
    if s.path in ("step", "step_ab2", "step_host", "fluid", "update"):
        s.f = cp.zeros_grid()
    n_red = 12 * len(q.wl.instances) + 6 * len(q.wl.boxes)
    s.red = torch.zeros(n_red, dtype=torch.float64, device=q.dev) if case["sums"] else None
    if s.path == "step_host":
        s.x_host = q.x.cpu().pin_memory()
        s.v_host = torch.empty(s.v.shape, dtype=s.v.dtype).pin_memory()
        s.red_host = torch.empty(n_red, dtype=torch.float64).pin_memory() if case["sums"] else None
        s.x = torch.empty_like(q.x)
    if s.path == "transfer":
        s.Fr, s.ur = q.F.clone().requires_grad_(), q.u.clone().requires_grad_()
    if s.path == "elastic":
        s.xr = q.x.clone().requires_grad_()
    if s.path == "fluid":
        s.Cn = torch.empty((6, q.N), dtype=q.dtype, device=q.dev)
    if s.path == "update":
        s.lam, s.vol = torch.empty_like(q.V0), torch.empty_like(q.V0)
    torch.cuda.synchronize()
    return s


def run(s):
    q, cp = s.q, s.cp
    c, b, g, over = cp.ctx, cp.batch, cp.grid, I.IFEM_SPREAD_OVERWRITE
    if s.path == "step":
        I.ifem_step_coupling(c, b, g, q.x, q.u, s.F, s.f, s.v, s.red, over)
        return {"F": s.F, "f": s.f, "v": s.v, "red": s.red}
    if s.path == "step_ab2":
        I.ifem_step_coupling_ab2(c, b, g, q.x, q.u, s.F, s.f, s.v, s.red, over, q.vp, q.dt, s.xn)
        return {"F": s.F, "f": s.f, "v": s.v, "x": s.xn, "red": s.red}
    if s.path == "step_host":
        I.ifem_step_coupling_host(c, b, g, s.x_host, s.x, q.u, s.F, s.f, s.v, s.v_host, s.red, s.red_host, over)
        return {"F": s.F, "f": s.f, "v": s.v_host, "red": s.red_host}
    if s.path == "transfer":
        f = AG.spread(s.Fr, q.x, cp)
        v = AG.interpolate(s.ur, q.x, cp)
        gF, gu = torch.autograd.grad([f, v], [s.Fr, s.ur], [q.gf, q.gv])
        return {"f": f.detach(), "v": v.detach(), "gF": gF, "gu": gu}
    if s.path == "elastic":
        F = AG.elastic_forces(s.xr, cp)
        (gx,) = torch.autograd.grad(F, s.xr, q.gF)
        return {"F": F.detach(), "gx": gx}
    if s.path == "fluid":
        I.ifem_interpolate(c, b, g, q.u, q.x, s.v)
        I.ifem_interpolate_cc(c, b, g, q.C, 6, q.x, s.Cn)
        I.ifem_compute_forces(c, b, q.x, s.F)
        I.ifem_fluid_stress_forces(c, b, q.x, s.v, s.Cn, ETA, BETA, RELAX, s.F, I.IFEM_FORCES_ACCUMULATE)
        I.ifem_spread(c, b, g, q.x, s.F, s.f, over)
        return {"v": s.v, "C": s.Cn, "F": s.F, "f": s.f}
    s.xn.copy_(q.x)
    I.ifem_ab2_update(c, b, s.xn, q.v, q.vp, q.dt)
    I.ifem_volume_correct(c, b, s.xn, q.V0, s.lam)
    I.ifem_volumes(c, b, s.xn, s.vol)
    I.ifem_indicator_source(c, b, g, s.xn, s.f, over)
    return {"x": s.xn, "lam": s.lam, "vol": s.vol, "G": s.f}


# ---------------------------------------------------------------- work
def work(case):
    """Node arrays and grid fields read and written once; touched grid values by the shells of the
    particles (about 15 per node over the three lattices, at most all of them)."""
    boxes, parts = _layout(case)
    tms = _templates(case["mix"], case["d"], boxes[0].h, case["path"] != "elastic")
    rs = 8 if case["precision"] == "fp64" else 4
    N = sum(tms[q[0]].n_nodes for q in parts)
    E3 = sum(tms[q[0]].n_elems for q in parts if tms[q[0]].kind == "membrane")
    E4 = sum(tms[q[0]].n_elems for q in parts if tms[q[0]].kind == "solid")
    G = sum(3 * bx.n ** 3 for bx in boxes)
    T = min(G, 15 * N)
    points = 27 if case["kernel"] == "mls27" else 64
    transfer = 2 * 3 * points * 2 * N
    forces = 130 * E3 + 400 * E4 + 600 * sum(tms[q[0]].n_nodes for q in parts if tms[q[0]].kb)
    node = rs * 3 * N
    path = case["path"]
    if path in ("step", "step_ab2", "step_host"):   # x, F, v; u read where touched, f written whole
        extra = {"step": 0, "step_ab2": 2 * node, "step_host": 2 * node}[path]
        return {"bytes": 3 * node + rs * (T + G) + extra, "flops": transfer + forces}
    if path == "transfer":   # f and gu written whole, gf and u read where touched; x, F, gv, v, gF
        return {"bytes": 5 * node + 2 * rs * (T + G), "flops": 2 * transfer}
    if path == "elastic":    # x, F, direction, gradient
        return {"bytes": 4 * node, "flops": 3 * forces}
    if path == "fluid":      # x, v, C (2 node arrays), F; u and C read where touched, f written
        return {"bytes": 5 * node + rs * (T + 2 * T + G), "flops": 2 * transfer + 2 * forces}
    return {"bytes": 4 * node + rs * G, "flops": transfer // 2 + 400 * E3}   # x read and written, v, vp; G


# ---------------------------------------------------------------- 64-bit values
def _groups(q, kinds=("membrane", "solid")):
    """(template, its instances, their nodes (instances, n_nodes)) of an _Inputs."""
    for t, tm in enumerate(q.wl.templates):
        mine = [i for i, it in enumerate(q.wl.instances) if it.tmpl == t]
        if mine and tm.kind in kinds:
            nodes = torch.as_tensor(q.off[:-1][mine], device=q.dev)[:, None] + torch.arange(tm.n_nodes, device=q.dev)
            yield tm, mine, nodes


def _corner(y, el, c):
    return y[:, torch.as_tensor(el[:, c].astype(np.int64), device=y.device)]


def _scatter(like, el, parts):
    """Sum of per-corner values parts[c] (instances, elements, ...) onto the nodes."""
    out = torch.zeros(like, dtype=torch.float64, device=parts[0].device)
    for c, v in enumerate(parts):
        out.index_add_(1, torch.as_tensor(el[:, c].astype(np.int64), device=out.device), v)
    return out


def _volumes(q, x):
    out = torch.zeros(len(q.wl.instances), dtype=torch.float64, device=q.dev)
    for tm, mine, nodes in _groups(q):
        y = x[:, nodes].permute(1, 2, 0)
        if tm.kind == "membrane":
            a, b, c = (_corner(y, tm.elems, k) for k in range(3))
        else:
            a, b, c = (_corner(y, tm.elems, k) - _corner(y, tm.elems, 0) for k in (1, 2, 3))
        out[mine] = (a * torch.linalg.cross(b, c)).sum(-1).sum(-1) / 6.0
    return out


def _elastic(tm, y):
    """Elastic forces (instances, nodes, 3) of one template at positions y."""
    X = torch.as_tensor(tm.X, device=y.device)[None]
    if tm.kind == "membrane":
        A, B, C = (_corner(X, tm.elems, k) for k in range(3))
        E1, E2 = B - A, C - A
        l1 = E1.norm(dim=-1, keepdim=True)
        nr = torch.linalg.cross(E1, E2)
        two = nr.norm(dim=-1, keepdim=True)
        e1 = E1 / l1
        e2 = torch.linalg.cross(nr / two, e1)
        Dm = torch.stack([torch.stack([l1[..., 0], (e1 * E2).sum(-1)], -1),
                          torch.stack([torch.zeros_like(l1[..., 0]), (e2 * E2).sum(-1)], -1)], -2)
        weight = 0.5 * two[..., None]
    else:
        x0 = _corner(X, tm.elems, 0)
        Dm = torch.stack([_corner(X, tm.elems, k) - x0 for k in (1, 2, 3)], -1)
        weight = (torch.linalg.det(Dm) / 6.0)[..., None, None]
    m = torch.linalg.inv(Dm)
    x0 = _corner(y, tm.elems, 0)
    F = torch.stack([_corner(y, tm.elems, k) - x0 for k in range(1, Dm.shape[-1] + 1)], -1) @ m
    Cg = F.mT @ F
    eye = torch.eye(Cg.shape[-1], dtype=y.dtype, device=y.device)
    if tm.kind == "membrane":
        I1, I2 = Cg.diagonal(dim1=-2, dim2=-1).sum(-1), torch.linalg.det(Cg)
        adj = I1[..., None, None] * eye - Cg
        if tm.law == "nh":
            S = tm.mu * eye - (tm.mu / I2 ** 2)[..., None, None] * adj
        else:
            S = (tm.mu * (I1 - 1.0))[..., None, None] * eye + (0.5 * tm.C * tm.mu * (I2 - 1.0) - tm.mu)[..., None, None] * adj
    else:
        J = torch.linalg.det(F)[..., None, None]
        Ci = torch.linalg.inv(Cg)
        S = 0.5 * tm.lam * (J * J - 1.0) * Ci + tm.mu * (eye - Ci)
    return _element_forces(tm, y, -weight * (F @ S @ m.mT))


def _element_forces(tm, y, f):
    """Node sums of element forces f (instances, elements, 3, corners 1..): corner 0 takes minus their sum."""
    per = [-f.sum(-1)] + [f[..., k] for k in range(f.shape[-1])]
    return _scatter(y.shape, tm.elems, per)


def _curvature(tm, y):
    """Mixed areas, unit normals, mean and Gaussian curvature and the corner cotangents of a membrane."""
    p = [_corner(y, tm.elems, k) for k in range(3)]
    fn = torch.linalg.cross(p[1] - p[0], p[2] - p[0])
    two = fn.norm(dim=-1)
    dot = [((p[(k + 1) % 3] - p[k]) * (p[(k + 2) % 3] - p[k])).sum(-1) for k in range(3)]
    cot = [t / two for t in dot]
    ang = [torch.atan2(two, t) for t in dot]
    obtuse = (dot[0] < 0) | (dot[1] < 0) | (dot[2] < 0)
    K, area = [], []
    for k in range(3):
        j, l = (k + 1) % 3, (k + 2) % 3
        ej, el = p[k] - p[j], p[k] - p[l]
        K.append(cot[l][..., None] * ej + cot[j][..., None] * el)
        vor = (cot[l] * (ej * ej).sum(-1) + cot[j] * (el * el).sum(-1)) / 8.0
        area.append(torch.where(obtuse, torch.where(dot[k] < 0, two / 4.0, two / 8.0), vor))
    shape = y.shape[:2]
    A = _scatter(shape, tm.elems, area)
    nrm = _scatter(y.shape, tm.elems, [fn] * 3)
    nrm = nrm / nrm.norm(dim=-1, keepdim=True)
    kH = 0.25 * (_scatter(y.shape, tm.elems, K) * nrm).sum(-1) / A
    kG = (2.0 * math.pi - _scatter(shape, tm.elems, ang)) / A
    return A, nrm, kH, kG, cot


def _bending(tm, y):
    A, nrm, kH, kG, cot = _curvature(tm, y)
    h = [_corner(kH, tm.elems, k) for k in range(3)]
    lap = _scatter(y.shape[:2], tm.elems, [cot[(k + 2) % 3] * (h[(k + 1) % 3] - h[k]) + cot[(k + 1) % 3] * (h[(k + 2) % 3] - h[k])
                                           for k in range(3)]) / (2.0 * A)
    return (2.0 * tm.kb * (lap + 2.0 * kH * (kH * kH - kG)) * A)[..., None] * nrm


def _forces(q, x):
    out = torch.zeros_like(x)
    for tm, _, nodes in _groups(q):
        y = x[:, nodes].permute(1, 2, 0)
        F = _elastic(tm, y) + (_bending(tm, y) if tm.kb else 0.0)
        out[:, nodes] = F.permute(2, 0, 1)
    return out


def _fluid_forces(q, x, u, C):
    out = torch.zeros_like(x)
    for tm, _, nodes in _groups(q, ("solid",)):
        y, w = x[:, nodes].permute(1, 2, 0), u[:, nodes].permute(1, 2, 0)
        c6 = C[:, nodes].permute(1, 2, 0)
        sym = [0, 3, 4, 3, 1, 5, 4, 5, 2]
        mean = sum(_corner(c6, tm.elems, k) for k in range(4)) / 4.0
        eye = torch.eye(3, dtype=y.dtype, device=y.device)
        poly = mean[..., sym].reshape(mean.shape[:2] + (3, 3)) - eye
        X = torch.as_tensor(tm.X, device=y.device)[None]

        def edges(a):
            return torch.stack([_corner(a, tm.elems, k) - _corner(a, tm.elems, 0) for k in (1, 2, 3)], -1)

        Dm = edges(X)
        m, V = torch.linalg.inv(Dm), (torch.linalg.det(Dm) / 6.0)[..., None, None]
        F = edges(y) @ m
        J, Fi = torch.linalg.det(F)[..., None, None], torch.linalg.inv(F)
        grad = edges(w) @ m @ Fi
        P = J * (ETA * (grad + grad.mT) + ETA * (1.0 - BETA) / RELAX * poly) @ Fi.mT
        out[:, nodes] = _element_forces(tm, y, V * (P @ m.mT)).permute(2, 0, 1)
    return out


def _stencil(q, case, x, o):
    """Per node: grid indices within its box's lattice (N, points) and weights, for lattice offset o."""
    box = np.array([it.box for it in q.wl.instances])
    n = torch.as_tensor(np.array([q.wl.boxes[b].n for b in box]), device=q.dev)[q.inst]
    L = torch.as_tensor(np.array([q.wl.boxes[b].L for b in box]), device=q.dev)[q.inst]
    s = (torch.as_tensor(q.origin, device=q.dev).T[:, q.inst] + x) * (n / L) - torch.tensor(o, dtype=torch.float64, device=q.dev)[:, None]
    mls = case["kernel"] == "mls27"
    width = 3 if mls else 4
    base = torch.floor(s + 0.5) - 1 if mls else torch.floor(s) - 1
    r = base[:, :, None] + torch.arange(width, device=q.dev) - s[:, :, None]   # (3, N, width)
    idx = torch.remainder(base.long()[:, :, None] + torch.arange(width, device=q.dev), n[None, :, None])
    flat = ((idx[2][:, :, None, None] * n[:, None, None, None] + idx[1][:, None, :, None]) * n[:, None, None, None]
            + idx[0][:, None, None, :]).reshape(len(n), -1)
    if not mls:
        a = r.abs()
        near = (3.0 - 2.0 * a + torch.sqrt((1.0 + 4.0 * a - 4.0 * a * a).clamp(min=0.0))) / 8.0
        far = (5.0 - 2.0 * a - torch.sqrt((-7.0 + 12.0 * a - 4.0 * a * a).clamp(min=0.0))) / 8.0
        ph = torch.where(a <= 1.0, near, torch.where(a <= 2.0, far, torch.zeros_like(a)))
        return flat, (ph[2][:, :, None, None] * ph[1][:, None, :, None] * ph[0][:, None, None, :]).reshape(len(n), -1), n, L, box
    y = torch.stack(torch.broadcast_tensors(r[0][:, None, None, :], r[1][:, None, :, None], r[2][:, :, None, None]), -1).reshape(len(n), 27, 3)
    rad = y.norm(dim=-1) / math.sqrt(3.0)
    w = torch.where(rad <= 0.5, 2.0 / 3.0 - 4.0 * rad ** 2 + 4.0 * rad ** 3,
                    torch.where(rad <= 1.0, 4.0 / 3.0 * (1.0 - rad) ** 3, torch.zeros_like(rad)))
    p = torch.cat([torch.ones_like(y[..., :1]), y], -1)
    mom = torch.einsum("nj,nja,njb->nab", w, p, p)
    rhs = torch.zeros((len(n), 4), dtype=torch.float64, device=q.dev)
    rhs[:, 0] = 1.0
    z = torch.linalg.solve(mom, rhs)
    return flat, w * (p * z[:, None, :]).sum(-1), n, L, box


def _transfer(q, case, x, u=None, F=None, density=True):
    """(v interpolated from u, f spread from F), each where given, over the three MAC lattices."""
    offs = np.concatenate([[0], np.cumsum([3 * bx.n ** 3 for bx in q.wl.boxes])])
    v = torch.empty_like(x) if u is not None else None
    f = torch.zeros(int(offs[-1]), dtype=torch.float64, device=q.dev) if F is not None else None
    for d in range(3):
        flat, w, n, L, box = _stencil(q, case, x, [0.0 if a == d else 0.5 for a in range(3)])
        flat = flat + (torch.as_tensor(offs[:-1][box], device=q.dev)[q.inst] + d * n ** 3)[:, None]
        if u is not None:
            v[d] = (w * u[flat]).sum(1)
        if F is not None:
            g = F[d] * (n / L) ** 3 if density else F[d]
            f.index_add_(0, flat.reshape(-1), (w * g[:, None]).reshape(-1))
    return v, f


def _sums(q, x, F, v, f):
    out = []
    count = torch.as_tensor(np.diff(q.off).astype(float), device=q.dev)

    def total(a):
        return torch.zeros((3, len(count)), dtype=torch.float64, device=q.dev).index_add_(1, q.inst, a)

    cen = total(x) / count
    out = torch.cat([cen, total(F), total(torch.linalg.cross((x - cen[:, q.inst]).T, F.T).T), total(v)]).T.reshape(-1)
    at, boxes = 0, []
    for bx in q.wl.boxes:
        n3 = bx.n ** 3
        boxes += [f[at + d * n3:at + (d + 1) * n3].sum() * bx.h ** 3 for d in range(3)] + [f.new_zeros(())] * 3
        at += 3 * n3
    return torch.cat([out, torch.stack(boxes)])


def _corrected(q, x):
    """Positions after the membrane volume correction, and its multiplier per particle."""
    x, lam = x.clone(), torch.zeros_like(q.V0)
    for tm, mine, nodes in _groups(q, ("membrane",)):
        y = x[:, nodes].permute(1, 2, 0)
        p = [_corner(y, tm.elems, k) for k in range(3)]
        al = _scatter(y.shape, tm.elems, [torch.linalg.cross(p[(k + 1) % 3], p[(k + 2) % 3]) for k in range(3)]) * (-1.0 / 12.0)
        a = [_corner(al, tm.elems, k) for k in range(3)]

        def cyc(s, t, r):
            return sum((s[k] * torch.linalg.cross(t[(k + 1) % 3], r[(k + 2) % 3])).sum(-1) for k in range(3)).sum(-1)

        A, B, C = cyc(a, a, a) / 18.0, cyc(p, a, a) / 6.0, cyc(a, p, p) / 6.0
        D = cyc(p, p, p) / 18.0 - q.V0[mine]
        z = torch.zeros_like(D)
        for _ in range(50):
            z = z - (((A * z + B) * z + C) * z + D) / ((3.0 * A * z + 2.0 * B) * z + C)
        lam[mine] = z
        x[:, nodes] = (y + z[:, None, None] * al).permute(2, 0, 1)
    return x, lam


def exact(case, seed):
    """run()'s outputs in 64 bits from the same inputs, in plain torch."""
    q = _Inputs(case, seed)
    x = q.x.double()
    path = case["path"]
    if path in ("step", "step_ab2", "step_host"):
        F = _forces(q, x)
        v, f = _transfer(q, case, x, q.u.double(), F)
        out = {"F": F, "f": f, "v": v, "red": _sums(q, x, F, v, f) if case["sums"] else None}
        if path == "step_ab2":
            out["x"] = x + q.dt * (1.5 * v - 0.5 * q.vp.double())
        return out
    if path == "transfer":
        v, f = _transfer(q, case, x, q.u.double(), q.F.double())
        gF, gu = _transfer(q, case, x, q.gf.double(), q.gv.double(), density=False)
        scale = torch.as_tensor([(bx.n / bx.L) ** 3 for bx in q.wl.boxes], dtype=torch.float64, device=q.dev)
        box = torch.as_tensor([it.box for it in q.wl.instances], device=q.dev)[q.inst]
        return {"f": f, "v": v, "gF": gF * scale[box], "gu": gu}
    if path == "elastic":
        xr = x.clone().requires_grad_()
        F = _forces_graph(q, xr)
        (gx,) = torch.autograd.grad(F, xr, q.gF.double())
        return {"F": F.detach(), "gx": gx}
    if path == "fluid":
        v, _ = _transfer(q, case, x, q.u.double())
        flat, w, n, _, box = _stencil(q, case, x, (0.5, 0.5, 0.5))
        start = np.concatenate([[0], np.cumsum([6 * bx.n ** 3 for bx in q.wl.boxes])])[:-1][box]
        flat = flat + torch.as_tensor(start, device=q.dev)[q.inst][:, None]
        field = q.C.double()
        C = torch.stack([(w * field[flat + (k * n ** 3)[:, None]]).sum(1) for k in range(6)])
        F = _forces(q, x) + _fluid_forces(q, x, v, C)
        return {"v": v, "C": C, "F": F, "f": _transfer(q, case, x, F=F)[1]}
    x, lam = _corrected(q, x + q.dt * (1.5 * q.v.double() - 0.5 * q.vp.double()))
    nA = torch.zeros_like(x)
    for tm, _, nodes in _groups(q, ("membrane",)):
        A, nrm, _, _, _ = _curvature(tm, x[:, nodes].permute(1, 2, 0))
        nA[:, nodes] = (A[..., None] * nrm).permute(2, 0, 1)
    return {"x": x, "lam": lam, "vol": _volumes(q, x), "G": _transfer(q, case, x, F=nA)[1]}


def _forces_graph(q, x):
    """Elastic forces as a differentiable function of x."""
    parts, order = [], []
    for tm, _, nodes in _groups(q):
        parts.append(_elastic(tm, x[:, nodes].permute(1, 2, 0)).permute(2, 0, 1).reshape(3, -1))
        order.append(nodes.reshape(-1))
    back = torch.empty(q.N, dtype=torch.long, device=q.dev)
    back[torch.cat(order)] = torch.arange(q.N, device=q.dev)
    return torch.cat(parts, 1)[:, back]
