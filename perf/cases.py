"""The workloads this framework is timed on, each through its public entry points.

What a user of the framework runs, over the range they run it: whole hydro steps (float32
and float64; 8^3, 16^3 and 32^3 blocks; uniform and refined meshes; both interface solvers,
contact steepening, the dual-energy field; the default sweep variant and tuned ones;
state in device or in host memory), one mesh adaptation (refresh, flags, octree rebuild,
remap), tracers, the multigrid Poisson solve in both precisions, and the gradient of a
rollout.

A hydro pass is two steps, an even and an odd cycle, because the sweep order alternates.
Its output is the interior of the state: the ghost layer is the step's scratch (every
consumer refreshes it first).

exact() evaluates the same formulas in plain torch float64 on the same inputs: ghost values
from the cell's level and position, three split PPM sweeps, coarse-fine flux correction,
the CFL minimum; the multigrid cycle on one periodic grid; trilinear tracers; the gradient
by torch's autograd.
"""
import math

import numpy as np
import torch

G = 4   # ghost depth of the blocks


# ---------------------------------------------------------------------------------- cases
def _step(name, **kw):
    c = dict(name=name, kind="step", root=4, n=16, levels=0, spheres=0, precision=4, outflow=False, hllc=False,
             steepening=False, dual=False, cfl_step=False, tuned=False, host=False, flow="blobs", geometry=1)
    c.update(kw)
    return c


def listed():
    return [
        # a shock tube on 4^3 blocks of 16^3, default variant: the first thing a user runs; launches and latency count
        _step("sod_f32_64blocks", outflow=True, flow="sod"),
        # a refined blast on 16^3 blocks, the ordinary adaptive run (steps between two adaptations)
        _step("blast_amr_f32_16", levels=3, spheres=6, tuned=True, flow="blast"),
        # the framework's main path: moving dense blobs on 32^3 blocks refined two levels, dt from the start state
        _step("blobs_amr_f32_32", root=12, n=32, levels=2, spheres=160, tuned=True, cfl_step=True),
        # the method variants in earnest: HLLC, steepening and the dual-energy field, every cell moving
        _step("variants_amr_f32_32", n=32, levels=1, spheres=8, hllc=True, steepening=True, dual=True, tuned=True,
              flow="abc"),
        # a float64 run on small refined blocks: reference solutions and parity studies
        _step("blobs_amr_f64_16", levels=2, spheres=10, precision=8),
        # the state kept in page-locked host memory, one library call per step
        _step("blobs_amr_f32_host", n=32, levels=2, spheres=6, tuned=True, host=True),
        # adaptation of a moving front: refresh, flags, rebuild, remap (every few steps of an adaptive run)
        dict(name="adapt_f32_16", kind="adapt", root=4, n=16, levels=4, spheres=3, precision=4, geometry=2),
        # tracers on a refined state, one lookup after an adaptation and one push
        dict(name="tracers_4m", kind="tracers", root=4, n=32, levels=2, spheres=6, precision=4, count=1 << 22,
             geometry=1),
        # self-gravity on a small periodic box, mixed precision: many short launches
        dict(name="poisson_mixed_64", kind="poisson", root=4, n=16, inner=4, cycles=8),
        # self-gravity on an ordinary box, mixed precision
        dict(name="poisson_mixed_256", kind="poisson", root=8, n=32, inner=4, cycles=8),
        # the same solve in float64
        dict(name="poisson_f64_128", kind="poisson", root=8, n=16, inner=8, cycles=8),
        # gradient of a loss on the final state of a float64 rollout: forward, recomputation, adjoint
        dict(name="gradient_f64_16", kind="gradient", root=4, n=16, levels=0, precision=8, steps=3, every=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["adapt", "tracers", "poisson", "gradient"])
    geometry = rng.randrange(1000)
    if kind == "step":
        n = rng.choice([8, 16, 32])
        levels = rng.choice([0, 1, 2, 3])
        root = rng.randint(1, {8: 12, 16: 7, 32: 5}[n] if levels < 3 else 3)
        f64 = rng.random() < 0.25
        if f64:
            root = min(root, {8: 6, 16: 3, 32: 2}[n])
        flow = rng.choice(["blobs", "abc", "blast"])
        dual = rng.random() < 0.2
        host = rng.random() < 0.15
        return {k: v for k, v in _step("", root=root, n=n, levels=levels, spheres=rng.randint(1, 8),
                                       precision=8 if f64 else 4, outflow=rng.random() < 0.3,
                                       hllc=rng.random() < 0.3, steepening=rng.random() < 0.3, dual=dual,
                                       cfl_step=not host and rng.random() < 0.5, tuned=rng.random() < 0.6,
                                       host=host, flow=flow, geometry=geometry).items() if k != "name"}
    if kind == "adapt":
        n = rng.choice([8, 16, 32])
        return dict(kind=kind, root=rng.randint(2, 4), n=n, levels=rng.randint(1, {8: 4, 16: 3, 32: 2}[n]),
                    spheres=rng.randint(1, 4), precision=rng.choice([4, 4, 8]), geometry=geometry)
    if kind == "tracers":
        return dict(kind=kind, root=rng.randint(2, 5), n=rng.choice([16, 32]), levels=rng.randint(0, 2),
                    spheres=rng.randint(1, 6), precision=rng.choice([4, 4, 8]),
                    count=int(_log(rng, 1 << 10, 1 << 22)) | 1, geometry=geometry)
    if kind == "poisson":
        n = rng.choice([8, 16, 32])
        return dict(kind=kind, root=rng.randint(1, {8: 20, 16: 12, 32: 8}[n]), n=n, inner=rng.choice([4, 4, 8]),
                    cycles=rng.randint(4, 8))
    return dict(kind=kind, root=rng.randint(2, 4), n=rng.choice([8, 16]), levels=0, precision=rng.choice([8, 4]),
                steps=rng.randint(1, 3), every=rng.randint(1, 3))


# ----------------------------------------------------------------------- meshes and states
def _spheres(case, shift=0.0):
    """Centres and radii of the case's spheres in the unit box (geometry fixed by the case)."""
    r = np.random.RandomState(case.get("geometry", 0) + 17)
    k = case.get("spheres", 0)
    c, rad = r.rand(k, 3), r.uniform(0.03, 0.09, k) * (4.0 / max(4, case["root"])) ** 0.75
    return (c + shift) % 1.0, rad


def _periodic(case):
    return (not case.get("outflow", False), True, True)


def _wrap(case, d):
    """Minimum image of a displacement d[..., 3] on the periodic axes."""
    p = torch.tensor([1.0 if v else 0.0 for v in _periodic(case)], dtype=d.dtype, device=d.device)
    return d - p * torch.round(d)


def _leaves(case, shift=0.0):
    """2:1 balanced leaf list [B, 4] (level, i, j, k) refined where a sphere's surface passes, in Morton order."""
    R, L = case["root"], case.get("levels", 0)
    cen, rad = _spheres(case, shift)
    per = np.array(_periodic(case), dtype=float)
    refined = [np.zeros((R << l,) * 3, bool) for l in range(L + 1)]      # [z, y, x]
    for l in range(L):
        w = 1.0 / (R << l)
        ax = (np.arange(R << l) + 0.5) * w
        for c, r in zip(cen, rad):
            near, far = [], []
            for a in range(3):
                d = ax - c[a]
                d = np.abs(d - per[a] * np.round(d))
                near.append(np.maximum(d - 0.55 * w, 0.0) ** 2)
                far.append((d + 0.55 * w) ** 2)
            lo = near[2][:, None, None] + near[1][None, :, None] + near[0][None, None, :]
            hi = far[2][:, None, None] + far[1][None, :, None] + far[0][None, None, :]
            refined[l] |= (lo < r * r) & (hi > r * r)
    for l in range(L - 1, 0, -1):        # parents of refined nodes and of their neighbours are refined
        grown = refined[l]
        for a in range(3):
            m = np.moveaxis(grown, a, 0)
            up, dn = np.zeros_like(m), np.zeros_like(m)
            up[1:], dn[:-1] = m[:-1], m[1:]
            if per[2 - a]:
                up[0], dn[-1] = m[-1], m[0]
            grown = np.moveaxis(m | up | dn, 0, a)
        h = R << (l - 1)
        refined[l - 1] |= grown.reshape(h, 2, h, 2, h, 2).any((1, 3, 5))
    out = []
    for l in range(L + 1):
        leaf = ~refined[l]
        if l:
            leaf &= refined[l - 1].repeat(2, 0).repeat(2, 1).repeat(2, 2)
        z, y, x = np.nonzero(leaf)
        out.append(np.stack([np.full_like(x, l), x, y, z], 1))
    lv = np.concatenate(out).astype(np.int64)
    key = np.zeros(len(lv), np.int64)
    for a in range(3):
        v = lv[:, 1 + a] << (L - lv[:, 0])
        for b in range(16):
            key |= ((v >> b) & 1) << (3 * b + a)
    return lv[np.argsort(key)]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _waves(seed, count=4):
    """A few random Fourier modes per field: the smooth part of a state, made from the seed alone."""
    r = np.random.RandomState(seed % (1 << 32))
    return r.randint(-2, 3, (5, count, 3)), r.uniform(0, 2 * math.pi, (5, count)), r.uniform(-1, 1, (5, count)) / count


def _fill(case, leaves, seed, U, shift=0.0, gamma=5.0 / 3.0):
    """The case's initial state, sampled at every cell centre of the padded blocks, into U[B, fields, N, N, N]."""
    dev, n = U.device, case["n"]
    N, flow = n + 2 * G, case.get("flow", "blobs")
    cen, rad = _spheres(case, shift)
    modes, phase, amp = _waves(seed)
    r = np.random.RandomState((seed * 7919 + 3) % (1 << 32))
    vel = 0.1 * r.randn(max(1, len(rad)), 3)
    contrast = 9.0 + 2.0 * r.rand(max(1, len(rad)))
    lv = torch.as_tensor(leaves, device=dev)
    w = 1.0 / (case["root"] * 2.0 ** lv[:, 0].double())
    off = (torch.arange(N, device=dev, dtype=torch.float64) - G + 0.5) / n
    for s in range(0, len(lv), 128):
        t = slice(s, s + 128)
        # x, y, z of the cells, each [b, 1.., N, ..1]
        p = [((lv[t, 1 + a].double().view(-1, 1) + off) * w[t].view(-1, 1)) for a in range(3)]
        p = [p[0][:, None, None, :], p[1][:, None, :, None], p[2][:, :, None, None]]
        f = []
        for q in range(5):      # separable products: one sine per axis
            v = 0.0
            for k, ph, am in zip(modes[q], phase[q], amp[q]):
                v = v + am * (torch.sin(2 * math.pi * k[0] * p[0] + ph) * torch.cos(2 * math.pi * k[1] * p[1] + 2 * ph)
                              * torch.cos(2 * math.pi * k[2] * p[2] + 3 * ph))
            f.append(v)
        rho, u, pr = 1.0 + 0.02 * f[0], [0.02 * f[1 + a] for a in range(3)], 1.0 + 0.02 * f[4]
        if flow == "sod":
            left = (p[0] < 0.5).expand_as(rho)
            rho, pr = torch.where(left, rho, 0.125 * rho), torch.where(left, pr, 0.1 * pr)
        elif flow == "smooth":
            rho, u, pr = 1.0 + 0.3 * f[0], [0.2 * f[1 + a] for a in range(3)], 1.0 + 0.3 * f[4]
        if flow in ("blobs", "abc", "blast"):
            box = torch.stack([q.amax(dim=(1, 2, 3)) + q.amin(dim=(1, 2, 3)) for q in p], 1) / 2
            half = w[t] * (0.5 + G / n)
            for i in range(len(rad)):
                c = torch.as_tensor(cen[i], device=dev)
                d = (_wrap(case, box - c).abs() - half.view(-1, 1)).clamp_min(0.0)
                b = torch.nonzero((d * d).sum(1) < rad[i] ** 2)[:, 0]
                if not len(b):
                    continue
                dd = [q[b] - c[a] for a, q in enumerate(p)]
                dd = [x - torch.round(x) if per else x for x, per in zip(dd, _periodic(case))]
                inside = dd[0] ** 2 + dd[1] ** 2 + dd[2] ** 2 < rad[i] ** 2
                if flow == "blast":
                    pr[b] = torch.where(inside, pr[b] * 5.0 * contrast[i], pr[b])
                else:
                    rho[b] = torch.where(inside, rho[b] * contrast[i], rho[b])
                    for a in range(3):
                        u[a][b] = torch.where(inside, u[a][b] + vel[i, a], u[a][b])
        if flow == "abc":
            k = 2 * math.pi
            u[0] = u[0] + 0.3 * (torch.sin(k * p[2]) + torch.cos(k * p[1]))
            u[1] = u[1] + 0.3 * (torch.sin(k * p[0]) + torch.cos(k * p[2]))
            u[2] = u[2] + 0.3 * (torch.sin(k * p[1]) + torch.cos(k * p[0]))
        ei = pr / (gamma - 1.0)
        E = ei + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        for q, v in enumerate((rho, rho * u[0], rho * u[1], rho * u[2], E, ei)[:U.shape[1]]):
            U[t, q] = v.to(U.dtype)
    return U


def _desc(case, gamma=5.0 / 3.0):
    from paper_1810_01319_gb300 import OUTFLOW, PERIODIC, make_desc
    return make_desc(root=(case["root"],) * 3, n=case["n"], max_level=case.get("levels", 0), hi=(1.0, 1.0, 1.0),
                     bc=tuple(PERIODIC if v else OUTFLOW for v in _periodic(case)),
                     precision=case.get("precision", 8), gamma=gamma, riemann=int(case.get("hllc", False)),
                     steepening=int(case.get("steepening", False)), dual_energy=int(case.get("dual", False)))


def _mesh(case, leaves):
    from paper_1810_01319_gb300 import EXEC_GRAPH, Mesh
    mesh = Mesh(_desc(case), leaves=leaves)
    mesh.set_exec(EXEC_GRAPH)
    if case.get("tuned"):       # what autotuning a float32 mesh of this kind picks; float64 takes the resident schedule
        mesh.set_sweep_variants([22, 21, 21] if case["precision"] == 4 else [1, 1, 1])
    return mesh


def _interior(U, n):
    return U[:, :, G:G + n, G:G + n, G:G + n]


# --------------------------------------------------------------------------- prepare, run
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "poisson":
        s["mesh"] = _mesh(dict(case, precision=8), _leaves(case))
        s["f"] = _poisson_rhs(case, seed)
        return s
    leaves = _leaves(case)
    s["mesh"] = mesh = _mesh(case, leaves)
    if kind == "adapt":         # the mesh follows the spheres' old places, the state their new ones
        s["U"] = _fill(case, leaves, seed, mesh.empty_state(), shift=_moved(case))
        return s
    flow = "smooth" if kind == "gradient" else case.get("flow", "blobs")
    s["U"] = U = _fill(dict(case, flow=flow), leaves, seed, mesh.empty_state())
    if kind == "step":
        s["dt"] = torch.zeros(1, dtype=torch.float64, device=U.device)
        s["totals"] = torch.zeros(5, dtype=torch.float64, device=U.device)
        if case["host"]:
            s["host"] = torch.empty(U.shape, dtype=U.dtype, pin_memory=True)
            s["host"].copy_(U)
            mesh.reduce(U, 0.4, dt_next=s["dt"])
            s["dt_host"] = float(s["dt"])
        elif not case["cfl_step"]:
            mesh.reduce(U, 0.4, dt_next=s["dt"])
    elif kind == "tracers":
        mesh.ghost_refresh(U)
        s["pos"] = _tracers(case, seed)
        s["dt"] = torch.full((1,), 0.02 / (case["root"] * case["n"]), dtype=torch.float64, device=U.device)
    elif kind == "gradient":
        s["dts"] = [0.1 / (case["root"] * case["n"])] * case["steps"]
        s["target"] = _interior(_fill(dict(case, flow="smooth"), leaves, seed + 1, torch.empty_like(U)),
                                case["n"]).contiguous()
        U.requires_grad_()
    return s


def run(s):
    case, mesh = s["case"], s["mesh"]
    kind, n = case["kind"], case["n"]
    if kind == "poisson":
        return mesh.poisson_solve(s["f"], case["cycles"], residuals=False, inner=case["inner"])[0]
    U = s["U"]
    if kind == "step":
        if case["host"]:
            for cycle in (0, 1):
                s["dt_host"], totals = mesh.hydro_step_host(s["host"], U, s["dt_host"], cycle, 0.4)
            return dict(U=_interior(s["host"], n), dt=s["dt_host"], totals=totals)
        for cycle in (0, 1):
            if case["cfl_step"]:
                mesh.hydro_step_cfl(U, cycle, 0.4, s["dt"], totals=s["totals"])
            else:
                mesh.hydro_step(U, s["dt"], cycle, 0.4, dt_next=s["dt"], totals=s["totals"])
        return dict(U=_interior(U, n), dt=s["dt"], totals=s["totals"])
    if kind == "adapt":
        from paper_1810_01319_gb300 import Mesh
        mesh.ghost_refresh(U)
        flags = mesh.refine_flags(U, field=0, tau=0.3, tau_c=0.075)
        new = Mesh(mesh.desc, mesh, flags.cpu().numpy())
        V = new.remap_from(mesh, U)
        return dict(flags=flags, leaves=new.leaves, old=U, new=_interior(V, n))
    if kind == "tracers":
        pos = s["pos"].clone()      # the user keeps the old positions
        leaf = mesh.particles_locate(pos)
        mesh.particles_push(U, pos, leaf, s["dt"])
        return dict(pos=pos, leaf=leaf)
    from paper_1810_01319_gb300.autograd import rollout
    U.grad = None
    out = _interior(rollout(mesh, U, s["dts"], 0, case["every"]), n)
    ((out - s["target"]) ** 2).sum().backward()
    return dict(U=out.detach(), grad=U.grad)


def work(case):
    kind = case["kind"]
    n = case["n"]
    if kind == "poisson":       # f in, phi out; about 25 operations a cell and sweep, five sweeps' worth of the fine grid a cycle
        M3 = (case["root"] * n) ** 3
        return {"bytes": 16 * M3, "flops": case["cycles"] * M3 * 140}
    B = len(_leaves(case))
    cells, prec = B * n ** 3, case["precision"]
    if kind == "tracers":       # position and leaf in and out, eight corners of four fields
        return {"bytes": case["count"] * (56 + 24 + 8 * 4 * prec), "flops": case["count"] * 150}
    if kind == "adapt":         # the state in, ghosts and the new state out
        return {"bytes": prec * 5 * (2 * cells + B * ((n + 2 * G) ** 3 - n ** 3)), "flops": cells * 30}
    if kind == "gradient":      # per step: forward and adjoint, the latter about four times the operations
        return {"bytes": 4 * case["steps"] * cells * 5 * prec, "flops": case["steps"] * cells * 1600 * 6}
    fields = 6 if case["dual"] else 5
    # about 530 operations a cell and sweep, three sweeps and two steps
    return {"bytes": 2 * 2 * cells * fields * prec, "flops": 2 * 3 * 530 * cells}


def _moved(case):
    return 0.6 / case["root"]


def _poisson_rhs(case, seed):
    g = torch.Generator(device=_device()).manual_seed(seed)
    return torch.randn(case["root"] ** 3, case["n"], case["n"], case["n"], dtype=torch.float64, device=_device(),
                       generator=g)


def _tracers(case, seed):
    g = torch.Generator(device=_device()).manual_seed(seed)
    return torch.rand(3, case["count"], dtype=torch.float64, device=_device(), generator=g)


# ------------------------------------------------------------------ the same in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        return _exact_poisson(case, _poisson_rhs(case, seed))
    leaves = _leaves(case)
    cells = len(leaves) * (case["n"] + 2 * G) ** 3
    if kind == "adapt":
        if cells > 2e8:
            return None
        tree = _Tree(case, leaves)
        dt = torch.float32 if case["precision"] == 4 else torch.float64
        U = _fill(case, leaves, seed, torch.empty((len(leaves), 5) + (case["n"] + 2 * G,) * 3, dtype=dt,
                                                 device=_device()), shift=_moved(case)).double()
        # the rebuilt mesh and its state have no floating arithmetic beyond what `old` shows
        return dict(flags=None, leaves=None, old=tree.padded(_interior(U, case["n"]).contiguous()), new=None)
    if cells > 4e8 or (kind == "gradient" and cells > 1.5e6):
        return None             # over 20 seconds, or its autograd tape over the card
    flow = "smooth" if kind == "gradient" else case.get("flow", "blobs")
    dt = torch.float32 if case["precision"] == 4 else torch.float64
    fields = 6 if case.get("dual") else 5
    P = torch.empty((len(leaves), fields) + (case["n"] + 2 * G,) * 3, dtype=dt, device=_device())
    P = _fill(dict(case, flow=flow), leaves, seed, P)
    U = _interior(P, case["n"]).double().contiguous()
    del P
    tree = _Tree(case, leaves)
    if kind == "tracers":
        return _exact_tracers(case, tree, U, _tracers(case, seed))
    if kind == "gradient":
        target = _fill(dict(case, flow="smooth"), leaves, seed + 1,
                       torch.empty((len(leaves), 5) + (case["n"] + 2 * G,) * 3, dtype=dt, device=_device()))
        target = _interior(target, case["n"]).double()
        step_dt = 0.1 / (case["root"] * case["n"])
        states = [U]
        for c in range(case["steps"]):
            with torch.no_grad():
                states.append(tree.step(states[-1], step_dt, c))
        lam = 2.0 * (states[-1] - target)
        for c in reversed(range(case["steps"])):
            V = states[c].detach().requires_grad_()
            lam, = torch.autograd.grad(tree.step(V, step_dt, c), V, lam)
        return dict(U=states[-1], grad=torch.nn.functional.pad(lam, (G,) * 6))
    h, totals = tree.reduce(U)
    for cycle in (0, 1):
        step = 0.4 * h
        start_totals = totals
        U = tree.step(U, step, cycle)
        h, totals = tree.reduce(U)
    if case["cfl_step"]:
        dt_out, tot = step, start_totals
    else:
        dt_out, tot = 0.4 * h, totals
    if case["host"]:
        return dict(U=U, dt=float(dt_out), totals=[float(v) for v in tot])
    return dict(U=U, dt=torch.tensor([dt_out], dtype=torch.float64), totals=tot)


def _exact_poisson(case, f):
    R, n = case["root"], case["n"]
    leaves = _leaves(case)
    M = R * n
    dev = f.device
    grid = torch.empty(M, M, M, dtype=torch.float64, device=dev)
    at = [(slice(k * n, k * n + n), slice(j * n, j * n + n), slice(i * n, i * n + n)) for _, i, j, k in leaves]
    for b, w in enumerate(at):
        grid[w] = f[b]

    def nb(p):
        return sum(torch.roll(p, s, d) for d in (2, 1, 0) for s in (1, -1))

    def sweeps(p, g, h, count):
        for _ in range(count):
            p = (1.0 - 6.0 / 7.0) * p + (6.0 / 7.0) * ((nb(p) - h * h * g) / 6.0)
        return p

    def residual(p, g, h):
        return g - (nb(p) - 6.0 * p) / (h * h)

    def vcycle(p, g, h):
        m = p.shape[0]
        if m == 1:
            return torch.zeros_like(p)
        if m % 2:
            return sweeps(p, g, h, 50)
        p = sweeps(p, g, h, 2)
        r = residual(p, g, h).reshape(m // 2, 2, m // 2, 2, m // 2, 2).mean((1, 3, 5))
        e = vcycle(torch.zeros_like(r), r, 2 * h)
        for d in (2, 1, 0):
            lo, hi = 0.75 * e + 0.25 * torch.roll(e, 1, d), 0.75 * e + 0.25 * torch.roll(e, -1, d)
            e = torch.stack([lo, hi], d + 1).flatten(d, d + 1)
        return sweeps(p + e, g, h, 2)

    grid -= grid.mean()
    p = torch.zeros_like(grid)
    for _ in range(case["cycles"]):
        p = vcycle(p, grid, 1.0 / M)
    p -= p.mean()
    return torch.stack([p[w] for w in at])


def _exact_tracers(case, tree, U, pos):
    n, L = case["n"], case["levels"]
    N = n + 2 * G
    P = tree.padded(U)
    R = case["root"] << L
    cover = torch.zeros(R, R, R, dtype=torch.int64, device=U.device)
    for b, (l, i, j, k) in enumerate(tree.leaves.tolist()):
        s = 1 << (L - l)
        cover[k * s:k * s + s, j * s:j * s + s, i * s:i * s + s] = b

    def leaf_of(x):
        c = (x * R).long().clamp(0, R - 1)
        return cover[c[2], c[1], c[0]]

    leaf = leaf_of(pos)
    lv = tree.lv[leaf]
    w = 1.0 / (case["root"] * 2.0 ** lv[:, 0].double())
    t = torch.stack([(pos[a] - lv[:, 1 + a] * w) * n / w - 0.5 for a in range(3)])
    i0 = torch.floor(t).long()
    fr = t - i0
    vel = torch.zeros_like(pos)
    flat = P.reshape(P.shape[0], 5, N ** 3)
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                cell = ((i0[2] + G + dz) * N + i0[1] + G + dy) * N + i0[0] + G + dx
                wt = ((fr[0] if dx else 1 - fr[0]) * (fr[1] if dy else 1 - fr[1]) * (fr[2] if dz else 1 - fr[2]))
                rho = flat[leaf, 0, cell]
                for a in range(3):
                    vel[a] += wt * flat[leaf, 1 + a, cell] / rho
    out = pos + 0.02 / (case["root"] * n) * vel
    out = torch.where(out < 0, out + 1.0, torch.where(out >= 1.0, out - 1.0, out))
    return dict(pos=out, leaf=None)


class _Tree:
    """The refined mesh in plain torch: a cell's value at a level and position, one hydro step, the reduction."""

    gamma = 5.0 / 3.0

    def __init__(self, case, leaves):
        self.case, self.leaves, self.n = case, leaves, case["n"]
        self.dev = _device()
        self.lv = torch.as_tensor(leaves, device=self.dev)
        self.maps = []
        for l in range(case["levels"] + 2):
            m = torch.full((case["root"] << l,) * 3, -1, dtype=torch.int64, device=self.dev)
            b = torch.nonzero(self.lv[:, 0] == l)[:, 0]
            m[self.lv[b, 3], self.lv[b, 2], self.lv[b, 1]] = b
            self.maps.append(m)
        self.dx = 1.0 / (case["root"] * self.n * 2.0 ** self.lv[:, 0].double())
        self.axes = {0: (0, 1, 2, 3, 4, 5), 1: (0, 2, 1, 3, 4, 5), 2: (0, 3, 1, 2, 4, 5)}

    # cells g = (x, y, z) of level l, indices inside the box
    def _leaf(self, l, g):
        n = self.n
        return self.maps[l][g[2] // n, g[1] // n, g[0] // n]

    def _load(self, U, b, g):
        n = self.n
        return U[b, :, g[2] % n, g[1] % n, g[0] % n]

    def _bound(self, l, g):
        M = (self.case["root"] << l) * self.n
        return [torch.remainder(v, M) if p else v.clamp(0, M - 1) for v, p in zip(g, _periodic(self.case))]

    def _mean(self, U, l, g):
        v = 0.0
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    h = [2 * g[0] + dx, 2 * g[1] + dy, 2 * g[2] + dz]
                    v = v + self._load(U, self._leaf(l + 1, h), h)
        return 0.125 * v

    def _value(self, U, l, g, slopes):
        """Values [K, fields]: copied, the mean of finer cells, or from the coarser cell (limited slopes, or as it is)."""
        own = self._leaf(l, g)
        fine = torch.zeros_like(own, dtype=torch.bool)
        if l + 1 <= self.case["levels"]:
            h = [2 * v for v in g]
            # any finer leaf under the node: all children that touch the asking leaf are leaves (2:1 balance)
            fine = (own < 0) & (self._leaf(l + 1, h) >= 0)
        parts, order = [], []
        for mask, f in ((own >= 0, lambda c: self._load(U, self._leaf(l, c), c)),
                        (fine, lambda c: self._mean(U, l, c)),
                        ((own < 0) & ~fine, lambda c: self._coarse(U, l, c, slopes))):
            k = torch.nonzero(mask)[:, 0]
            if len(k):
                parts.append(f([v[k] for v in g]))
                order.append(k)
        return torch.cat(parts)[torch.argsort(torch.cat(order))]

    def _coarse(self, U, l, g, slopes):
        c = [v >> 1 for v in g]
        Uc = self._load(U, self._leaf(l - 1, c), c)
        if not slopes:
            return Uc
        v = Uc
        for a in range(3):
            e = []
            for s in (-1, 1):
                h = list(c)
                h[a] = h[a] + s
                e.append(self._value(U, l - 1, self._bound(l - 1, h), False))
            lo, hi = Uc - e[0], e[1] - Uc
            d = torch.where(lo * hi > 0, torch.where(lo.abs() <= hi.abs(), lo, hi), torch.zeros_like(lo))
            v = v + 0.25 * (2.0 * (g[a] & 1).double() - 1.0)[:, None] * d
        return v

    def padded(self, U, at=None):
        """U[B, fields, n, n, n] with its ghost layers; `at`: of these leaves only."""
        n, N = self.n, self.n + 2 * G
        at = torch.arange(len(self.lv), device=self.dev) if at is None else at
        out = []
        r = torch.arange(N, device=self.dev) - G
        for part in at.split(max(1, 4_000_000 // N ** 3)):
            block = torch.empty((len(part), N ** 3, U.shape[1]), dtype=U.dtype, device=self.dev)
            pieces, order = [], []
            for l in self.lv[part, 0].unique().tolist():
                k = torch.nonzero(self.lv[part, 0] == l)[:, 0]
                q = [self.lv[part[k], 1 + a].view(-1, 1) * n + r for a in range(3)]
                q = [q[0][:, None, None, :].expand(-1, N, N, N), q[1][:, None, :, None].expand(-1, N, N, N),
                     q[2][:, :, None, None].expand(-1, N, N, N)]
                v = self._value(U, l, self._bound(l, [x.reshape(-1) for x in q]), True)
                pieces.append(v.view(len(k), N ** 3, -1))
                order.append(k)
            block = torch.cat(pieces)[torch.argsort(torch.cat(order))]
            out.append(block.transpose(1, 2).reshape(len(part), U.shape[1], N, N, N))
        return torch.cat(out)

    def step(self, U, dt, cycle):
        n = self.n
        parts, faces = [], []
        for at in torch.arange(len(self.lv), device=self.dev).split(max(1, 3_000_000 // (n + 2 * G) ** 3)):
            P = self.padded(U, at)
            dtdx = (dt / self.dx[at]).view(-1, 1, 1, 1)
            fx = [None] * 3
            for axis in (0, 1, 2) if cycle % 2 == 0 else (2, 1, 0):
                P, fx[axis] = self._sweep(P, axis, dtdx)
            parts.append(_interior(P, n))
            faces.append(fx)
        V = torch.cat(parts)
        if self.case["levels"] == 0:
            return V
        flux = [[torch.cat([f[a][s] for f in faces]) for s in (0, 1)] for a in range(3)]    # [B, fields, t2, t1]
        for axis in range(3):
            for s in (0, 1):
                V = self._correct(V, flux, axis, s, dt)
        return V

    def _correct(self, V, flux, axis, s, dt):
        n, R = self.n, self.case["root"]
        t1, t2 = (1, 2) if axis == 0 else ((0, 2) if axis == 1 else (0, 1))
        for l in range(self.case["levels"]):
            b = torch.nonzero(self.lv[:, 0] == l)[:, 0]
            ijk = [self.lv[b, 1 + a].clone() for a in range(3)]
            ijk[axis] = ijk[axis] + (1 if s else -1)
            inside = (ijk[axis] >= 0) & (ijk[axis] < (R << l)) | _periodic(self.case)[axis]
            ijk[axis] = torch.remainder(ijk[axis], R << l)
            c = [2 * v for v in ijk]
            c[axis] = c[axis] + (0 if s else 1)
            k = torch.nonzero(inside & (self.maps[l + 1][c[2], c[1], c[0]] >= 0))[:, 0]
            if not len(k):
                continue
            rows = []
            for o2 in (0, 1):
                row = []
                for o1 in (0, 1):
                    h = [v[k].clone() for v in c]
                    h[t1] = h[t1] + o1
                    h[t2] = h[t2] + o2
                    f = flux[axis][1 - s][self.maps[l + 1][h[2], h[1], h[0]]]
                    row.append(f.reshape(len(k), -1, n // 2, 2, n // 2, 2).mean((3, 5)))
                rows.append(torch.cat(row, 3))
            mean = torch.cat(rows, 2)
            d = (dt / self.dx[b[k]]).view(-1, 1, 1, 1) * (flux[axis][s][b[k]] - mean) * (1.0 if s else -1.0)
            W = V.movedim(4 - axis, -1)      # view: [B, fields, t2, t1, axis]
            W[b[k], :, :, :, n - 1 if s else 0] += d
        return V

    def reduce(self, U):
        g = self.gamma
        h, tot = math.inf, 0.0
        for at in torch.arange(len(self.lv), device=self.dev).split(512):
            rho, m, E = U[at, 0], U[at, 1:4], U[at, 4]
            v = m / rho[:, None]
            src = E - 0.5 * rho * (v * v).sum(1)
            if self.case.get("dual"):
                src = torch.where(src > 1e-3 * E, src, U[at, 5])
            c = torch.sqrt(g * (g - 1.0) * src / rho)
            h = min(h, float((self.dx[at].view(-1, 1, 1, 1) / (v.abs().amax(1) + c)).min()))
            tot = tot + (U[at, :5].sum((2, 3, 4)) * (self.dx[at] ** 3)[:, None]).sum(0)
        return h, tot

    # --------------------------------------------------------------- one PPM sweep
    def _primitive(self, q):
        rho = q[0].clamp_min(1e-10)
        v = [m / rho for m in q[1:4]]
        src = q[4] - 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        if len(q) == 6:
            src = torch.where(src > 1e-3 * q[4], src, q[5])
        p = ((self.gamma - 1.0) * src).clamp_min(1e-20)
        return [rho, *v, p] + ([q[5] / rho] if len(q) == 6 else [])

    def _sweep(self, P, axis, dtdx):
        n, N, case = self.n, self.n + 2 * G, self.case
        comp = self.axes[axis][:P.shape[1]]
        V = P.movedim(4 - axis, -1)
        q = [V[:, k] for k in comp]
        W = self._primitive(q)
        F, uf = self._fluxes(W, dtdx)               # interfaces 3+1/2 .. N-5+1/2
        new = [None] * len(comp)
        for k, f in enumerate(F):
            new[k] = q[k][..., G:G + n] - dtdx * (f[..., 1:] - f[..., :-1])
        if len(comp) == 6:
            new[5] = new[5] - dtdx * W[4][..., G:G + n] * (uf[..., 1:] - uf[..., :-1])
            rho = new[0].clamp_min(1e-10)
            ei = new[4] - 0.5 * (new[1] ** 2 + new[2] ** 2 + new[3] ** 2) / rho
            new[5] = torch.where(ei > 0.1 * new[4], ei, new[5])
        inv = [comp.index(k) for k in range(len(comp))]
        new = torch.stack([new[i] for i in inv], 1)
        Q = torch.cat([V[..., :G], new, V[..., G + n:]], -1).movedim(-1, 4 - axis)
        face = [torch.stack([F[i][:, G:G + n, G:G + n, e] for i in inv], 1) for e in (0, n)]
        return Q, face

    def _fluxes(self, W, dtdx):
        case = self.case
        N = W[0].shape[-1]
        c = lambda a, lo, hi: a[..., lo:hi]  # noqa: E731
        zero = torch.zeros((), dtype=torch.float64, device=W[0].device)
        dm, ai = [], []
        for a in W:
            dl, dr = a[..., 1:-1] - a[..., :-2], a[..., 2:] - a[..., 1:-1]
            m = torch.minimum(0.5 * (dl + dr).abs(), 2.0 * torch.minimum(dl.abs(), dr.abs()))
            dm.append(torch.where(dl * dr > 0, torch.sign(dl) * m, zero))                   # cells 1 .. N-2
            ai.append(0.5 * (a[..., 1:N - 2] + a[..., 2:N - 1]) - (dm[-1][..., 1:] - dm[-1][..., :-1]) / 6.0)
        p, un = W[4], W[1]
        d1, d2 = c(p, 3, N - 1) - c(p, 1, N - 3), c(p, 4, N) - c(p, 0, N - 4)
        hit = ((d1.abs() > 0.33 * torch.minimum(c(p, 3, N - 1), c(p, 1, N - 3)))
               & (c(un, 1, N - 3) > c(un, 3, N - 1)) & (d2 != 0))
        ft = torch.where(hit, (10.0 * (d1 / torch.where(d2 != 0, d2, zero + 1) - 0.75)).clamp(0.0, 1.0), zero)
        s = c(p, 4, N - 2) - c(p, 2, N - 4)
        f0, fm, fp = c(ft, 1, N - 5), c(ft, 0, N - 6), c(ft, 2, N - 4)
        flat = torch.where(s > 0, torch.maximum(f0, fm), torch.where(s < 0, torch.maximum(f0, fp), f0))
        Wc, aL, aR = [c(a, 3, N - 3) for a in W], [], []
        for k, a in enumerate(Wc):
            l, r = c(ai[k], 1, N - 5), c(ai[k], 2, N - 4)
            if k == 0 and case.get("steepening"):
                rho = W[0]
                Dm = c(rho, 3, N - 3) - 2 * c(rho, 2, N - 4) + c(rho, 1, N - 5)
                Dp = c(rho, 5, N - 1) - 2 * c(rho, 4, N - 2) + c(rho, 3, N - 3)
                rm, rp, pm, pp = c(rho, 2, N - 4), c(rho, 4, N - 2), c(p, 2, N - 4), c(p, 4, N - 2)
                dr = rp - rm
                off = ((Dp * Dm > 0) | (dr.abs() < 0.01 * torch.minimum(rp.abs(), rm.abs()))
                       | (self.gamma * 0.1 * dr.abs() / torch.minimum(rp, rm)
                          < (pp - pm).abs() / torch.minimum(pp, pm)))
                eta = torch.where(off, zero, -(Dp - Dm) / (6.0 * torch.where(off, zero + 1, dr)))
                eta = (20.0 * (eta - 0.05)).clamp(0.0, 1.0)
                l = l * (1 - eta) + (rm + 0.5 * c(dm[0], 1, N - 5)) * eta
                r = r * (1 - eta) + (rp - 0.5 * c(dm[0], 3, N - 3)) * eta
            l, r = flat * a + (1 - flat) * l, flat * a + (1 - flat) * r
            d, mid = r - l, a - 0.5 * (l + r)
            ext = (r - a) * (a - l) <= 0
            aL.append(torch.where(ext, a, torch.where(d * mid > d * d / 6.0, 3 * a - 2 * r, l)))
            aR.append(torch.where(ext, a, torch.where(-d * d / 6.0 > d * mid, 3 * a - 2 * l, r)))
        Wm, Wp = self._trace(Wc, aL, aR, dtdx, zero)
        solve = self._hllc if case.get("hllc") else self._two_shock
        return solve([c(x, 0, N - 7) for x in Wp], [c(x, 1, N - 6) for x in Wm], zero)

    def _trace(self, W, aL, aR, dtdx, zero):
        rho, un, p = W[0], W[1], W[4]
        csq = self.gamma * p / rho
        cs = torch.sqrt(csq)
        a6 = [6.0 * (w - 0.5 * (l + r)) for w, l, r in zip(W, aL, aR)]
        out = []
        for side in (-1, 1):        # left edge (waves moving left), right edge (waves moving right)
            edge = aR if side > 0 else aL

            def avg(k, lam):        # mean of the parabola over what the wave carries to the edge
                x = (side * lam * dtdx)
                return edge[k] - side * 0.5 * x * ((aR[k] - aL[k]) - side * (1.0 - 2.0 / 3.0 * x) * a6[k])

            fast, slow = un + side * cs, un - side * cs
            gone = side * fast > 0
            ref = [torch.where(gone, avg(k, fast), edge[k]) for k in range(len(W))]
            back, still = side * slow > 0, side * un > 0
            beta = torch.where(back, (ref[4] - avg(4, slow)) * 0.5 / csq
                               - side * (ref[1] - avg(1, slow)) * 0.5 * rho / cs, zero)
            b0 = torch.where(still, (ref[0] - avg(0, un)) - (ref[4] - avg(4, un)) / csq, zero)
            st = [(ref[0] - (b0 + beta)).clamp_min(1e-10), ref[1] + side * cs / rho * beta,
                  None, None, (ref[4] - csq * beta).clamp_min(1e-20)]
            for k in (2, 3):
                st[k] = torch.where(still, avg(k, un), ref[k])
            st += [torch.where(still, avg(k, un), ref[k]) for k in range(5, len(W))]
            out.append(st)
        return out

    def _flux_of(self, r, u, t, p, e):
        E = p / (self.gamma - 1.0) + 0.5 * r * (u * u + t[0] * t[0] + t[1] * t[1])
        return [r * u, r * u * u + p, r * u * t[0], r * u * t[1], u * (E + p)] + [r * u * x for x in e], E

    def _two_shock(self, L, R, zero):
        g = self.gamma
        g1 = (g + 1.0) / (2.0 * g)
        (rL, uL, pL), (rR, uR, pR) = ((S[0], S[1], S[4]) for S in (L, R))
        CL, CR = torch.sqrt(g * pL * rL), torch.sqrt(g * pR * rR)
        ps = ((CR * pL + CL * pR + CL * CR * (uL - uR)) / (CL + CR)).clamp_min(1e-20)
        for it in range(6):
            WL, WR = CL * torch.sqrt(1 + g1 * (ps / pL - 1)), CR * torch.sqrt(1 + g1 * (ps / pR - 1))
            vL, vR = uL - (ps - pL) / WL, uR + (ps - pR) / WR
            ZL, ZR = 2 * WL ** 3 / (WL * WL + CL * CL), 2 * WR ** 3 / (WR * WR + CR * CR)
            if it < 5:
                ps = (ps - ZL * ZR * (vR - vL) / (ZL + ZR)).clamp_min(1e-20)
        us = (ZL * vL + ZR * vR) / (ZL + ZR)
        left = us >= 0
        pick = lambda a, b: torch.where(left, a, b)  # noqa: E731
        r0, u0, p0, W0 = pick(rL, rR), pick(uL, uR), pick(pL, pR), pick(WL, WR)
        t, e = [pick(L[k], R[k]) for k in (2, 3)], [pick(L[k], R[k]) for k in range(5, len(L))]
        sg = torch.where(left, zero - 1, zero + 1)
        tau = 1 / r0 - (ps - p0) / (W0 * W0)
        rs = torch.where(tau > 0, 1 / torch.where(tau > 0, tau, zero + 1), zero + 1e-10).clamp_min(1e-10)
        c0, cs = torch.sqrt(g * p0 / r0), torch.sqrt(g * ps / rs)
        shock = ps > p0
        head = torch.where(shock, sg * u0 + W0 / r0, sg * u0 + c0)
        tail = torch.where(shock, head, sg * us + cs)
        outer = head <= 0
        star = ~outer & (tail > 0)
        w = head / torch.where(outer | star, zero + 1, head - tail)
        w = torch.where(outer, zero, torch.where(star, zero + 1, w))
        r, u, p = (torch.where(star, b, a + w * (b - a)) for a, b in ((r0, rs), (u0, us), (p0, ps)))
        return self._flux_of(r, u, t, p, e)[0], u

    def _hllc(self, L, R, zero):
        g = self.gamma
        cL, cR = torch.sqrt(g * L[4] / L[0]), torch.sqrt(g * R[4] / R[0])
        SL, SR = torch.minimum(L[1] - cL, R[1] - cR), torch.maximum(L[1] + cL, R[1] + cR)
        mL, mR = L[0] * (SL - L[1]), R[0] * (SR - R[1])
        Ss = ((R[4] - L[4]) + (mL * L[1] - mR * R[1])) / (mL - mR)
        left = (SL >= 0) | (Ss >= 0)
        K = [torch.where(left, a, b) for a, b in zip(L, R)]
        S, m = torch.where(left, SL, SR), torch.where(left, mL, mR)
        F, E = self._flux_of(K[0], K[1], K[2:4], K[4], K[5:])
        outer = torch.where(left, SL >= 0, ~(SR > 0))
        fac = m / (S - Ss)
        Us = [fac, fac * Ss, fac * K[2], fac * K[3], fac * (E / K[0] + (Ss - K[1]) * (Ss + K[4] / m))]
        Us += [fac * e for e in K[5:]]
        Uc = [K[0], K[0] * K[1], K[0] * K[2], K[0] * K[3], E] + [K[0] * e for e in K[5:]]
        F = [torch.where(outer, f, f + S * (a - b)) for f, a, b in zip(F, Us, Uc)]
        return F, torch.where(outer, K[1], Ss)
