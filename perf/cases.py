"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values.  `kind` says which call it is:

  step     one or more time steps of a discrete-velocity flow on a tree
           (transport, moments, collision), as the time loop of a run makes
           them; `coll` is bgk, entropic, none, hs (hard-sphere collision
           integral) or learned (network operator with hard-sphere fallback);
  fields   the macroscopic fields and the kinetic/fluid flags of a stored
           flow, as a run reads them between steps;
  lbm      a block of lattice Boltzmann steps and the fields after it;
  mlp      loss and gradient of the collision network on a batch of pairs,
           one evaluation of its training.

`exact` restates each call in 64 bits with plain torch: the tree from its
specification, the upwind stencils on it, and the arithmetic.
"""
import functools
import math

import numpy as np
import torch

import paper_1503_00707_gb300 as D

TABLE_SEED = 20150303
GAMMA = 5.0 / 3.0
PREC = {"f64": D.F64, "f32": D.F32, "bf16": D.BF16}
TYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
ESIZE = {"f64": 8, "f32": 4, "bf16": 2}
COLL = {"none": D.COLL_NONE, "bgk": D.COLL_BGK, "entropic": D.COLL_BGK_ENTROPIC, "hs": D.COLL_HS,
        "learned": D.COLL_LEARNED}
LAYERS = ((64, 256), (256, 256), (256, 256), (256, 64))


def _flow(name, tree, nx, ny, nz, vmax, mach, kn, prec, coll, steps, **more):
    return dict(name=name, kind="step", tree=tree, nx=nx, ny=ny, nz=nz, vmax=vmax, mach=mach, kn=kn, prec=prec,
                coll=coll, steps=steps, trials=0, fields=False, **more)


def listed():
    sphere = dict(dim=3, r=0.1, beta=3.0)
    return [
        # the smallest run: 2D periodic quadtree (904 cells x 8^3) with a density bump, FP64, a block of steps and
        # its fields: what a first test or a parameter scan does, where launches and latency count
        dict(_flow("bump2d_f64", "bump", 8, 8, 8, 4.0, 0.0, 0.05, "f64", "bgk", 10, dim=2, base=4, top=6, r=0.2,
                   beta=0.0), fields=True),
        # an ordinary rarefied run: Mach-3 sphere flow, 27k cells x 16^3, FP32
        _flow("sphere16_f32", "sphere", 16, 16, 16, 6.0, 3.0, 0.1, "f32", "bgk", 4, dim=3, base=4, top=6, r=0.15,
              beta=3.25),
        # the production flow: Mach-5 sphere, 159k cells x 24^3 (8.8 GB a buffer), FP32 and BF16 storage
        _flow("sphere24_f32", "sphere", 24, 24, 24, 8.0, 5.0, 0.01, "f32", "bgk", 1, dim=3, base=5, top=7, r=0.1,
              beta=7.5),
        _flow("sphere24_bf16", "sphere", 24, 24, 24, 8.0, 5.0, 0.01, "bf16", "bgk", 1, dim=3, base=5, top=7, r=0.1,
              beta=7.5),
        # relaxation towards the entropic equilibrium, 18k cells x 24^3
        _flow("sphere24_entropic", "sphere", 24, 24, 24, 8.0, 5.0, 0.01, "f32", "entropic", 1, base=4, top=6,
              **sphere),
        # the hard-sphere collision integral: the homogeneous-relaxation box (16.6k cells x 16^3) and the Mach-3
        # flow (12k cells x 24^3)
        dict(_flow("hs_box16", "box", 16, 16, 16, 6.0, 0.0, 0.02, "f32", "hs", 1, dim=3, base=4, top=5, r=0.42,
                   beta=0.0), trials=128),
        dict(_flow("hs_sphere24", "sphere", 24, 24, 24, 8.0, 3.0, 0.003, "f32", "hs", 1, dim=3, base=3, top=5, r=0.15,
                   beta=3.5), trials=128),
        # the learned operator where the local Knudsen number allows it, the hard-sphere integral elsewhere
        dict(_flow("learned_sphere24", "sphere", 24, 24, 24, 8.0, 3.0, 0.003, "f32", "learned", 1, dim=3, base=3,
                   top=5, r=0.15, beta=3.5), trials=128),
        # output of a run: fields and kinetic flags of 18k cells x 24^3
        dict(kind="fields", name="fields24_f32", tree="sphere", dim=3, base=4, top=6, r=0.1, beta=3.0, nx=24, ny=24,
             nz=24, vmax=8.0, mach=5.0, kn=0.01, prec="f32", coll="bgk"),
        # lattice Boltzmann: a small 2D flow around a disk (FP64), f read back for a checkpoint, and the Ma-0.5 sphere
        # on 602k cells (FP32)
        dict(kind="lbm", name="lbm_disk_q9", tree="disk", dim=2, base=4, top=7, r=0.1, beta=3.0, lattice=9,
             prec="f64", speed=0.1, omega=0.5, steps=30, whole=True),
        dict(kind="lbm", name="lbm_sphere_q19", tree="sphere", dim=3, base=6, top=9, r=0.1, beta=3.0, lattice=19,
             prec="f32", speed=0.5 / math.sqrt(3.0), omega=0.85, steps=100, whole=False),
        # training of the collision network
        dict(kind="mlp", name="mlp_grad", rows=8192),
    ]


def draw(rng):
    def grid(most, unit):
        """(nx, ny, nz, vmax, mach): a node spacing of about 1, and a stream that the grid holds."""
        while True:
            nx, ny, nz = 2 * rng.randint(4, 12), 2 * rng.randint(4, 12), unit * rng.randint(8 // unit, 24 // unit)
            if nx * ny * nz <= most:
                vmax = min(8.0, 0.5 * min(nx, ny, nz))
                return nx, ny, nz, vmax, round(rng.uniform(0.0, max(0.2, (vmax - 4.0) / 1.3)), 2)

    def tree():
        # cells of a sphere tree: about 8^base plus a band; the bases and tops below stay under 30k
        base, top = rng.choice(((2, 4), (3, 4), (3, 5), (3, 6), (4, 5), (4, 6)))
        return dict(base=base, top=top, r=round(rng.uniform(0.08, 0.15), 3), beta=round(rng.uniform(1.5, 3.0), 2))

    what = rng.choice(("step", "step", "step", "plane", "hs", "hs", "learned", "fields", "lbm", "lbm", "mlp"))
    if what == "step":
        prec = rng.choice(("f32", "f32", "bf16", "bf16", "f64"))
        nx, ny, nz, vmax, mach = grid(4096 if prec == "f64" else 13824, 4 if prec == "f64" else 8)
        return _flow("", "sphere", nx, ny, nz, vmax, mach, round(math.exp(rng.uniform(math.log(0.02), 0.0)), 4), prec,
                     rng.choice(("bgk", "bgk", "entropic", "none")), rng.randint(1, 3), dim=3, **tree())
    if what == "plane":
        nx, ny, nz, vmax, _ = grid(4096, 8)
        return dict(_flow("", "bump", nx, ny, nz, vmax, 0.0, round(rng.uniform(0.05, 1.0), 3),
                          rng.choice(("f64", "f32")), "bgk", rng.randint(1, 20), dim=2, base=rng.randint(3, 5),
                          top=rng.randint(5, 7), r=round(rng.uniform(0.1, 0.3), 3), beta=0.0))
    if what == "hs":
        # the node spacing is the same on every axis
        n = rng.choice((8, 16, 16, 24))
        t = tree()
        t["top"] = min(t["top"], 5)
        t["base"] = min(t["base"], 3)
        return dict(_flow("", "sphere", rng.choice((n, n, n - 2)), n, n, 0.375 * n if n > 8 else 4.0,
                          round(rng.uniform(0.1, 1.5), 2), round(rng.uniform(0.003, 0.1), 4), "f32", "hs", 1, dim=3,
                          **t), trials=rng.choice((32, 64, 128)))
    if what == "learned":
        n = rng.choice((8, 16, 16))
        t = tree()
        t["top"] = min(t["top"], 5)
        t["base"] = min(t["base"], 3)
        return dict(_flow("", "sphere", n, n, n, 0.375 * n if n > 8 else 4.0, round(rng.uniform(0.1, 1.5), 2),
                          round(rng.uniform(0.002, 0.01), 4), "f32", "learned", 1, dim=3, **t),
                    trials=rng.choice((32, 64, 128)))
    if what == "fields":
        prec = rng.choice(("f32", "bf16", "f64"))
        nx, ny, nz, vmax, mach = grid(4096 if prec == "f64" else 13824, 4 if prec == "f64" else 8)
        return dict(kind="fields", name="", tree="sphere", dim=3, nx=nx, ny=ny, nz=nz, vmax=vmax, mach=mach, kn=0.05,
                    prec=prec, coll="bgk", **tree())
    if what == "lbm":
        if rng.random() < 0.3:
            return dict(kind="lbm", name="", tree="disk", dim=2, base=rng.randint(3, 5), top=rng.randint(6, 8),
                        r=round(rng.uniform(0.08, 0.2), 3), beta=3.0, lattice=9, prec=rng.choice(("f64", "f32")),
                        speed=0.1, omega=round(rng.uniform(0.2, 0.9), 2), steps=rng.randint(5, 100), whole=True)
        base, top = rng.choice(((3, 5), (4, 6), (4, 7), (5, 7), (5, 8), (6, 8)))
        return dict(kind="lbm", name="", tree="sphere", dim=3, base=base, top=top, r=round(rng.uniform(0.08, 0.12), 3),
                    beta=3.0, lattice=rng.choice((19, 27)), prec=rng.choice(("f32", "f32", "f64")), speed=0.25,
                    omega=round(rng.uniform(0.2, 0.85), 2), steps=rng.randint(10, 60), whole=False)
    return dict(kind="mlp", name="", rows=int(math.exp(rng.uniform(math.log(100), math.log(60000)))))


# ---------------------------------------------------------------- inputs

def _bc(case):
    # periodic box; disk: inflow, outflow, periodic in y; sphere: inflow at x = 0, outflow elsewhere
    return {"bump": (0,) * 6, "box": (0,) * 6, "disk": (1, 2, 0, 0, 0, 0), "sphere": (1, 2, 2, 2, 2, 2)}[case["tree"]]


def _spec(case):
    ball = case["tree"] in ("bump", "box")
    return dict(dim=case["dim"], base_level=case["base"], max_level=max(case["base"], case["top"]),
                pred=D.PRED_BALL if ball else D.PRED_SHELL, c=(0.5, 0.5, 0.5), r=case["r"], beta=case["beta"],
                solid=0 if ball else 1, bc=_bc(case))


def _axes(case):
    """(n, hi): nodes and half-width of each velocity axis; hard-sphere grids have one spacing."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["coll"] in ("hs", "learned"):
        h = 2.0 * case["vmax"] / case["nz"]
        return n, tuple(0.5 * h * k for k in n)
    return n, (case["vmax"],) * 3


def _config(case):
    n, hi = _axes(case)
    u = (case["mach"] * math.sqrt(GAMMA), 0.0, 0.0)
    return dict(_spec(case), n=n, lo=tuple(-h for h in hi), hi=hi, fs_rho=1.0, fs_u=u, fs_T=1.0,
                coll=COLL[case["coll"]], kn=case["kn"], precision=case["prec"])


def _start(case, nc, xyz, seed):
    """Maxwellian mixture (w, rho, u, T) of every cell: the flow's start with seeded cell-wise perturbations."""
    g = np.random.default_rng(seed)
    if case["tree"] == "box":  # two beams of seeded weights, directions, speeds and temperatures
        w1, z, ph = g.uniform(0.3, 0.7, nc), g.uniform(-1, 1, nc), g.uniform(0, 2 * math.pi, nc)
        a = g.uniform(1.0, 2.0, (2, nc))
        st = np.sqrt(1 - z * z)
        d = np.stack([st * np.cos(ph), st * np.sin(ph), z], 1)
        return (np.stack([w1, 1 - w1], 1), np.ones((nc, 2)), np.stack([a[0][:, None] * d, -a[1][:, None] * d], 1),
                g.uniform(0.4, 0.8, (nc, 2)))
    if case["coll"] in ("hs", "learned"):  # two opposite beams, 5% perturbed: away from equilibrium everywhere
        e = 0.05
        w1 = 0.5 * (1 + e * g.uniform(-1, 1, nc))
        a = 1.5 * (1 + e * g.uniform(-1, 1, (2, nc)))
        d = np.stack([np.ones(nc), e * g.uniform(-1, 1, nc), e * g.uniform(-1, 1, nc)], 1)
        return (np.stack([w1, 1 - w1], 1), np.ones((nc, 2)), np.stack([a[0][:, None] * d, -a[1][:, None] * d], 1),
                0.6 * (1 + e * g.uniform(-1, 1, (nc, 2))))
    rho = 1 + 0.05 * g.uniform(-1, 1, (nc, 1))
    if case["tree"] == "bump":
        r2 = ((xyz[:, :2] - 0.5) ** 2).sum(1)
        rho += 0.2 * np.exp(-r2 / 0.01)[:, None]
    u = 0.05 * g.uniform(-1, 1, (nc, 1, 3))
    u[:, 0, 0] += case["mach"] * math.sqrt(GAMMA)
    return np.ones((nc, 1)), rho, u, 1 + 0.05 * g.uniform(-1, 1, (nc, 1))


def _dt(case, cfl_dt):
    if case["coll"] in ("hs", "learned"):  # dt/Kn max(P B) stays below 1
        return min(cfl_dt / 16, case["kn"] / 1000)
    # nu dt stays below 1 behind the bow shock: rho up to 4, T up to 1 + M^2 / 3
    return min(cfl_dt, 0.5 * case["kn"] / (1.6 * 4 * math.sqrt(1 + case["mach"] ** 2 / 3)))


def _weights(seed):
    """A network near the relaxation a -> -0.3 a: SiLU units in pairs (silu(z) - silu(-z) = z) carry the modes, the
    other units and a seeded perturbation of every weight make the rest of a trained network's work."""
    g = np.random.default_rng(seed + 17)
    eye, parts = np.eye(64), []
    for k, (i, o) in enumerate(LAYERS):
        w = g.standard_normal((o, i)) * 0.002
        pair = np.concatenate([eye, -eye])
        if k == 0:
            w[:128, :64] += pair
        elif k < 3:
            w[:128, :128] += np.concatenate([pair, -pair], 1)
        else:
            w[:, :128] += -0.3 * pair.T
        parts += [w.ravel(), g.standard_normal(o) * 0.002]
    return np.concatenate(parts).astype(np.float32)


def _pairs(rows, seed):
    """Projections of perturbed Maxwellians on the Hermite modes (1 in the first, small elsewhere) and their
    relaxation, with noise."""
    g = np.random.default_rng(seed)
    x = g.standard_normal((rows, 64)) * (0.3 / (1.0 + np.arange(64) / 8.0))
    x[:, 0] = 1.0
    t = -0.4 * x + 0.05 * g.standard_normal((rows, 64))
    return x.astype(np.float32), t.astype(np.float32)


class _DeviceF:
    """One of a solver's f buffers as torch sees device memory; keeps the solver, which owns it, alive."""

    def __init__(self, solver, ptr, prec):
        kind = {"f64": "<f8", "f32": "<f4", "bf16": "<i2"}[prec]
        self.solver = solver
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (solver.ncells, solver.nv), "typestr": kind,
                                         "version": 3}


class _Flow:
    """A solver and the views of its two f buffers."""

    def __init__(self, solver, case):
        self.solver, self.prec, self.views = solver, case["prec"], {}

    def f(self):
        ptr = self.solver.f_device_ptr()[0]
        if ptr not in self.views:
            t = torch.as_tensor(_DeviceF(self.solver, ptr, self.prec), device="cuda")
            self.views[ptr] = t.view(torch.bfloat16) if self.prec == "bf16" else t
        return self.views[ptr]


def _lbm_config(case):
    return dict(_spec(case), lattice=case["lattice"], fs_rho=1.0, fs_u=(case["speed"], 0.0, 0.0),
                precision=case["prec"])


def _lbm_start(case, nc, seed):
    g = np.random.default_rng(seed)
    u = np.zeros((nc, 3))
    u[:, 0] = case["speed"]
    u[:, :case["dim"]] += 0.02 * g.uniform(-1, 1, (nc, case["dim"]))
    return 1 + 0.02 * g.uniform(-1, 1, nc), u


def prepare(case, seed):
    if case["kind"] == "mlp":
        s = D.Solver(D.F32, D.COLL_NONE, 1.0)
        g = np.random.default_rng(seed + 5)
        s.set_weights(np.concatenate([np.concatenate([g.standard_normal(i * o) / math.sqrt(i), np.zeros(o)])
                                      for i, o in LAYERS]))
        x, t = _pairs(case["rows"], seed)
        return dict(kind="mlp", solver=s, x=x, t=t)
    if case["kind"] == "lbm":
        s = D.lbm_solver_from_config(_lbm_config(case))
        dt = s.lbm_dt_cfl(0.3)
        s.lbm_init(*_lbm_start(case, s.ncells, seed))
        return dict(kind="lbm", solver=s, steps=case["steps"], dt=dt, tau=dt / case["omega"],
                    whole=case["whole"])
    s = D.solver_from_config(_config(case))
    s.init_maxwellian(*_start(case, s.ncells, s.centres()[0], seed))
    if case["kind"] == "fields":
        return dict(kind="fields", solver=s)
    if case["trials"]:
        s.set_collision_tables(case["trials"], TABLE_SEED)
    if case["coll"] == "learned":
        s.set_weights(_weights(seed))
        s.learned_configure(0.05)
    return dict(kind="step", solver=s, flow=_Flow(s, case), steps=case["steps"], dt=_dt(case, s.dt_cfl(0.4)),
                fields=case["fields"])


def run(state):
    s = state["solver"]
    if state["kind"] == "mlp":
        loss, grad = s.mlp_loss_grad(state["x"], state["t"])
        return {"loss": loss, "grad": grad}
    if state["kind"] == "lbm":
        s.lbm_step(state["steps"], state["dt"], state["tau"])
        rho, u = s.lbm_moments()
        return {"rho": rho, "u": u, "f": s.lbm_get_f()} if state["whole"] else {"rho": rho, "u": u}
    if state["kind"] == "fields":
        rho, u, temp = s.moments()
        flags, count = s.flag_kinetic(0.05)
        return {"rho": rho, "u": u, "T": temp, "kinetic": flags, "count": count}
    s.step(state["steps"], state["dt"])
    if state["fields"]:
        rho, u, temp = s.step_moments()
        return {"f": state["flow"].f(), "rho": rho, "u": u, "T": temp}
    return {"f": state["flow"].f()}


# ---------------------------------------------------------------- what a pass cannot do without

@functools.lru_cache(maxsize=None)
def _cells(spec):
    s = D.Solver(D.F32, D.COLL_NONE, 1.0)
    s.build_tree(D.tree_spec(**dict(spec)))
    return s.ncells


def work(case):
    """f read and written once a step; a fields pass reads f and writes its fields; hard-sphere trials take five
    operations (those with a weight), BGK about 30 a value, a projection or reconstruction of the learned term
    about 30."""
    if case["kind"] == "mlp":
        macs = sum(i * o for i, o in LAYERS)
        return {"bytes": case["rows"] * 64 * 8 + D.MLP_NPARAM * 8, "flops": 6.0 * macs * case["rows"]}
    nc = _cells(tuple(sorted(_spec(case).items())))
    es = ESIZE[case["prec"]]
    if case["kind"] == "lbm":
        values = nc * case["lattice"] * case["steps"]
        return {"bytes": values * 2 * es + nc * (32 + 8 * case["lattice"] * case["whole"]), "flops": values * 30.0}
    values = nc * case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "fields":
        return {"bytes": values * es + nc * 48, "flops": values * 13.0}
    out = nc * 40 if case["fields"] else 0
    ops = 30.0
    if case["coll"] in ("hs", "learned"):
        weights = _tables(*_axes(case)[0], _axes(case)[1], case["trials"])[3]
        ops += 5.0 * case["trials"] * float((weights != 0).mean())
    return {"bytes": case["steps"] * values * 2 * es + out, "flops": case["steps"] * values * ops}


# ---------------------------------------------------------------- 64 bits

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grow(a, per):
    """OR of a boolean grid over the neighbours of every box, diagonal ones too (wrapped where periodic)."""
    for d in range(a.dim()):
        b = a.clone()
        for sh in (1, -1):
            r = torch.roll(a, sh, d)
            if not per[d]:
                r = r.clone()
                r.select(d, 0 if sh == 1 else a.shape[d] - 1).zero_()
            b |= r
        a = b
    return a


def _pool(a):
    for d in range(a.dim()):
        s = list(a.shape)
        s[d:d + 1] = [s[d] // 2, 2]
        a = a.reshape(s).any(d + 1)
    return a


def _repeat(a):
    for d in range(a.dim()):
        a = a.repeat_interleave(2, d)
    return a


@functools.lru_cache(maxsize=1)
def _mesh(spec):
    """The balanced tree: (xyz, h, sources [cell][2 dim][K], their weights as shares of the side, wall marks).  A
    source is a cell, the cell itself at an outflow or wall, or the inflow ghost (number ncells)."""
    s, dev = dict(spec), _dev()
    dim, base, top, bc = s["dim"], s["base_level"], s["max_level"], s["bc"]
    per = [bc[2 * d] == D.BC_PERIODIC for d in range(dim)]
    cen = torch.tensor(s["c"][:dim], dtype=torch.float64, device=dev)

    def boxes(lev):
        return torch.stack(torch.meshgrid(*[torch.arange(2 ** lev, device=dev)] * dim, indexing="ij"), -1)

    split, exists = [], torch.ones((1,) * dim, dtype=torch.bool, device=dev)
    for lev in range(top):
        if lev < base:
            want = torch.ones_like(exists)
        else:
            h, near, far = 2.0 ** -lev, 0.0, 0.0
            for d in range(dim):
                lo = torch.arange(2 ** lev, device=dev, dtype=torch.float64) * h
                hi, shape = lo + h, [1] * dim
                shape[d] = -1
                t = torch.clamp(torch.maximum(lo - cen[d], cen[d] - hi), min=0.0)
                near = near + (t * t).reshape(shape)
                far = far + torch.maximum((lo - cen[d]).abs(), (hi - cen[d]).abs()).square().reshape(shape)
            if s["pred"] == D.PRED_BALL:
                want = near <= s["r"] ** 2
            else:
                outer, inner = s["r"] + s["beta"] * h, s["r"] - s["beta"] * h
                want = near <= outer * outer
                if inner > 0:
                    want &= far >= inner * inner
        split.append(want & exists)
        exists = _repeat(split[lev])
    for lev in range(top - 2, -1, -1):
        # the neighbours of a split box at the next level all exist
        split[lev] |= _pool(_grow(split[lev + 1], per))
    leaf = []
    for lev in range(top + 1):
        e = _repeat(split[lev - 1]) if lev else torch.ones((1,) * dim, dtype=torch.bool, device=dev)
        leaf.append(e & ~split[lev] if lev < top else e)
    ix = [torch.nonzero(m) for m in leaf]
    key, lev_of = [], []
    for lev in range(top + 1):
        c, k = ix[lev] << (top - lev), torch.zeros(len(ix[lev]), dtype=torch.int64, device=dev)
        for b in range(top):
            for d in range(dim):
                k |= ((c[:, d] >> b) & 1) << (dim * b + d)
        key.append(k)
        lev_of.append(torch.full_like(k, lev))
    key, lev_of, ix_all = torch.cat(key), torch.cat(lev_of), torch.cat(ix)
    h = 2.0 ** -lev_of.double()
    xyz = (ix_all.double() + 0.5) * h[:, None]
    solid = ((xyz - cen).square().sum(1) < s["r"] ** 2) if s["solid"] else torch.zeros_like(key, dtype=torch.bool)
    order = torch.argsort(key)
    order = order[~solid[order]]
    nc = len(order)
    number = torch.full_like(key, -1)
    number[order] = torch.arange(nc, device=dev)
    # per level: cell number, -1 solid, -2 split further, -3 within a coarser leaf
    grid, at = [], 0
    for lev in range(top + 1):
        g = torch.full(leaf[lev].shape, -3, dtype=torch.int32, device=dev)
        if lev < top:
            g[split[lev]] = -2
        g[tuple(ix[lev].T)] = number[at:at + len(ix[lev])].int()
        at += len(ix[lev])
        grid.append(g)
    K = 2 ** (dim - 1)
    src = torch.arange(nc, device=dev)[:, None, None].repeat(1, 2 * dim, K)
    share = torch.zeros(nc, 2 * dim, K, dtype=torch.float64, device=dev)
    wall = torch.zeros(nc, 2 * dim, K, dtype=torch.bool, device=dev)
    cx, cl = ix_all[order], lev_of[order]
    for lev in range(top + 1):
        me = torch.nonzero(cl == lev)[:, 0]
        if not len(me):
            continue
        for d in range(dim):
            for side in range(2):
                col, nb = 2 * d + side, cx[me].clone()
                nb[:, d] += 1 if side else -1
                off = (nb[:, d] < 0) | (nb[:, d] >= 2 ** lev)
                nb[:, d] %= 2 ** lev
                share[me, col, 0] = 1.0
                edge = off & (not per[d])
                kind = bc[col]
                if kind == D.BC_INFLOW:
                    src[me[edge], col, 0] = nc
                if kind == D.BC_WALL:
                    wall[me[edge], col, 0] = True
                g = torch.where(edge, -9, grid[lev][tuple(nb.T)].long())
                if lev:
                    c = torch.nonzero(g == -3)[:, 0]
                    g[c] = grid[lev - 1][tuple((nb[c] >> 1).T)].long()
                same = g >= 0
                src[me[same], col, 0] = g[same]
                wall[me[g == -1], col, 0] = True
                f = torch.nonzero(g == -2)[:, 0]
                if len(f):
                    share[me[f], col] = 1.0 / K
                    for k in range(K):
                        c, bit = 2 * nb[f], 0
                        for e in range(dim):
                            if e == d:
                                c[:, e] += 0 if side else 1
                            else:
                                c[:, e] += (k >> bit) & 1
                                bit += 1
                        v = grid[lev + 1][tuple(c.T)].long()
                        src[me[f], col, k] = torch.where(v >= 0, v, me[f])
                        wall[me[f], col, k] = v < 0
    return xyz[order], h[order], src, share, wall


def _nodes(case):
    """Per axis the node values, by sign and distance from zero; [8][P] x 3 node values in storage order."""
    n, hi = _axes(case)
    dev = _dev()
    pos = [(torch.arange(k // 2, dtype=torch.float64, device=dev) + 0.5) * (2 * h / k) for k, h in zip(n, hi)]
    m = torch.stack(torch.meshgrid(*pos, indexing="ij"), -1).reshape(-1, 3)
    sign = torch.tensor([[1.0 if (o >> (2 - d)) & 1 else -1.0 for d in range(3)] for o in range(8)],
                        dtype=torch.float64, device=dev)
    return m, sign, math.prod(2 * h / k for k, h in zip(n, hi))


def _rows(n, size):
    return [(a, min(n, a + size)) for a in range(0, n, size)]


def _maxwell(xi, rho, u, temp):
    d2 = 0.0
    for d in range(3):
        d2 = d2 + (xi[None, :, d] - u[:, d:d + 1]).square()
    return (rho / (2 * math.pi * temp) ** 1.5)[:, None] * torch.exp(-d2 / (2 * temp[:, None]))


def _stored(case, seed):
    """The start as stored, [cells + 1][nv] (the last row the inflow ghost), in 64 bits."""
    dev = _dev()
    xyz, h = _mesh(tuple(sorted(_spec(case).items())))[:2]
    nc = len(h)
    m, sign, dv = _nodes(case)
    xi = (sign[:, None] * m[None]).reshape(-1, 3)
    xyz3 = torch.full((nc, 3), 0.5, dtype=torch.float64)
    xyz3[:, :case["dim"]] = xyz.cpu()
    w, rho, u, temp = (torch.as_tensor(np.asarray(a), device=dev) for a in _start(case, nc, xyz3.numpy(), seed))
    f = torch.empty(nc + 1, len(xi), dtype=torch.float64, device=dev)
    for a, b in _rows(nc, 4096):
        v = 0.0
        for k in range(w.shape[1]):
            v = v + w[a:b, k, None] * _maxwell(xi, rho[a:b, k], u[a:b, k], temp[a:b, k])
        f[a:b] = v.to(TYPE[case["prec"]])
    one = torch.ones(1, dtype=torch.float64, device=dev)
    stream = torch.tensor([[case["mach"] * math.sqrt(GAMMA), 0, 0]], dtype=torch.float64, device=dev)
    fs = _maxwell(xi, one, stream, one)
    f[nc] = fs[0].to(TYPE[case["prec"]])
    return f, xi, dv


def _transport(case, f, dt):
    _, h, src, share, wall = _mesh(tuple(sorted(_spec(case).items())))
    m = _nodes(case)[0]
    nc, P = len(h), len(m)
    out = torch.empty_like(f)
    out[nc] = f[nc]
    v = f.view((nc + 1) * 8, P)
    K = src.shape[2]
    for o in range(8):
        own = f.view(nc + 1, 8, P)[:nc, o]
        acc = own * (1 - (dt / h)[:, None] * m[None, :, :case["dim"]].sum(-1))
        for d in range(case["dim"]):
            bit = 1 << (2 - d)
            col = 2 * d + (0 if o & bit else 1)
            for k in range(K):
                w = dt * share[:, col, k] / h
                at = torch.nonzero(w)[:, 0] if k else None
                if at is None:
                    row = src[:, col, k] * 8 + torch.where(wall[:, col, k], o ^ bit, o)
                    acc += w[:, None] * m[None, :, d] * v[row]
                elif len(at):
                    row = src[at, col, k] * 8 + torch.where(wall[at, col, k], o ^ bit, o)
                    acc.index_add_(0, at, w[at, None] * m[None, :, d] * v[row])
        out.view(nc + 1, 8, P)[:nc, o] = acc
    return out


def _moments(f, xi, dv):
    """rho, u, T of the rows of f."""
    basis = torch.cat([torch.ones_like(xi[:, :1]), xi, xi.square().sum(1, keepdim=True)], 1)
    s = torch.cat([f[a:b] @ basis for a, b in _rows(len(f), 16384)])
    u = s[:, 1:4] / s[:, :1]
    return s[:, 0] * dv, u, (s[:, 4] / s[:, 0] - u.square().sum(1)) / 3


def _phi(c):
    """(1, c, |c|^2 - 3), [..., 5]"""
    return torch.cat([torch.ones_like(c[..., :1]), c, c.square().sum(-1, keepdim=True) - 3], -1)


def _relax(case, f, xi, dv, dt, entropic):
    nc = len(f) - 1
    size = max(1, (1 << 27) // xi.shape[0])
    for a, b in _rows(nc, size):
        rho, u, temp = _moments(f[a:b], xi, dv)
        phi = _phi((xi[None] - u[:, None]) / temp.sqrt()[:, None, None])
        target = _maxwell(xi, rho, u, temp)
        want = torch.zeros(b - a, 5, dtype=torch.float64, device=f.device)
        want[:, 0] = rho
        e = torch.zeros_like(want)
        for _ in range(12 if entropic else 1):
            now = target * torch.exp((phi @ e[..., None])[..., 0]) if entropic else target
            wp = phi * (now * dv)[..., None]
            d = torch.linalg.solve(phi.transpose(1, 2) @ wp, want - wp.sum(1))
            if not entropic or float(d.abs().max()) < 1e-11:
                break
            e += d
        now = now * (1 + (phi @ d[..., None])[..., 0])
        nu = math.sqrt(8 / math.pi) * rho * temp.sqrt() / case["kn"]
        f[a:b] += dt * nu[:, None] * (now - f[a:b])


def _mix(seed, n):
    """Draw n of the SplitMix64 stream, in [0, 1)."""
    with np.errstate(over="ignore"):
        x = np.uint64(seed) + (n.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x ^= x >> np.uint64(31)
    return (x >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


@functools.lru_cache(maxsize=2)
def _tables(nx, ny, nz, hi, trials):
    """Partner, post-collision nodes and weight of every trial of every node, [nv][trials]."""
    n = np.array([nx, ny, nz])
    h = 2.0 * np.array(hi) / n
    k = np.stack(np.meshgrid(*[np.arange(x // 2) for x in n], indexing="ij"), -1).reshape(-1, 3)
    node = np.concatenate([np.where([(o >> (2 - d)) & 1 for d in range(3)], n // 2 + k, n // 2 - 1 - k)
                           for o in range(8)])
    nv = len(node)
    where = np.empty(nv, dtype=np.int64)
    where[(node[:, 0] * ny + node[:, 1]) * nz + node[:, 2]] = np.arange(nv)
    xi = -np.array(hi) + (node + 0.5) * h
    s = np.arange(nv * trials, dtype=np.uint64) * np.uint64(3)
    gam = (_mix(TABLE_SEED, s) * nv).astype(np.int64)
    z, ph = 2 * _mix(TABLE_SEED, s + np.uint64(1)) - 1, 2 * math.pi * _mix(TABLE_SEED, s + np.uint64(2))
    st = np.sqrt(np.maximum(0.0, 1 - z * z))
    om = np.stack([st * np.cos(ph), st * np.sin(ph), z], 1)
    a, b = np.repeat(xi, trials, 0), xi[gam]
    g = np.sqrt((a - b)[:, 0] ** 2 + (a - b)[:, 1] ** 2 + (a - b)[:, 2] ** 2)
    ok, at = np.ones(len(g), dtype=bool), []
    for sgn in (0.5, -0.5):
        t = (0.5 * (a + b) + sgn * g[:, None] * om + np.array(hi)) / h - 0.5
        t = np.sign(t) * np.floor(np.abs(t) + 0.5)
        ok &= ((t >= 0) & (t <= n - 1)).all(1)
        t = np.clip(t, 0, n - 1).astype(np.int64)
        at.append(where[(t[:, 0] * ny + t[:, 1]) * nz + t[:, 2]])
    w = (nv * h.prod() / (math.sqrt(2.0) * trials) * g * ok).astype(np.float32)
    return tuple(x.reshape(nv, trials) for x in (gam, at[0], at[1], w))


def _collide(case, f, xi, dv, which):
    """The hard-sphere term of the cells `which` of f, corrected."""
    n, hi = _axes(case)
    gam, l, m, w = (torch.as_tensor(x, device=f.device) for x in _tables(*n, hi, case["trials"]))
    for a, b in _rows(len(which), max(1, (1 << 26) // len(xi))):
        c = which[a:b]
        v = f[c]
        vt = v.T.contiguous()
        B, C = torch.zeros_like(vt), torch.zeros_like(vt)
        for k in range(case["trials"]):
            wk = w[:, k, None].double()
            B.addcmul_(wk, vt[gam[:, k]])
            C.addcmul_(vt[l[:, k]] * wk, vt[m[:, k]])
        B, C = B.T, C.T
        _, u, temp = _moments(v, xi, dv)
        phi = _phi((xi[None] - u[:, None]) / temp.sqrt()[:, None, None])
        loss = v * B
        wp = phi * loss[..., None]
        d = torch.linalg.solve(phi.transpose(1, 2) @ wp, (phi * (C - loss)[..., None]).sum(1))
        yield c, C - loss * (1 + (phi @ d[..., None])[..., 0])


def _silu_net(p, x):
    at = 0
    for k, (i, o) in enumerate(LAYERS):
        w, b = p[at:at + i * o].reshape(o, i), p[at + i * o:at + i * o + o]
        at += i * o + o
        x = x @ w.T + b
        if k < 3:
            x = x * torch.sigmoid(x)
    return x


def _kn_local(case, rho, u, temp):
    """(Kn / rho) times the largest gradient, by least squares over the neighbours weighted with area / distance^2."""
    xyz, h, src, share, wall = _mesh(tuple(sorted(_spec(case).items())))
    nc, dim, bc = len(h), case["dim"], _bc(case)
    q = torch.cat([rho[:, None], temp[:, None], u], 1)
    mine = torch.arange(nc, device=h.device)[:, None, None]
    use = (share > 0) & ~wall & (src != mine) & (src < nc)
    j = torch.where(use, src, mine).reshape(nc, -1)
    d = xyz[j] - xyz[:, None]
    for k in range(dim):
        if bc[2 * k] == D.BC_PERIODIC:
            d[..., k] -= torch.round(d[..., k])
    area = (share * (h ** (dim - 1))[:, None, None] * use).reshape(nc, -1)
    w = torch.where(area > 0, area / d.square().sum(-1).clamp(min=1e-300), 0.0)
    wd = w[..., None] * d
    g = torch.linalg.solve(d.transpose(1, 2) @ wd, wd.transpose(1, 2) @ (q[j] - q[:, None]))
    top = torch.stack([g[:, :, 0].norm(dim=1) / rho, g[:, :, 1].norm(dim=1) / temp,
                       g[:, :, 2:].flatten(1).norm(dim=1) / temp.sqrt()]).max(0).values
    return case["kn"] / rho * top


def _hermite(c):
    he = (torch.ones_like(c), c, (c * c - 1) / math.sqrt(2.0), (c * c - 3) * c / math.sqrt(6.0))
    he = torch.stack(he, -1)
    return torch.einsum("...a,...b,...c->...abc", he[..., 0, :], he[..., 1, :], he[..., 2, :]).flatten(-3)


def _learned(case, f, xi, dv, dt, seed):
    nc = len(f) - 1
    p = torch.as_tensor(_weights(seed), device=f.device).double()
    parts = [_moments(f[a:b], xi, dv) for a, b in _rows(nc, 16384)]
    rho, u, temp = (torch.cat([x[k] for x in parts]) for k in range(3))
    low = torch.nonzero(_kn_local(case, rho, u, temp) < 0.05)[:, 0]
    left = torch.ones(nc, dtype=torch.bool, device=f.device)
    new = f.clone()
    for a, b in _rows(len(low), max(1, (1 << 23) // len(xi))):
        c = low[a:b]
        v = f[c]
        cc = (xi[None] - u[c][:, None]) / temp[c].sqrt()[:, None, None]
        H, M, phi = _hermite(cc), _maxwell(xi, rho[c], u[c], temp[c]), _phi(cc)
        o = [_silu_net(p, (x[..., None] * H).sum(1) * dv / rho[c][:, None]) for x in (v, M)]
        raw = M * (rho[c] * temp[c].sqrt())[:, None] * (H @ (o[0] - o[1])[..., None])[..., 0]
        mp = phi * M[..., None]
        d = torch.linalg.solve(phi.transpose(1, 2) @ mp, (phi * raw[..., None]).sum(1))
        Q = raw - M * (phi @ d[..., None])[..., 0]
        good = (Q * torch.log(v.clamp(min=1e-300))).sum(1) <= 1e-5 * Q.abs().sum(1)
        new[c[good]] = (v + dt / case["kn"] * Q)[good]
        left[c[good]] = False
    for c, term in _collide(case, f, xi, dv, torch.nonzero(left)[:, 0]):
        new[c] = f[c] + dt / case["kn"] * term
    return new


def _exact_lbm(case, seed):
    xyz, h, src, share, wall = _mesh(tuple(sorted(_spec(case).items())))
    dev, nc, dim, Q = h.device, len(h), case["dim"], case["lattice"]
    c = [(x, y, z) for r in range(4) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)
         if x * x + y * y + z * z == r and (dim == 3 or z == 0) and (Q != 19 or r < 3)]
    w = {9: (4 / 9, 1 / 9, 1 / 36, 0), 19: (1 / 3, 1 / 18, 1 / 36, 0), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[Q]
    w = torch.tensor([w[sum(x * x for x in v)] for v in c], dtype=torch.float64, device=dev)
    cv = torch.tensor(c, dtype=torch.float64, device=dev)

    def feq(rho, u):
        cu = cv @ u.T
        return w[:, None] * rho[None] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * u.square().sum(1)[None])

    rho, u = (torch.as_tensor(x, device=dev) for x in _lbm_start(case, nc, seed))
    inflow = feq(torch.ones(1, dtype=torch.float64, device=dev),
                 torch.tensor([[case["speed"], 0, 0]], dtype=torch.float64, device=dev))
    f = torch.cat([feq(rho, u), inflow], 1).to(TYPE[case["prec"]]).double()
    dt = 0.3 * float(h.min()) / max(sum(abs(x) for x in v) for v in c)
    dth = dt / h
    for _ in range(case["steps"]):
        g = torch.empty_like(f)
        g[:, nc] = f[:, nc]
        for i, v in enumerate(c):
            own = f[i, :nc]
            acc = own * (1 - dth * sum(abs(x) for x in v))
            for d in range(dim):
                if v[d]:
                    mir = c.index(tuple(-x if e == d else x for e, x in enumerate(v)))
                    col = 2 * d + (0 if v[d] > 0 else 1)
                    val = torch.where(wall[:, col], f[mir][src[:, col]], f[i][src[:, col]])
                    acc = acc + dth * (share[:, col] * val).sum(1)
            g[i, :nc] = acc
        rho = g[:, :nc].sum(0)
        u = (g[:, :nc].T @ cv) / rho[:, None]
        g[:, :nc] -= case["omega"] * (g[:, :nc] - feq(rho, u))
        f = g
    rho = f[:, :nc].sum(0)
    out = {"rho": rho, "u": (f[:, :nc].T @ cv) / rho[:, None]}
    if case["whole"]:
        out["f"] = f[:, :nc].T.contiguous()
    return {k: v.cpu().numpy() for k, v in out.items()}


def exact(case, seed):
    if case["kind"] == "mlp":
        g = np.random.default_rng(seed + 5)
        p = np.concatenate([np.concatenate([g.standard_normal(i * o) / math.sqrt(i), np.zeros(o)]) for i, o in LAYERS])
        p = torch.as_tensor(p.astype(np.float32), device=_dev()).double().requires_grad_()
        x, t = (torch.as_tensor(a, device=_dev()).double() for a in _pairs(case["rows"], seed))
        loss = (_silu_net(p, x) - t).square().mean()
        loss.backward()
        return {"loss": float(loss), "grad": p.grad}
    if case["kind"] == "lbm":
        return _exact_lbm(case, seed)
    f, xi, dv = _stored(case, seed)
    nc = len(f) - 1
    if case["kind"] == "fields":
        rho, u, temp = _moments(f[:nc], xi, dv)
        return {"rho": rho.cpu().numpy(), "u": u.cpu().numpy(), "T": temp.cpu().numpy(), "kinetic": None, "count": None}
    hmin = float(_mesh(tuple(sorted(_spec(case).items())))[1].min())
    dt = _dt(case, 0.4 * hmin / float(_nodes(case)[0][:, :case["dim"]].sum(1).max()))
    for _ in range(case["steps"]):
        f = _transport(case, f, dt)
        if case["fields"]:
            rho, u, temp = _moments(f[:nc], xi, dv)
        if case["coll"] in ("bgk", "entropic"):
            _relax(case, f, xi, dv, dt, case["coll"] == "entropic")
        elif case["coll"] == "hs":
            new = f.clone()
            for c, term in _collide(case, f, xi, dv, torch.arange(nc, device=f.device)):
                new[c] = f[c] + dt / case["kn"] * term
            f = new
        elif case["coll"] == "learned":
            f = _learned(case, f, xi, dv, dt, seed)
    if case["fields"]:
        return {"f": f[:nc], "rho": rho.cpu().numpy(), "u": u.cpu().numpy(), "T": temp.cpu().numpy()}
    return {"f": f[:nc]}
