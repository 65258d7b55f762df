"""The work a user of this library has it do, as cases that can be timed.

A case is one block of a run between two read-backs: some time steps of one
simulation (or of a batch of replicas) and then the fields a monitor or a
snapshot takes, or one call of the warm-start network.  Everything goes
through the package's public entry points.  Snapshots of a single- or
reduced-precision run are kept in single precision, those of an FP64 run in
double.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import warmstart, workloads as W


# ----------------------------------------------------------------- the cases
def _pore(name, nx, ny, nz, thickness, radius, beads, steps, read, **kw):
    """A membrane pierced by a pore with a threaded chain (periodic box)."""
    c = dict(kind="pore", name=name, nx=nx, ny=ny, nz=nz, thickness=thickness, radius=radius, beads=beads,
             steps=steps, read=read, charge=-1.0, salt=0.005, field=5e-3, solver="mg", precision="f32", tol=1e-8,
             warm=0)
    c.update(kw)
    return c


def listed():
    return [
        # a small box of ragged extents, as in the parity tests: launches and latency count
        _pore("small_pore", 40, 24, 36, 4, 4.0, 8, 40, "n,j,phi"),
        # the charged slit in FP64 with the paper's SOR to 1e-10: the reference-quality run
        dict(kind="slit", name="slit_f64", nx=32, ny=32, nz=32, beads=8, steps=10, read="n,j,phi", charge=-1.0,
             wall=-0.01, salt=0.01, field=1e-3, solver="sor", precision="f64", tol=1e-10, warm=0),
        # the translocation run: the usual production box, default solver
        _pore("pore", 64, 64, 128, 8, 4.0, 32, 40, "n,phi"),
        # the same box with the paper's Chebyshev SOR
        _pore("pore_sor", 64, 64, 128, 8, 4.0, 32, 3, "n,phi", solver="sor"),
        # the same box in FP64: reference runs for the reduced formats
        _pore("pore_f64", 64, 64, 128, 8, 4.0, 32, 10, "n,phi", precision="f64"),
        # the paper's own pore (charged lining, harmonic chain of 100 beads), with the current it reports
        dict(kind="paper", name="paper_pore", nx=64, ny=64, nz=160, thickness=40, radius=6.0, beads=100, steps=30,
             read="n,phi,current", salt=100.0, field=0.05, solver="mg", precision="f32", tol=1e-8, warm=0),
        # a larger pore with 16-bit storage of the populations
        _pore("pore_large_fp16", 128, 128, 256, 8, 6.0, 64, 10, "n,phi", precision="fp16"),
        # the benchmark's pore: the largest single box
        _pore("pore_huge", 256, 256, 512, 16, 8.0, 128, 10, "n,phi", salt=0.01, field=2e-3),
        # independent replicas of uneven size stepped together
        dict(kind="replicas", name="replicas", count=10, first=1000, steps=8, read="n,phi", solver="mg",
             precision="f32", tol=1e-8),
        # the warm-start network: training on whole coarse grids, and one evaluation
        dict(kind="train", name="net_train", nx=16, ny=16, nz=32, samples=64, iters=10, batch=8, periodic=7),
        dict(kind="eval", name="net_eval", nx=32, ny=32, nz=64, periodic=7),
    ]


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _coarsest(dims, periodic):
    """Cells left when the multigrid hierarchy has halved the box as far as it does."""
    d = list(dims)
    while d[0] * d[1] * d[2] > 1024 and all(v >= 2 and not (p and v % 4) for v, p in zip(d, periodic)):
        d = [(v + 1) // 2 for v in d]
    return d[0] * d[1] * d[2]


def draw(rng):
    kind = rng.choice(["pore"] * 8 + ["slit"] * 3 + ["paper"] + ["replicas"] * 2 + ["train"] + ["eval"])
    if kind in ("pore", "slit", "paper"):
        solver = rng.choice(["mg", "mg", "mg", "sor"])
        precision = rng.choice(["f32", "f32", "f32", "fp16", "bf16", "f64"])
        # boxes from the smallest to 128 x 128 x 256 (SOR and FP64 to the production box)
        top = 4.2e6 if solver == "mg" and precision != "f64" else 6e5
        q = 4 if solver == "mg" else 2
        odd = rng.choice([0, 1]) if kind == "slit" else 0  # closed in z: any extent there
        while True:
            N = _spread(rng, 2e4, top)
            a = (N / rng.uniform(1.5, 3.0)) ** (1 / 3)
            nx, ny = (max(20, q * round(a * rng.uniform(0.8, 1.25) / q)) for _ in range(2))
            nz = max(28, q * round(N / (nx * ny) / q))
            nz = min(nz, q * int(top / (nx * ny) / q)) + odd
            # the library refuses multigrid where too many cells are left
            if solver == "sor" or _coarsest((nx, ny, nz), (1, 1, kind != "slit")) <= 4500:
                break
        work = nx * ny * nz * (30 if solver == "sor" else 1) * (10 if precision == "f64" else 1)
        steps = int(max(2, min(40, 2e7 / work)))
        if kind == "slit":
            return dict(kind="slit", nx=nx, ny=ny, nz=nz, beads=rng.randint(2, 8), steps=steps,
                        read="n,j,phi", charge=-0.1, wall=-rng.choice([0.0, 0.005, 0.01]), salt=0.01, field=1e-3,
                        solver=solver, precision=precision, tol=rng.choice([1e-8, 1e-10]) if precision == "f64" else 1e-8,
                        warm=0)
        if kind == "paper":
            return dict(kind="paper", nx=nx, ny=ny, nz=nz, thickness=max(4, nz // 4), radius=rng.choice([4.0, 5.0, 6.0]),
                        beads=rng.randint(8, 24), steps=steps, read="n,phi,current", salt=rng.choice([10.0, 100.0]),
                        field=rng.choice([0.0, 0.05]), solver=solver, precision=precision, tol=1e-8, warm=0)
        t = rng.choice([4, 6, 8, 12])
        return dict(kind="pore", nx=nx, ny=ny, nz=nz, thickness=t, radius=rng.uniform(3.5, min(8.0, nx / 4, ny / 4)),
                    beads=rng.randint(4, max(5, min(96, nz // 2))), steps=steps, read=rng.choice(["n,phi", "phi", "n,j,phi"]),
                    charge=-0.1, salt=rng.uniform(0.004, 0.02), field=rng.choice([0.0, 2e-3, 5e-3]), solver=solver,
                    precision=precision, tol=1e-8, warm=2 if rng.random() < 0.2 and nz % 4 + nx % 4 + ny % 4 == 0 else 0)
    if kind == "replicas":
        return dict(kind="replicas", count=rng.randint(2, 12), first=rng.randint(2000, 9000), steps=rng.randint(2, 6),
                    read="n,phi", solver=rng.choice(["mg", "mg", "mg", "sor"]), precision=rng.choice(["f32", "f32", "fp16"]),
                    tol=1e-8 if rng.random() < 0.5 else 1e-6)
    nx, ny, nz = (rng.randint(9, 33) for _ in range(3))
    if kind == "train":
        return dict(kind="train", nx=nx, ny=ny, nz=nz, samples=rng.randint(8, 64), iters=rng.randint(3, 10),
                    batch=rng.choice([1, 4, 8]), periodic=rng.choice([0, 3, 7]))
    m = rng.choice([1, 2, 4])
    return dict(kind="eval", nx=nx * m, ny=ny * m, nz=nz * m, periodic=rng.choice([0, 3, 7]))


# ----------------------------------------------------------------- inputs
def _membrane(c):
    z0 = c["nz"] // 2 - c["thickness"] // 2
    return z0, z0 + c["thickness"] - 1


def _workload(c, seed):
    s = dict(seed_init=seed, seed_noise=seed + 1)
    if c["kind"] == "slit":
        wl = W.charged_slit(c["nx"], c["ny"], c["nz"], wall_charge=c["wall"], salt=c["salt"], n_beads=c["beads"],
                            bead_charge=c["charge"], E=(c["field"], 0.0, 0.0), precision=c["precision"], tol=c["tol"], **s)
    elif c["kind"] == "paper":
        wl = W.paper_pore(c["nx"], c["ny"], c["nz"], membrane=_membrane(c), radius=c["radius"], salt_mM=c["salt"],
                          n_beads=c["beads"], E=(0.0, 0.0, c["field"]), precision=c["precision"], tol=c["tol"],
                          seed_chain=seed + 2, **s)
        # the paper generator adds no noise of its own: seeded, as in the other workloads
        rng = np.random.default_rng(seed)
        wl.n_init[1:] += np.where(wl.solid == 0, rng.uniform(-1e-4, 1e-4, (2,) + wl.solid.shape), 0.0)
    else:
        wl = W.translocation(c["nx"], c["ny"], c["nz"], membrane=_membrane(c), radius=c["radius"], salt=c["salt"],
                             n_beads=c["beads"], bead_charge=c["charge"], E=(0.0, 0.0, c["field"]),
                             precision=c["precision"], tol=c["tol"], seed_chain=seed + 2, **s)
    if c["solver"] == "mg":
        return wl.replace(flags=W.FLAG_POISSON_MG)
    # the spectral radius and test interval of the production SOR run
    return wl.replace(rho_jacobi=0.9999 if c["kind"] != "slit" else 0.0,
                      poisson_check_every=4 if c["kind"] != "slit" else 1, poisson_max_iter=20000)


def _replicas(c, seed):
    wls = W.replica_set(n_rep=c["count"], seed=c["first"], precision=c["precision"])
    out = []
    for r, wl in enumerate(wls):
        # the boxes and chains are the case's, the ion noise and the bead noise the seed's
        rng = np.random.default_rng(seed * 1000 + r)
        fluid = wl.solid == 0
        n = wl.n_init.copy()
        amp = 0.4 * float(n[1][fluid].min())
        n[1:] += np.where(fluid, rng.uniform(-amp, amp, (2,) + fluid.shape), 0.0)
        flags = W.FLAG_POISSON_MG if c["solver"] == "mg" else 0
        out.append(wl.replace(n_init=n, seed=seed * 1000 + r, flags=flags, poisson_tol=c["tol"],
                              rho_jacobi=0.0 if flags else 0.9999, poisson_check_every=1 if flags else 4,
                              poisson_max_iter=20000))
    return out


def _periodic(c):
    return tuple((c["periodic"] >> a) & 1 for a in range(3))


def _smooth(a, rounds):
    for _ in range(rounds):
        for ax in (-1, -2, -3):
            a = 0.5 * a + 0.25 * (np.roll(a, 1, ax) + np.roll(a, -1, ax))
    return a


def _net_samples(c, seed, count):
    """Inputs and target as the warm start's recorder scales them: a short-range
    change of the source, a smooth potential, a smooth zero-mean change of it."""
    rng = np.random.default_rng(seed)
    shape = (count, c["nz"], c["ny"], c["nx"])
    db, ph = _smooth(rng.standard_normal(shape), 1), _smooth(rng.standard_normal(shape), 6)
    db, ph = db / db.std(), ph / ph.std()
    t = _smooth(db, 3) + 0.1 * ph
    t -= t.mean(axis=(1, 2, 3), keepdims=True)
    t /= t.std()
    return np.stack([db, ph], axis=1).astype(np.float32), t.astype(np.float32)


def _net_weights(seed):
    w = warmstart.init_params(seed)
    return (w + 0.01 * np.random.default_rng(seed + 7).standard_normal(w.size)).astype(np.float32)


def _settle(step, handles, wls, set_beads):
    """What a run is started from: the initial populations and beads, with the
    potential of a short settling run (a start from zero potential is a
    transient of a few solves that no production run repeats)."""
    step(5)
    w = torch.tensor(_WT, dtype=torch.float64).reshape(1, 19, 1)
    for r, (h, wl) in enumerate(zip(handles, wls)):
        phi = E.ekl_get_fields(h, wl.n_nodes, wl.n_beads, ("phi",))["phi"]
        f0 = w * torch.from_numpy(wl.n_init).reshape(3, 1, -1)
        E.ekl_set_state(h, f0.numpy(), phi, 0)
        if wl.n_beads:
            set_beads(r, wl.R, wl.V, wl.charge, wl.chain)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("pore", "slit", "paper"):
        wl = _workload(case, seed)
        sim = E.Simulation(wl)
        if case["solver"] == "mg":
            _settle(sim.step, [sim.h], [wl], lambda r, *beads: sim.set_beads(*beads))
        if case["warm"]:
            # a network of the size in use; a small output scale, as of a trained one
            sim.set_warmstart(_net_weights(seed), (1.0, 0.1, 1e-3), level=case["warm"])
        return dict(kind="sim", case=case, sim=sim)
    if kind == "replicas":
        wls = _replicas(case, seed)
        batch = E.Batch(wls)
        if case["solver"] == "mg":
            _settle(batch.step, [v.h for v in batch.reps], wls,
                    lambda r, *beads: E.ekl_batch_set_beads(batch.h, r, *beads))
        return dict(kind="batch", case=case, batch=batch)
    if kind == "train":
        x, t = _net_samples(case, seed, case["samples"])
        return dict(kind="train", case=case, x=x, t=t, w=_net_weights(seed), seed=seed)
    x, _ = _net_samples(case, seed, 1)
    return dict(kind="eval", case=case, x=x[0], w=_net_weights(seed))


# ----------------------------------------------------------------- one pass
def _kept(a, precision):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return t if precision == "f64" else t.to(torch.float32)


def _snapshot(view, case):
    read = case["read"].split(",")
    f = view.fields(tuple(k for k in read if k != "current") + ("R", "V"))
    out = {k: _kept(v, case["precision"]) for k, v in f.items() if v is not None}
    if "current" in read:
        out["current"] = _kept(view.current(2)[3:], case["precision"])
    return out


def run(state):
    case = state["case"]
    if state["kind"] == "sim":
        state["sim"].step(case["steps"])
        return _snapshot(state["sim"], case)
    if state["kind"] == "batch":
        state["batch"].step(case["steps"])
        return [_snapshot(rep, case) for rep in state["batch"].reps]
    dims = (case["nx"], case["ny"], case["nz"])
    if state["kind"] == "train":
        w, curve = E.ekl_net_train_grid(dims, _periodic(case), state["x"], state["t"], None, state["w"], case["iters"],
                                        case["batch"], 1e-3, state["seed"])
        return dict(w=w, curve=curve)
    return dict(y=E.ekl_net_eval(dims, _periodic(case), state["x"], state["w"]))


# ----------------------------------------------------------------- what a pass cannot do without
def _step_bytes(N, fluid, precision):
    """Populations in and out, the potential in and out, the link word."""
    s = {"f64": 8, "f32": 4}.get(precision, 2)
    return fluid * (2 * 57 * s + 16) + 4 * N


def work(case):
    kind = case["kind"]
    if kind in ("train", "eval"):
        n = case["nx"] * case["ny"] * case["nz"]
        macs = 27 * (2 * 16 + 2 * 16 * 16 + 16)
        if kind == "eval":
            return {"bytes": 12 * n + 4 * E.EKL_NET_PARAMS, "flops": 2 * macs * n}
        used = min(case["samples"], case["iters"] * case["batch"])
        return {"bytes": 12 * n * used + 8 * E.EKL_NET_PARAMS, "flops": 3 * 2 * macs * n * case["iters"] * case["batch"]}
    if kind == "replicas":
        boxes = [(w.n_nodes, int((w.solid == 0).sum())) for w in W.replica_set(n_rep=case["count"], seed=case["first"])]
    else:
        plane = case["nx"] * case["ny"]
        N = plane * case["nz"]
        walls = 2 * plane if kind == "slit" else case["thickness"] * (plane - math.pi * case["radius"] ** 2)
        boxes = [(N, N - int(walls))]
    per = {"n": 3, "j": 9, "phi": 1, "current": 0}
    arrays = sum(per[k] for k in case["read"].split(","))
    b = f = 0
    for N, fluid in boxes:
        b += case["steps"] * _step_bytes(N, fluid, case["precision"]) + 8 * arrays * N
        f += case["steps"] * fluid * 1200
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------- 64-bit values
# The step written out from the method's equations in torch FP64: stream with
# halfway bounce-back, moments, Poisson (conjugate gradients to 1e-12), beads,
# collision.  No code of the package is used beyond the workload it describes.
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
      (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_OPP = [0] + [p + 1 if p % 2 else p - 1 for p in range(1, 19)]
_WT = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_FACES = [(-1, 0, 0), (1, 0, 0), (0, -1, 0), (0, 1, 0), (0, 0, -1), (0, 0, 1)]
_KT = 1.0 / 3.0


def _philox(c, key):
    c = [v.astype(np.uint64) for v in c]
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    m32 = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


class _Exact:
    def __init__(self, wl, dev):
        self.wl, self.dev, self.step_no = wl, dev, 0
        f64 = dict(dtype=torch.float64, device=dev)
        self.fluid = torch.from_numpy(wl.solid == 0).to(dev)
        self.open = [self.shift(self.fluid, (-d[0], -d[1], -d[2]), True) & self.fluid for d in _FACES]
        self.deg = sum(o.to(torch.float64) for o in self.open)
        self.blocked = [~self.shift(self.fluid, c, True) for c in _C]
        self.nf = float(self.fluid.sum())
        fl = self.fluid.to(torch.float64)
        n0 = torch.from_numpy(wl.n_init).to(dev) * fl
        self.fs = torch.stack([torch.stack([w * n0[a] for w in _WT]) for a in range(3)])
        self.phi = torch.zeros(wl.solid.shape, **f64)
        self.c4 = 4 * math.pi * wl.bjerrum
        share = torch.zeros(wl.solid.shape, **f64)
        if wl.surface_charge is not None:
            touch = sum(self.shift(self.fluid, (-d[0], -d[1], -d[2]), True).to(torch.float64) for d in _FACES)
            sc = torch.from_numpy(wl.surface_charge).to(dev)
            share = torch.where(touch > 0, sc / touch.clamp(min=1), torch.zeros_like(sc)) * (1 - fl)
        # charge of the wall node across each face of a node
        self.ghost = [self.shift(share, (-d[0], -d[1], -d[2]), True) * fl for d in _FACES]
        self.src_wall = sum(self.ghost)
        self.R = None if wl.R is None else wl.R.copy()
        self.V = None if wl.V is None else wl.V.copy()

    def shift(self, a, c, outside_zero=False):
        """a at x - c; with outside_zero, 0 where that lies beyond a closed face."""
        r = torch.roll(a, (c[2], c[1], c[0]), (-3, -2, -1))
        if outside_zero:
            for ax, d, per in ((-1, c[0], self.wl.periodic[0]), (-2, c[1], self.wl.periodic[1]),
                               (-3, c[2], self.wl.periodic[2])):
                if d and not per:
                    r.narrow(ax, 0 if d > 0 else a.shape[ax] - 1, 1).zero_()
        return r

    def streamed(self):
        return torch.stack([torch.stack([torch.where(self.blocked[p], self.fs[a, _OPP[p]], self.shift(self.fs[a, p], _C[p]))
                                         for p in range(19)]) for a in range(3)]) * self.fluid

    @staticmethod
    def moments(f):
        n = f.sum(1)
        j = torch.stack([sum(c[k] * f[:, p] for p, c in enumerate(_C) if c[k]) for k in range(3)], 1)
        return n, j

    def solve(self, rho):
        b = torch.where(self.fluid, self.c4 * (rho - (rho * self.fluid).sum() / self.nf), torch.zeros_like(rho))

        def A(v):
            out = self.deg * v
            for d, o in zip(_FACES, self.open):
                out -= o * self.shift(v, (-d[0], -d[1], -d[2]))
            return out

        x, bb = self.phi, float((b * b).sum())
        r = b - A(x)
        p, rr = r.clone(), (r * r).sum()
        for it in range(20000):
            q = A(p)
            al = rr / (p * q).sum().clamp(min=1e-300)
            x = x + al * p
            r = r - al * q
            new = (r * r).sum()
            if it % 16 == 15 and float(new) <= 1e-24 * bb:
                break
            p = r + (new / rr.clamp(min=1e-300)) * p
            rr = new
        return x

    def gradient(self, phi):
        v = []
        for d, o, g in zip(_FACES, self.open, self.ghost):
            v.append(torch.where(o, self.shift(phi, (-d[0], -d[1], -d[2])), phi + self.c4 * g))
        return torch.stack([(v[2 * k + 1] - v[2 * k]) * 0.5 for k in range(3)]) * self.fluid

    def stencil(self):
        nz, ny, nx = self.wl.solid.shape
        dims = np.array([nx, ny, nz])
        base = np.floor(self.R).astype(int)
        fr = self.R - base
        ids, ws = [], []
        for k in range(8):
            o = np.array([k & 1, (k >> 1) & 1, (k >> 2) & 1])
            q = base + o
            inside = np.ones(len(q), bool)
            for a in range(3):
                if self.wl.periodic[a]:
                    q[:, a] %= dims[a]
                else:
                    inside &= (q[:, a] >= 0) & (q[:, a] < dims[a])
            q = np.clip(q, 0, dims - 1)
            w = np.prod(np.where(o, fr, 1 - fr), axis=1) * inside * (self.wl.solid[q[:, 2], q[:, 1], q[:, 0]] == 0)
            ids.append(q[:, 0] + nx * (q[:, 1] + ny * q[:, 2]))
            ws.append(w)
        ids, ws = np.stack(ids, 1), np.stack(ws, 1)
        return ids, ws / ws.sum(1, keepdims=True)

    def image(self, d):
        for a, L in enumerate((self.wl.nx, self.wl.ny, self.wl.nz)):
            if self.wl.periodic[a]:
                d[..., a] -= L * np.rint(d[..., a] / L)
        return d

    @staticmethod
    def wca(eps, sig, d):
        r2 = (d * d).sum(-1)
        near = (r2 < 2 ** (1 / 3) * sig * sig) & (r2 > 0)
        r2 = np.where(near, r2, 1.0)
        s6 = (sig * sig / r2) ** 3
        return np.where(near, 24 * eps * (2 * s6 * s6 - s6) / r2, 0.0)[..., None] * d

    def forces(self):
        wl, R = self.wl, self.R
        F = np.zeros_like(R)
        chain = wl.chain
        d = self.image(R[:-1] - R[1:])
        r2 = (d * d).sum(1)
        if wl.bond_kind == W.BOND_FENE:
            fac = -wl.bond_k / (1 - r2 / wl.bond_r0 ** 2)
        else:
            r = np.sqrt(r2)
            fac = -wl.bond_k * (r - wl.bond_l0) / r
        fb = np.where(chain[:-1] == chain[1:], fac, 0.0)[:, None] * d
        F[:-1] += fb
        F[1:] -= fb
        pair = self.image(R[:, None] - R[None])
        fp = self.wca(wl.wca_eps, wl.wca_sigma, pair)
        i = np.arange(len(R))
        if wl.bond_kind == W.BOND_HARMONIC:
            fp[(np.abs(i[:, None] - i[None]) <= 1) & (chain[:, None] == chain[None])] = 0.0
        F += fp.sum(1)
        # wall nodes within reach
        rc = int(math.ceil(2 ** (1 / 6) * wl.wall_sigma)) + 1
        o = np.arange(-rc, rc + 1)
        off = np.stack(np.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
        q = np.floor(R).astype(int)[:, None] + off[None]
        dims = np.array([wl.nx, wl.ny, wl.nz])
        w, inside = q.copy(), np.ones(q.shape[:2], bool)
        for a in range(3):
            if wl.periodic[a]:
                w[..., a] %= dims[a]
            else:
                inside &= (w[..., a] >= 0) & (w[..., a] < dims[a])
        w = np.clip(w, 0, dims - 1)
        wall = inside & (wl.solid[w[..., 2], w[..., 1], w[..., 0]] == 1)
        F += (self.wca(wl.wall_eps, wl.wall_sigma, R[:, None] - q) * wall[..., None]).sum(1)
        return F

    def beads(self, n, j, grad, ids, ws):
        wl = self.wl
        at = torch.from_numpy(ids).to(self.dev)
        nn = n.reshape(3, -1)[:, at].cpu().numpy()
        jj = j.reshape(3, 3, -1)[:, :, at].cpu().numpy()
        gg = grad.reshape(3, -1)[:, at].cpu().numpy()
        u = np.where(nn[:, None] > 0, jj / np.where(nn > 0, nn, 1.0)[:, None], 0.0)
        nR, uR, gR = (nn * ws).sum(-1), (u * ws).sum(-1), (gg * ws).sum(-1)  # [s,b], [s,3,b], [3,b]
        gam = wl.bead_xi * nR / nR.sum(0)
        gt = gam.sum(0)
        q, M, nsub = wl.charge, wl.bead_mass, wl.md_substeps
        dt = 1.0 / nsub
        amp = np.sqrt(2 * gt * wl.bead_kT / dt)
        acc = np.zeros_like(uR)
        nb = len(q)
        Fe = q[:, None] * _KT * (np.array(wl.E_app)[None] - gR.T)
        drag = np.einsum("sb,skb->bk", gam, uR)
        L = np.array([wl.nx, wl.ny, wl.nz], float)
        for sub in range(nsub):
            F = self.forces()
            o = _philox([np.arange(nb), np.full(nb, sub | (1 << 24)), np.full(nb, self.step_no & 0xFFFFFFFF),
                         np.full(nb, self.step_no >> 32)], wl.seed)
            xi = math.sqrt(3) * (2 * (np.stack(o[:3], 1).astype(np.float64) + 0.5) / 2 ** 32 - 1)
            self.V = (M * self.V / dt + drag + F + Fe + amp[:, None] * xi) / (M / dt + gt)[:, None]
            acc += dt * -gam[:, None] * (uR - self.V.T[None])
            self.R = self.R + dt * self.V
            for a in range(3):
                if wl.periodic[a]:
                    self.R[:, a] = np.where(self.R[:, a] < 0, self.R[:, a] + L[a],
                                            np.where(self.R[:, a] >= L[a], self.R[:, a] - L[a], self.R[:, a]))
        f = torch.zeros(9, n[0].numel(), dtype=torch.float64, device=self.dev)
        val = (acc[..., None] * ws).reshape(9, -1)
        f.index_add_(1, at.reshape(-1), torch.from_numpy(val).to(self.dev))
        return f.reshape((3, 3) + tuple(n.shape[1:])) / torch.where(n > 0, n, torch.ones_like(n))[:, None]

    def collide(self, f, n, j, grad, drag):
        wl = self.wl
        safe = torch.where(n > 0, n, torch.ones_like(n))
        E0 = torch.tensor(wl.E_app, dtype=torch.float64, device=self.dev).reshape(3, 1, 1, 1)
        G, av, h = [], [], []
        for s in range(3):
            body = torch.tensor(wl.body_force[s], dtype=torch.float64, device=self.dev).reshape(3, 1, 1, 1)
            g = body + wl.valence[s] * _KT * (E0 - grad)
            G.append(g if drag is None else g + drag[s])
            av.append(j[s] / safe[s] + 0.5 * G[s])
            h.append(0.5 * _KT / (wl.diffusivity[s] if wl.diffusivity[s] > 0 else wl.diffusivity[1]))
        den = sum(n[s] / (1 + h[s]) for s in range(3))
        den = torch.where(den > 0, den, torch.ones_like(den))
        us = sum(n[s] * av[s] / (1 + h[s]) for s in range(3)) / den
        for s in range(3):
            u = (av[s] + h[s] * us) / (1 + h[s])
            P = G[s] - 2 * h[s] * (u - us)
            om = 1 / wl.tau[s]
            u2, Pu = (u * u).sum(0), (P * u).sum(0)
            for p, (c, w) in enumerate(zip(_C, _WT)):
                cu, cP = (sum((c[k] * v[k] for k in range(3) if c[k]), torch.zeros_like(u2)) for v in (u, P))
                eq = w * n[s] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * u2)
                S = w * n[s] * (3 * cP + 9 * cu * cP - 3 * Pu)
                self.fs[s, p] = (f[s, p] - om * (f[s, p] - eq) + (1 - 0.5 * om) * S) * self.fluid

    def step(self):
        f = self.streamed()
        n, j = self.moments(f)
        rho = sum(self.wl.valence[s] * n[s] for s in range(3)) + self.src_wall
        if self.R is not None:
            ids, ws = self.stencil()
            rho.reshape(-1).index_add_(0, torch.from_numpy(ids.reshape(-1)).to(self.dev),
                                       torch.from_numpy((self.wl.charge[:, None] * ws).reshape(-1)).to(self.dev))
        self.phi = self.solve(rho)
        grad = self.gradient(self.phi)
        drag = self.beads(n, j, grad, ids, ws) if self.R is not None else None
        self.collide(f, n, j, grad, drag)
        self.step_no += 1

    def snapshot(self, case):
        n, j = self.moments(self.streamed())
        read = case["read"].split(",")
        out = {"R": self.R, "V": self.V}
        if "n" in read:
            out["n"] = n.reshape(3, -1)
        if "j" in read:
            out["j"] = j.reshape(3, 3, -1)
        if "phi" in read:
            phi = self.phi * self.fluid
            out["phi"] = ((phi - phi.sum() / self.nf) * self.fluid).reshape(-1)
        if "current" in read:
            z = self.wl.nz // 2
            out["current"] = sum(self.wl.valence[s] * j[s, 2, z].sum() for s in range(3)).reshape(1)
        return out


def _net_layers(w):
    w, out, o = w.double(), [], 0
    for ci, co in ((2, 16), (16, 16), (16, 16), (16, 1)):
        k = w[o:o + co * ci * 27].reshape(co, ci, 3, 3, 3)
        o += co * ci * 27
        out.append((k, w[o:o + co]))
        o += co
    return out


def _net(x, w, periodic):
    a = x.double()[None]
    layers = _net_layers(w)
    for i, (k, b) in enumerate(layers):
        for ax, per in zip((4, 3, 2), periodic):
            lo, hi = a.narrow(ax, a.shape[ax] - 1, 1), a.narrow(ax, 0, 1)
            a = torch.cat([lo, a, hi] if per else [torch.zeros_like(lo), a, torch.zeros_like(hi)], ax)
        a = torch.nn.functional.conv3d(a, k, b)
        a = torch.relu(a) if i < 3 else a
    return a[0, 0]


def _net_trained(case, seed, dev):
    x, t = (torch.from_numpy(v).to(dev) for v in _net_samples(case, seed, case["samples"]))
    w = torch.from_numpy(_net_weights(seed)).to(dev).double()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    state, mask, curve = seed, (1 << 64) - 1, []
    for it in range(case["iters"]):
        w.requires_grad_(True)
        loss = 0.0
        for _ in range(case["batch"]):  # samples in the order of the published splitmix64 generator
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            s = (z ^ (z >> 31)) % case["samples"]
            loss = loss + ((_net(x[s], w, _periodic(case)) - t[s].double()) ** 2).mean() / case["batch"]
        g, = torch.autograd.grad(loss, w)
        curve.append(float(loss))
        with torch.no_grad():  # Adam (Kingma and Ba)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            w = w - 1e-3 * (m / (1 - 0.9 ** (it + 1))) / ((v / (1 - 0.999 ** (it + 1))).sqrt() + 1e-8)
    return dict(w=w.detach().cpu(), curve=np.array(curve))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "train":
        return _net_trained(case, seed, dev)
    if kind == "eval":
        x, _ = _net_samples(case, seed, 1)
        return dict(y=_net(torch.from_numpy(x[0]).to(dev), torch.from_numpy(_net_weights(seed)).to(dev),
                           _periodic(case)).cpu())
    wls = _replicas(case, seed) if kind == "replicas" else [_workload(case, seed)]
    # conjugate gradients without a preconditioner: iterations grow with the box
    cost = sum(case["steps"] * (w.n_nodes + 2e5) * max(w.nx, w.ny, w.nz) for w in wls)
    if cost > 1.6e10:
        return None
    out = []
    for wl in wls:
        ex = _Exact(wl, dev)
        for _ in range(case["steps"]):
            ex.step()
        out.append({k: torch.as_tensor(v).cpu() for k, v in ex.snapshot(case).items()})
    return out if kind == "replicas" else out[0]
