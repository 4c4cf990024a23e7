"""The work whose speed counts: what a program that uses this engine has it do,
through the public entry points, from a few hundred particles to millions.

A case is a dict of plain values; ``kind`` names what a pass does:

* ``run``      -- a handle advances a block of steps, then its state and
                  observables are read (the main loop of a simulation);
* ``forces``   -- a list rebuild and one force evaluation of a loaded state
                  (analysis of given configurations);
* ``static``   -- the allocation-free force on device buffers of the caller;
* ``profile``  -- a binned velocity profile of a loaded state, as the flow
                  validations take every few steps;
* ``ensemble`` -- many small boxes advanced together by the ensemble kernel;
* ``serve``    -- a batch of independent boxes through the serving loop.

What a pass returns is held in FP32 wherever the engine computes it in FP32
(the FP64 arrays of the API only widen it).  Positions are folded into the
periodic box, where a last-bit difference at the seam reads as a whole box
length; so a pass returns each particle's displacement over the pass (minimum
image), the bookkeeping of a diffusion measurement, beside the velocities.
Total momentum is left out: it is zero up to rounding.

A fluid is chaotic: a last-bit difference grows about tenfold in 40 steps.  A
pass is therefore short (real runs repeat it thousands of times), so that its
outputs can be compared.
"""
import math

import numpy as np
import torch

import paper_1311_0402_gb300 as dpd

RC = 1.0


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest common simulation: a 3,000-particle fluid (tests, smoke
        # check, method development); launches and latency decide
        dict(name="fluid 3k", kind="run", lx=10.0, ly=10.0, lz=10.0, rho=3.0, species=1, chains=0.0, a=25.0,
             gamma=4.5, s=1.0, dt=0.01, lam=0.5, skin=0.3, det=0, body_mode=0, body=0.0, steps=32, every=0),
        # flow validation box: reverse Poiseuille, s = 1/2
        dict(name="poiseuille 32k", kind="run", lx=40.0, ly=20.0, lz=10.0, rho=4.0, species=1, chains=0.0, a=18.75,
             gamma=4.5, s=0.5, dt=0.01, lam=0.5, skin=0.3, det=0, body_mode=2, body=0.055, steps=24, every=0),
        # the largest box of the serving stream on its own handle, statistics
        # logged after every step as a production run logs them
        dict(name="statistics 81k", kind="run", lx=30.0, ly=30.0, lz=30.0, rho=3.0, species=1, chains=0.0, a=25.0,
             gamma=4.5, s=1.0, dt=0.01, lam=0.5, skin=0.4, det=0, body_mode=0, body=0.0, steps=20, every=1),
        # reproducible run (fixed summation order) at another lambda, in a
        # ragged box whose cells and bricks come out odd
        dict(name="deterministic 210k", kind="run", lx=61.3, ly=47.9, lz=23.8, rho=3.0, species=1, chains=0.0, a=25.0,
             gamma=4.5, s=1.0, dt=0.01, lam=0.65, skin=0.3, det=1, body_mode=0, body=0.0, steps=16, every=0),
        # three species with bonded chains: the amphiphile workload
        dict(name="amphiphile 786k", kind="run", lx=64.0, ly=64.0, lz=64.0, rho=3.0, species=3, chains=0.1, a=25.0,
             gamma=4.5, s=1.0, dt=0.005, lam=0.5, skin=0.4, det=0, body_mode=0, body=0.0, steps=24, every=0),
        # the headline fluid, larger than the L2 cache
        dict(name="fluid 3M", kind="run", lx=100.0, ly=100.0, lz=100.0, rho=3.0, species=1, chains=0.0, a=25.0,
             gamma=4.5, s=1.0, dt=0.01, lam=0.5, skin=0.4, det=0, body_mode=0, body=0.0, steps=16, every=0),
        # one configuration after another analysed: list and force, dense
        # two-species fluid (rho = 8), general weight exponent
        dict(name="rebuild and forces 250k", kind="forces", lx=36.5, ly=31.0, lz=27.6, rho=8.0, species=2, a=18.75,
             gamma=4.5, s=0.25, dt=0.01, skin=0.3, det=0),
        # a plug-in's force call on a small system: latency
        dict(name="static 3k", kind="static", lx=10.0, ly=10.0, lz=10.0, rho=3.0, species=1, a=25.0, gamma=4.5, s=1.0,
             dt=0.01, body_mode=0, body=0.0),
        # the same call near the largest size it takes
        dict(name="static 131k", kind="static", lx=41.0, ly=35.0, lz=30.0, rho=3.0, species=2, a=25.0, gamma=4.5,
             s=0.5, dt=0.01, body_mode=1, body=0.05),
        # the transient flow validation's box and bins
        dict(name="profile 262k", kind="profile", lx=59.4123, ly=118.825, lz=7.42654, rho=5.0, nbins=60),
        # many small boxes at once (parameter sweeps), L 6..10
        dict(name="ensemble 128 boxes", kind="ensemble", boxes=128, lmin=6, lmax=10, rho=3.0, s=1.0, dt=0.01, lam=0.5,
             steps=32),
        # a batch of requests of uneven size, L 6..30, through the serving loop
        dict(name="serve 24 boxes", kind="serve", boxes=24, lmin=6, lmax=30, rho=3.0, s=1.0, dt=0.01, lam=0.5,
             skin=0.3, steps_min=80, steps_max=120),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, n, rho, least=3.2):
    """Side lengths of a box of about n particles, ratios up to about 3."""
    v = n / rho
    r = [math.exp(rng.uniform(-0.5, 0.5)) for _ in range(3)]
    k = (v / (r[0] * r[1] * r[2])) ** (1.0 / 3.0)
    return [round(max(least, k * x), 2) for x in r]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "run", "forces", "static", "static", "profile", "ensemble",
                       "serve"])
    a, gamma = round(rng.uniform(15.0, 40.0), 2), round(rng.uniform(3.0, 6.0), 2)
    rho = rng.choice([3.0, 3.0, 4.0, 5.0])
    s = rng.choice([1.0, 1.0, 0.5, 0.25])
    if kind == "run":
        n = _log(rng, 600, 2.5e6)
        lx, ly, lz = _box(rng, n, rho)
        species = rng.choice([1, 1, 2, 3])
        mode = rng.choice([0, 0, 1, 2])
        s = rng.choice([1.0, 1.0, 0.5])
        if n > 1e5:
            a = min(a, 30.0)
        return dict(kind=kind, lx=lx, ly=ly, lz=lz, rho=rho, species=species,
                    chains=rng.choice([0.0, 0.1]) if species == 3 else 0.0, a=a, gamma=gamma, s=s,
                    dt=rng.choice([0.01, 0.005]), lam=rng.choice([0.5, 0.5, 0.65]), skin=rng.choice([0.3, 0.4, 0.5]),
                    det=rng.choice([0, 0, 1]), body_mode=mode, body=0.055 if mode else 0.0, steps=rng.randint(8, 14),
                    every=rng.choice([0, 0, 1, 5]))
    if kind == "forces":
        rho = rng.choice([3.0, 5.0, 8.0])
        lx, ly, lz = _box(rng, _log(rng, 2000, 6e5), rho)
        return dict(kind=kind, lx=lx, ly=ly, lz=lz, rho=rho, species=rng.choice([1, 2]), a=a, gamma=gamma, s=s,
                    dt=0.01, skin=rng.choice([0.3, 0.4]), det=rng.choice([0, 1]))
    if kind == "static":
        lx, ly, lz = _box(rng, _log(rng, 200, 1.1e5), rho)
        mode = rng.choice([0, 1, 2])
        return dict(kind=kind, lx=lx, ly=ly, lz=lz, rho=rho, species=rng.choice([1, 2]), a=a, gamma=gamma, s=s,
                    dt=0.01, body_mode=mode, body=0.055 if mode else 0.0)
    if kind == "profile":
        lx, ly, lz = _box(rng, _log(rng, 5000, 1e6), rho)
        return dict(kind=kind, lx=lx, ly=ly, lz=lz, rho=rho, nbins=rng.randint(20, 200))
    if kind == "ensemble":
        lmin = rng.randint(4, 7)
        return dict(kind=kind, boxes=int(_log(rng, 8, 200)), lmin=lmin, lmax=rng.randint(lmin, 10), rho=3.0,
                    s=rng.choice([1.0, 0.5]), dt=0.01, lam=rng.choice([0.5, 0.65]), steps=rng.randint(16, 30))
    lmin = rng.randint(6, 12)
    return dict(kind=kind, boxes=rng.randint(6, 18), lmin=lmin, lmax=rng.randint(lmin, 30), rho=3.0, s=s, dt=0.01,
                lam=0.5, skin=rng.choice([0.3, 0.4]), steps_min=60, steps_max=rng.randint(60, 100))


# ------------------------------------------------------------------ the inputs
def _count(case):
    return max(1, int(round(case["rho"] * case["lx"] * case["ly"] * case["lz"])))


def _fold(x, box):
    """FP32 positions inside the box, as the engine stores them."""
    x = np.mod(x, box).astype(np.float32)
    lim = np.asarray(box, np.float32)
    return np.where(x >= lim, np.float32(0.0), x)


def _maxwell(g, n):
    v = g.standard_normal((n, 3))
    v -= v.mean(axis=0, keepdims=True)
    return v.astype(np.float32)


def _a_matrix(case):
    """Like species repel with a; the last of three (tails) repels the others
    three times as strongly, the second of two by half more."""
    k, a = case["species"], case["a"]
    m = np.full((k, k), a)
    if k == 2:
        m[0, 1] = m[1, 0] = 1.5 * a
    if k == 3:
        m[0, 2] = m[2, 0] = m[1, 2] = m[2, 1] = 3.0 * a
    return m


def _state(case, seed):
    """x, v (FP32), species, bonds of one box, from the seed alone."""
    g = np.random.default_rng(seed)
    box = np.array([case["lx"], case["ly"], case["lz"]])
    n = _count(case)
    x = g.random((n, 3)) * box
    species = bonds = None
    k = case.get("species", 1)
    if k > 1:
        species = g.integers(0, k, n).astype(np.int32)
    if case.get("chains", 0.0) > 0.0:
        # chains of one head and three tails, random walks of step 0.7
        m = int(round(case["chains"] * n / 4.0))
        step = g.standard_normal((m, 3, 3))
        step *= 0.7 / np.linalg.norm(step, axis=2, keepdims=True)
        x[:4 * m] = (x[:m, None, :] + np.concatenate([np.zeros((m, 1, 3)), np.cumsum(step, axis=1)], axis=1)).reshape(-1, 3)
        species = np.zeros(n, np.int32)
        species[:4 * m] = np.tile(np.array([1, 2, 2, 2], np.int32), m)
        b = (np.arange(m, dtype=np.uint32)[:, None] * 4 + np.arange(3, dtype=np.uint32)[None, :]).reshape(-1)
        bonds = np.stack([b, b + 1], axis=1).astype(np.uint32)
    return _fold(x, box), _maxwell(g, n), species, bonds


def _boxes(case, seed):
    """The boxes of an ensemble or a serving batch: every size of the range in
    turn, step counts spread evenly; parameters and states from the seed."""
    g = np.random.default_rng(seed)
    out = []
    for k in range(case["boxes"]):
        L = float(case["lmin"] + k % (case["lmax"] - case["lmin"] + 1))
        box = (L, L, L)
        n = int(round(case["rho"] * L ** 3))
        steps = case["steps"] if "steps" in case else (
            case["steps_min"] + k * 7919 % 101 * (case["steps_max"] - case["steps_min"]) // 100)
        out.append(dict(box=box, n=n, a=float(g.uniform(15.0, 40.0)), gamma=float(g.uniform(3.0, 6.0)),
                        seed=int(g.integers(1, 1 << 30)), steps=steps,
                        x=_fold(g.random((n, 3)) * np.array(box), np.array(box)), v=_maxwell(g, n)))
    return out


def _pinned(n):
    return torch.zeros((n, 3), dtype=torch.float64, pin_memory=True)


def _body(case):
    return (case["body"], 0.0, 0.0)


def _moved(x, last, box):
    """Minimum-image displacement since `last`, which becomes x (FP32, GPU)."""
    d = x - last
    d -= box * torch.round(d / box)
    last.copy_(x)
    return d


def _origin(boxes):
    """What the displacements of many boxes are measured from."""
    return dict(last=torch.from_numpy(np.concatenate([b["x"] for b in boxes])).float().cuda(),
                box=torch.cat([torch.full((b["n"], 1), b["box"][0]) for b in boxes]).cuda())


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ensemble", "serve"):
        boxes = _boxes(case, seed)
        if kind == "ensemble":
            ens = dpd.Ensemble()
            ids = [ens.add(b["box"], [[b["a"]]], b["gamma"], 1.0, RC, case["s"], case["dt"], b["x"], b["v"],
                           lam=case["lam"], seed=b["seed"]) for b in boxes]
            ens.step(0)  # the initial forces
            ens.sync()
            return dict(case=case, ens=ens, ids=ids, **_origin(boxes))
        srv = dpd.Server(max_active=32, chunk_steps=100, skin=case["skin"])
        for b in boxes:
            b["x"], b["v"] = b["x"].astype(np.float64), b["v"].astype(np.float64)
        return dict(case=case, srv=srv, boxes=boxes, **_origin(boxes))
    x, v, species, bonds = _state(case, seed)
    box = (case["lx"], case["ly"], case["lz"])
    n = x.shape[0]
    if kind == "static":
        pos, vel = torch.zeros((n, 4)), torch.zeros((n, 4))
        pos[:, :3], vel[:, :3] = torch.from_numpy(x), torch.from_numpy(v)
        if species is not None:
            pos[:, 3] = torch.from_numpy(species.view(np.float32))  # the bits of the species
        prm = dpd.dpd_static_params_from(box, _a_matrix(case), case["gamma"], 1.0, RC, case["s"], case["dt"], seed=seed,
                                         body_mode=case["body_mode"], body=_body(case))
        return dict(case=case, prm=prm, n=n, pos=pos.cuda(), vel=vel.cuda(),
                    tag=torch.arange(n, dtype=torch.int32, device="cuda"),
                    out=torch.zeros((n, 4), device="cuda"))
    if kind == "profile":
        sim = dpd.Sim(box, [[15.0]], 4.5, 1.0, RC, 1.0, 0.01, skin=0.4)
        sim.set_state(x, v)
        return dict(case=case, sim=sim)
    kw = {}
    if kind == "run":
        kw = dict(lam=case["lam"], body_mode=case["body_mode"], body=_body(case))
    sim = dpd.Sim(box, _a_matrix(case), case["gamma"], 1.0, RC, case["s"], case["dt"], skin=case["skin"], seed=seed,
                  deterministic=case["det"], **kw)
    sim.set_state(x, v, species=species)
    if bonds is not None:
        sim.set_bonds(bonds, 100.0, 0.7)
    if kind == "forces":
        return dict(case=case, sim=sim)
    every = case["every"]
    return dict(case=case, sim=sim, x=_pinned(n), v=_pinned(n), last=torch.from_numpy(x).cuda(),
                box=torch.tensor(box, dtype=torch.float32, device="cuda"), obs=dpd.ObsBuffer(case["steps"] // every) if every else None)


# -------------------------------------------------------------------- the pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        sim, every = state["sim"], case["every"]
        if every:
            # the log: a record every few steps, read after the block
            buf = state["obs"]
            for k in range(buf.k):
                sim.step_async(every)
                sim.observables_async(buf, k)
            sim.step_async(case["steps"] - buf.k * every)
            sim.sync()
            rec = [buf.get(k) for k in range(buf.k)]
        else:
            sim.step(case["steps"])
            rec = [sim.observables()]
        sim.state(state["x"].numpy(), state["v"].numpy())
        # the analysis works on the GPU, in FP32
        x, v = (state[k].to("cuda", non_blocking=True).float() for k in "xv")
        return dict(moved=_moved(x, state["last"], state["box"]), v=v,
                    temperature=np.array([o["temperature"] for o in rec], np.float32),
                    pressure=np.array([o["pressure"] for o in rec], np.float32))
    if kind == "forces":
        state["sim"].build_neighbors()
        return state["sim"].forces().astype(np.float32)
    if kind == "static":
        dpd.dpd_forces_static(state["prm"], state["n"], state["pos"].data_ptr(), state["vel"].data_ptr(),
                              state["tag"].data_ptr(), 7, state["out"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if kind == "profile":
        sums, counts = state["sim"].profile(1, 0, case["nbins"])
        return dict(sums=sums, counts=counts)
    if kind == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        ens.sync()
        got = [ens.state(i)[:2] for i in state["ids"]]
        x, v = (torch.from_numpy(np.concatenate([g[q] for g in got])).cuda().float() for q in (0, 1))
        return dict(moved=_moved(x, state["last"], state["box"]), v=v)
    srv = state["srv"]
    tickets = [srv.submit(b["box"], [[b["a"]]], b["gamma"], 1.0, RC, case["s"], case["dt"], b["x"], b["v"], b["steps"],
                          seed=b["seed"]) for b in state["boxes"]]
    got = [srv.wait(t) for t in tickets]
    if any(r["status"] != 0 for r in got):
        raise RuntimeError("a box failed")
    x, v = (torch.from_numpy(np.concatenate([r[q] for r in got])).cuda().float() for q in "xv")
    return dict(moved=_moved(x, state["last"].clone(), state["box"]), v=v,
                temperature=np.array([r["obs"]["temperature"] for r in got], np.float32))


# -------------------------------------------------------------- what it is worth
# FP32/INT32 operations of an interacting pair (distance, weights, pair hash,
# Gaussian, force, both sums) and of a particle's integration
PAIR_OPS, PARTICLE_OPS = 100.0, 25.0


def _sizes(case):
    """[(particles, density, evaluations)] of a pass."""
    if case["kind"] in ("ensemble", "serve"):
        L3 = sum(L ** 3 for L in range(case["lmin"], case["lmax"] + 1)) / (case["lmax"] - case["lmin"] + 1)
        steps = case["steps"] if "steps" in case else 0.5 * (case["steps_min"] + case["steps_max"])
        return case["boxes"] * case["rho"] * L3, case["rho"], steps
    return _count(case), case["rho"], case["steps"] if case["kind"] == "run" else 1


def work(case):
    """Positions, velocities in and out once a pass; unique pairs inside r_c
    of a uniform fluid, evaluated once a step."""
    n, rho, steps = _sizes(case)
    if case["kind"] == "profile":
        return {"bytes": 8.0 * n + 16.0 * case["nbins"], "flops": 2.0 * n}
    pairs = 0.5 * rho * 4.0 / 3.0 * math.pi * RC ** 3 * n
    integrate = PARTICLE_OPS * n if case["kind"] in ("run", "ensemble", "serve") else 0.0
    back = 24.0 if case["kind"] in ("run", "ensemble", "serve") else 12.0
    return {"bytes": (24.0 + back) * n, "flops": steps * (PAIR_OPS * pairs + integrate)}


# ---------------------------------------------------- the same in 64 bits, plainly
class _Exact:
    """DPD boxes side by side in FP64 torch: all pairs inside r_c found anew
    at every evaluation, over cells of side >= r_c."""

    def __init__(self, boxes, s, dt, lam, body_mode=0, body=0.0):
        """boxes: dicts of box, x, v, species, a (k x k), gamma, seed (kT = 1)."""
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f8 = dict(dtype=torch.float64, device=dev)
        self.dev, self.s, self.dt, self.lam, self.body_mode, self.body = dev, s, dt, lam, body_mode, body
        sizes = [len(b["x"]) for b in boxes]
        self.x = torch.cat([torch.from_numpy(np.asarray(b["x"], np.float64)) for b in boxes]).to(dev)
        self.v = torch.cat([torch.from_numpy(np.asarray(b["v"], np.float64)) for b in boxes]).to(dev)
        self.moved = torch.zeros_like(self.x)
        self.of = torch.repeat_interleave(torch.arange(len(boxes)), torch.tensor(sizes)).to(dev)
        self.ends = np.cumsum([0] + sizes)
        self.tag = torch.cat([torch.arange(k) for k in sizes]).to(dev)
        self.L = torch.tensor([b["box"] for b in boxes], **f8)
        self.sp = None
        if boxes[0].get("species") is not None:
            self.sp = torch.cat([torch.from_numpy(b["species"].astype(np.int64)) for b in boxes]).to(dev)
        self.a = torch.tensor(np.array([np.asarray(b["a"], np.float64) for b in boxes]), **f8)
        self.gamma = torch.tensor([b["gamma"] for b in boxes], **f8)
        self.k0 = torch.tensor([b["seed"] & 0xFFFFFFFF for b in boxes], device=dev)
        self.k1 = torch.tensor([b["seed"] >> 32 for b in boxes], device=dev)
        self.bonds = None
        # cells of all boxes, and the 13 forward neighbours of each with the
        # box lengths to add to their positions
        nc = [[max(1, int(l / (RC * (1 + 1e-9)))) for l in b["box"]] for b in boxes]
        self.nc = torch.tensor(nc, device=dev)
        base = np.cumsum([0] + [c[0] * c[1] * c[2] for c in nc])
        self.base, self.ncell = torch.tensor(base[:-1], device=dev), int(base[-1])
        fwd = [(0, 0, 0)] + [(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1) if (k, j, i) > (0, 0, 0)]
        self.near, self.shift = [], []
        for o in fwd:
            near, shift = [], []
            for c, b, at in zip(nc, boxes, base[:-1]):
                cz, cy, cx = np.meshgrid(*[np.arange(c[q]) for q in (2, 1, 0)], indexing="ij")
                idx, sh = [], []
                for p, q in ((cx, 0), (cy, 1), (cz, 2)):
                    t = p + o[q]
                    sh.append(np.where(t < 0, -b["box"][q], np.where(t >= c[q], b["box"][q], 0.0)).reshape(-1))
                    idx.append(np.mod(t, c[q]))
                near.append(((idx[2] * c[1] + idx[1]) * c[0] + idx[0]).reshape(-1) + at)
                shift.append(np.stack(sh, axis=1))
            self.near.append(torch.from_numpy(np.concatenate(near)).to(dev))
            self.shift.append(torch.from_numpy(np.concatenate(shift)).to(dev))

    def pairs(self):
        """i, j, x_i - x_j of every pair inside r_c."""
        x, L = self.x, self.L[self.of]
        nc = self.nc[self.of]
        c3 = torch.minimum((x / L * nc).long().clamp(min=0), nc - 1)
        cell = self.base[self.of] + (c3[:, 2] * nc[:, 1] + c3[:, 1]) * nc[:, 0] + c3[:, 0]
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=self.ncell)
        start = torch.cumsum(count, 0) - count
        cap = int(count.max())
        table = torch.full((self.ncell, cap), -1, dtype=torch.int64, device=self.dev)
        sorted_cell = cell[order]
        table[sorted_cell, torch.arange(len(x), device=self.dev) - start[sorted_cell]] = order
        xs = torch.cat([x, torch.full((1, 3), 1e9, dtype=torch.float64, device=self.dev)])  # slot -1
        out = []
        chunk = max(1, 40_000_000 // (cap * cap))
        upper = torch.triu(torch.ones((cap, cap), dtype=torch.bool, device=self.dev), 1)
        for k, (near, shift) in enumerate(zip(self.near, self.shift)):
            for c0 in range(0, self.ncell, chunk):
                A, B = table[c0:c0 + chunk], table[near[c0:c0 + chunk]]
                xa, xb = xs[A], xs[B] + shift[c0:c0 + chunk, None, :]
                d2 = torch.zeros((A.shape[0], cap, cap), dtype=torch.float64, device=self.dev)
                for q in range(3):
                    t = xa[:, :, None, q] - xb[:, None, :, q]
                    d2 += t * t
                ok = (d2 < RC * RC) & (A >= 0)[:, :, None] & (B >= 0)[:, None, :]
                if k == 0:
                    ok &= upper
                c, p, q = torch.nonzero(ok, as_tuple=True)
                out.append((A[c, p], B[c, q], xa[c, p] - xb[c, q]))
        return tuple(torch.cat([o[q] for o in out]) for q in range(3))

    def tea(self, v0, v1, k0, k1, rounds):
        m, total = 0xFFFFFFFF, 0
        k2, k3 = 0x243F6A88, 0x85A308D3
        for _ in range(rounds):
            total = (total + 0x9E3779B9) & m
            v0 = (v0 + ((((v1 << 4) + k0) & m) ^ ((v1 + total) & m) ^ (((v1 >> 5) + k1) & m))) & m
            v1 = (v1 + ((((v0 << 4) + k2) & m) ^ ((v0 + total) & m) ^ (((v0 >> 5) + k3) & m))) & m
        return v0, v1

    def force(self, vel, step):
        """The total force at x with velocities vel; also the virial by box."""
        rev = torch.zeros_like(self.tag)
        for b in range(32):
            rev |= ((self.tag >> b) & 1) << (31 - b)
        s0, s1 = self.tea(rev, torch.full_like(rev, step & 0xFFFFFFFF), self.k0[self.of], self.k1[self.of], 16)
        sig = s0 ^ s1
        i, j, d = self.pairs()
        r = (d * d).sum(1).sqrt()
        keep = r > 0
        i, j, d, r = i[keep], j[keep], d[keep], r[keep]
        of = self.of[i]
        e = d / r[:, None]
        w = (1.0 - r / RC).clamp(min=0.0)
        wr = w ** self.s
        A, B = self.tea(torch.minimum(sig[i], sig[j]), torch.maximum(sig[i], sig[j]), self.k0[of], self.k1[of], 4)
        xi = (-2.0 * torch.log((A + 1).double() * 2.0 ** -32)).sqrt() * torch.cos(math.pi * (B & 0x7FFFFFFF).double() * 2.0 ** -31)
        xi = torch.where(B >= 1 << 31, -xi, xi)
        a = self.a[of, 0, 0] if self.sp is None else self.a[of, self.sp[i], self.sp[j]]
        g = self.gamma[of]
        F = a * w - g * wr * wr * (e * (vel[i] - vel[j])).sum(1) + (2.0 * g / self.dt).sqrt() * wr * xi
        f = torch.zeros_like(self.x)
        f.index_add_(0, i, F[:, None] * e)
        f.index_add_(0, j, -F[:, None] * e)
        vir = torch.zeros(len(self.L), dtype=torch.float64, device=self.dev).index_add_(0, of, a * w * r)
        if self.bonds is not None:
            p, q = self.bonds[:, 0], self.bonds[:, 1]
            d = self.x[p] - self.x[q]
            L = self.L[self.of[p]]
            d = d - L * torch.round(d / L)
            r = (d * d).sum(1).sqrt()
            t = -100.0 * (r - 0.7)
            f.index_add_(0, p, (t / r)[:, None] * d)
            f.index_add_(0, q, -(t / r)[:, None] * d)
            vir.index_add_(0, self.of[p], t * r)
        if self.body_mode == 1:
            f[:, 0] += self.body
        elif self.body_mode == 2:
            f[:, 0] += torch.where(self.x[:, 1] < 0.5 * self.L[self.of][:, 1], self.body, -self.body)
        self.virial = vir
        return f

    def displacement(self):
        L = self.L[self.of]
        return self.moved - L * torch.round(self.moved / L)

    def observe(self):
        """Temperature and pressure by box."""
        n = torch.bincount(self.of).double()
        v2 = torch.zeros(len(self.L), dtype=torch.float64, device=self.dev).index_add_(0, self.of, (self.v ** 2).sum(1))
        t = torch.where(n > 1, v2 / (3.0 * n - 3.0), torch.zeros_like(n))
        return t.cpu().numpy(), ((v2 + self.virial) / (3.0 * self.L.prod(1))).cpu().numpy()

    def advance(self, steps, after=None):
        f = self.force(self.v, 0)
        L = self.L[self.of]
        for k in range(steps):
            dx = self.dt * self.v + 0.5 * self.dt ** 2 * f
            self.moved += dx
            self.x = self.x + dx
            self.x = self.x - L * torch.floor(self.x / L)
            fn = self.force(self.v + self.lam * self.dt * f, k + 1)
            self.v = self.v + 0.5 * self.dt * (f + fn)
            f = fn
            if after is not None:
                after(k + 1)


def exact(case, seed):
    kind = case["kind"]
    n, _, steps = _sizes(case)
    if n * steps > 1.0e8:
        return None  # minutes in FP64
    if kind in ("ensemble", "serve"):
        boxes = _boxes(case, seed)
        for b in boxes:
            b["a"] = [[b["a"]]]
        sys = _Exact(boxes, case["s"], case["dt"], case["lam"])
        rows = [slice(int(p), int(q)) for p, q in zip(sys.ends[:-1], sys.ends[1:])]
        moved, v, temp = [None] * len(boxes), [None] * len(boxes), np.zeros(len(boxes))

        def after(k):
            done = [b for b, box in enumerate(boxes) if box["steps"] == k]
            if done:
                t = sys.observe()[0]
                for b in done:
                    moved[b], v[b], temp[b] = sys.displacement()[rows[b]].cpu(), sys.v[rows[b]].cpu(), t[b]

        sys.advance(max(b["steps"] for b in boxes), after)
        out = dict(moved=torch.cat(moved), v=torch.cat(v))
        if kind == "serve":
            out["temperature"] = temp
        return out
    x, v, species, bonds = _state(case, seed)
    if kind == "profile":
        nb = case["nbins"]
        # the bin of a position is decided in FP32, the precision it is held in
        b = np.minimum((x[:, 1] * np.float32(np.float32(nb) / np.float32(case["ly"]))).astype(np.int64), nb - 1)
        return dict(sums=np.bincount(b, weights=v[:, 0].astype(np.float64), minlength=nb),
                    counts=np.bincount(b, minlength=nb).astype(np.float64))
    box = dict(box=(case["lx"], case["ly"], case["lz"]), x=x, v=v, species=species, a=_a_matrix(case), gamma=case["gamma"],
               seed=seed)
    sys = _Exact([box], case["s"], case["dt"], case.get("lam", 0.5), case.get("body_mode", 0), case.get("body", 0.0))
    if kind == "forces":
        return sys.force(sys.v, 0)
    if kind == "static":
        return torch.cat([sys.force(sys.v, 7), torch.zeros((len(x), 1), dtype=torch.float64, device=sys.dev)], dim=1)
    if bonds is not None:
        sys.bonds = torch.from_numpy(bonds.astype(np.int64)).to(sys.dev)
    temp, press = [], []
    every = case["every"] or case["steps"]

    def log(k):
        if k % every == 0:
            t, p = sys.observe()
            temp.append(t[0])
            press.append(p[0])

    sys.advance(case["steps"], log)
    return dict(moved=sys.displacement(), v=sys.v, temperature=np.array(temp), pressure=np.array(press))
