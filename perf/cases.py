"""What a user of this framework has it do, as measurable cases.

A case names a kind of work and its sizes.  `listed` gives the fixed cases,
`draw` more of the same ranges, `prepare` what a program holds before the call
(contexts, batches, trainers, device arrays), `run` one pass through the public
entry points, `work` the bytes and operations that a pass cannot do without and
`exact` its outputs in 64-bit arithmetic where they have such a value.

Kinds of pass
  cycle        one simulation: some MD/CR-MC cycles (one MD step around one
               sweep of trials), then the state is read
  batch        replicas side by side: some captured cycles, then every
               replica's configuration is read into arrays on the GPU
  batch_io     a host program drives the step: every replica's configuration is
               uploaded from pinned memory, one cycle, everything is read back
  electrolyte  replicas of the weak-acid electrolyte under the global schedule
               (DSF or Ewald electrostatics): sweeps, or MD steps around sweeps
  forces       one conservative force evaluation, the forces read
  train        minibatch steps of the delayed-acceptance surrogate, the weights
               and Adam's moments read

The configurations are made here rather than by `workloads`, whose placement by
rejection takes seconds: chains are self-avoiding walks on a cubic lattice with
bonds of about 0.97 sigma, ions and single groups sit at random on a coarser
lattice with jitter, clear of the chains.  Sizes and parameters are those of the
systems in `workloads` and of the benchmark.
"""
import math

import numpy as np
import torch

from paper_2109_07527_gb300 import crmc, workloads as W

DT, GAMMA = 0.005, 1.0
CONTEXT_TUNING = 26  # sweeps after which a context's launch-shape tuner has settled
BATCH_TUNING = 50    # the same for a batch
FLOPS_PER_ROW = 2 * (48 * 128 + 2 * 128 * 128) + 2 * (4 * 128 * 128 + 128 * 48)  # training: forward and backward


def listed():
    return [
        # the smallest simulation: one short polyacid in a small box, a few cycles between two samples
        dict(name="chain_cycle", kind="cycle", system="chains", chains=1, beads=50, L=40.0, rc=10.0, pairs=64,
             pH=5.0, pK=5.0, pIS=2.0, trials=10, cycles=4),
        # one replica of the polyelectrolyte solution at its pKa
        dict(name="solution_cycle", kind="cycle", system="chains", chains=16, beads=200, L=120.0, rc=12.0, pairs=4000,
             pH=4.5, pK=4.5, pIS=1.066, trials=10, cycles=4),
        # the large box: 20,000 sites, 50,000 ions
        dict(name="large_box_cycle", kind="cycle", system="chains", chains=100, beads=200, L=250.0, rc=12.0,
             pairs=25000, pH=4.5, pK=4.5, pIS=1.226, trials=10, cycles=4),
        # two charge-regulating nanoparticles as rigid bodies in salt solution
        dict(name="nanoparticles", kind="cycle", system="nanoparticles", sites=1000, L=100.0, radius=5.0, gap=12.0,
             pIS=1.69897, pH=7.0, trials=10, cycles=4),
        # the benchmark's titration curve: thirteen pH points of the polyelectrolyte solution in one batch
        dict(name="ph_sweep", kind="batch", replicas=13, chains=16, beads=200, L=120.0, pairs=4000, pK=4.5,
             pIS=1.066, pH_lo=2.0, pH_hi=8.0, trials=10, cycles=4, da=False),
        # the same driven by a host program that uploads and reads every configuration at every step
        dict(name="ph_sweep_host_driven", kind="batch_io", replicas=13, chains=16, beads=200, L=120.0, pairs=4000,
             pK=4.5, pIS=1.066, pH_lo=2.0, pH_hi=8.0, trials=10, cycles=1, da=False),
        # the same with a surrogate in front of the exact energies
        dict(name="ph_sweep_delayed", kind="batch", replicas=13, chains=16, beads=200, L=120.0, pairs=4000, pK=4.5,
             pIS=1.066, pH_lo=2.0, pH_hi=8.0, trials=10, cycles=2, da=True),
        # a ragged batch: 64 single chains of 50 to 1000 beads, boxes of 37 to 100 sigma, pH 2 to 10
        dict(name="titration_ragged", kind="batch", replicas=64, chains=1, beads_lo=50, beads_hi=1000, pK=5.0,
             pIS=2.0, pH_lo=2.0, pH_hi=10.0, trials=10, cycles=4, da=False),
        # the method comparison's electrolyte: one trial at a time in each box, boxes side by side
        dict(name="electrolyte_sweeps", kind="electrolyte", replicas=128, acids=500, L=100.0, rc=20.0, trials=250,
             kmax=0, sweeps=2, md=False),
        # the same under Ewald electrostatics, with an MD step around each sweep
        dict(name="electrolyte_ewald", kind="electrolyte", replicas=64, acids=500, L=100.0, rc=20.0, trials=250,
             kmax=16, sweeps=2, md=True),
        # the forces of a charged polyelectrolyte solution for a caller's own integrator
        dict(name="solution_forces", kind="forces", chains=16, beads=200, L=120.0, rc=12.0, pairs=4000, ionised=0.3),
        # the surrogate's training on recorded trials
        dict(name="surrogate_training", kind="train", batch=32768, steps=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "nanoparticles", "batch", "batch", "ragged", "batch_io", "electrolyte",
                       "electrolyte", "forces", "train"])
    if kind == "cycle":  # one chain to the large box, at the densities of the solutions
        beads = int(_log(rng, 20, 200))
        chains = int(_log(rng, 1, 100))
        L = round(max(40.0, (chains * beads / _log(rng, 0.8e-3, 1.9e-3)) ** (1.0 / 3.0)), 2)
        L = min(L, 250.0)
        rc = 12.0 if L > 48.5 else 10.0
        return dict(kind="cycle", system="chains", chains=chains, beads=beads, L=L, rc=rc,
                    pairs=int(L ** 3 * _log(rng, 1e-3, 2.3e-3)), pH=round(rng.uniform(3.0, 7.0), 2), pK=4.5,
                    pIS=round(rng.uniform(1.1, 2.0), 3), trials=rng.randint(5, 16), cycles=rng.randint(1, 4))
    if kind == "nanoparticles":
        sites = int(_log(rng, 200, 1000))
        return dict(kind="cycle", system="nanoparticles", sites=sites, L=round(rng.uniform(60.0, 100.0), 1),
                    radius=5.0, gap=round(rng.uniform(11.5, 20.0), 2), pIS=round(rng.uniform(1.7, 2.5), 3),
                    pH=round(rng.uniform(5.0, 9.0), 2), trials=rng.randint(5, 12), cycles=rng.randint(1, 4))
    if kind in ("batch", "batch_io"):
        L = round(rng.uniform(56.0, 120.0), 2)
        lo = round(rng.uniform(2.0, 5.0), 2)
        return dict(kind=kind, replicas=rng.randint(2, 13), chains=max(1, int(16 * (L / 120.0) ** 3)),
                    beads=rng.randint(150, 200), L=L, pairs=int(4000 * (L / 120.0) ** 3), pK=4.5, pIS=1.066, pH_lo=lo,
                    pH_hi=round(lo + rng.uniform(1.0, 3.0), 2), trials=rng.randint(5, 10),
                    cycles=1 if kind == "batch_io" else rng.randint(1, 3), da=rng.random() < 0.25)
    if kind == "ragged":
        lo = int(_log(rng, 50, 120))
        return dict(kind="batch", replicas=rng.randint(5, 64), chains=1, beads_lo=lo,
                    beads_hi=int(_log(rng, 2 * lo, 1000)), pK=5.0, pIS=2.0, pH_lo=2.0,
                    pH_hi=round(rng.uniform(6.0, 10.0), 2), trials=rng.randint(5, 12), cycles=rng.randint(1, 4),
                    da=False)
    if kind == "electrolyte":
        kmax = rng.choice([0, 0, rng.randint(6, 16)])
        acids = int(_log(rng, 100, 500))
        L = round(max(41.0, (acids / 5e-4) ** (1.0 / 3.0)), 2)
        return dict(kind="electrolyte", replicas=int(_log(rng, 1, 64)), acids=acids, L=L, rc=20.0,
                    trials=rng.randint(100, 250), kmax=kmax, sweeps=rng.randint(1, 2), md=rng.random() < 0.5)
    if kind == "forces":
        L = round(_log(rng, 40.0, 250.0), 2)
        return dict(kind="forces", chains=max(1, int(16 * (L / 120.0) ** 3)), beads=rng.randint(50, 200), L=L,
                    rc=12.0 if L > 48.5 else 10.0, pairs=int(4000 * (L / 120.0) ** 3),
                    ionised=round(rng.uniform(0.05, 0.9), 2))
    return dict(kind="train", batch=128 * int(_log(rng, 1, 256)), steps=rng.randint(2, 16))


# ---------------------------------------------------------------- configurations
def _walks(rng, L, chains, beads):
    """Self-avoiding walks on a cubic lattice of spacing L / G, about 0.97: lattice points and spacing."""
    G = int(L / 0.97)
    taken, points = set(), []
    dirs = rng.integers(0, 6, 8 * chains * beads + 4096).tolist()
    moves = ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))
    k = 0
    for _ in range(chains):
        while True:  # until a walk of full length has been grown
            p = tuple(rng.integers(0, G, 3).tolist())
            walk, here = [p], {p}
            if p in taken:
                continue
            stuck = 0
            while len(walk) < beads and stuck < 40:
                d = moves[dirs[k]]
                k = (k + 1) % len(dirs)
                q = ((p[0] + d[0]) % G, (p[1] + d[1]) % G, (p[2] + d[2]) % G)
                if q in here or q in taken:
                    stuck += 1
                    continue
                stuck = 0
                p = q
                walk.append(p)
                here.add(p)
            if len(walk) == beads:
                break
        taken |= here
        points += walk
    return np.array(points, np.int64).reshape(-1, 3), L / G, G


def _coarse(rng, L, G, count, beads=None, clear=None):
    """`count` points at random on a lattice of twice the spacing with jitter (no two closer than about 1.3),
    none next to a point of `beads`, and only where clear(xyz) holds."""
    s, H = L / G, (G - 1) // 2
    free = np.ones((H, H, H), bool)
    if beads is not None and len(beads):
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dz in (-1, 0, 1):
                    q = (beads + (dx, dy, dz)) % G
                    q = q[(q % 2 == 0).all(1)] // 2
                    q = q[(q < H).all(1)]
                    free[q[:, 0], q[:, 1], q[:, 2]] = False
    at = np.flatnonzero(free.ravel())
    at = rng.permutation(at)
    xyz = np.stack(np.unravel_index(at, free.shape), 1) * (2.0 * s) + rng.uniform(-0.3, 0.3, (len(at), 3))
    if clear is not None:
        xyz = xyz[clear(xyz)]
    if len(xyz) < count:
        raise ValueError("the box is too small for its ions")
    return _wrapped(xyz[:count], L)


def _wrapped(x, L):
    x = np.mod(x, L).astype(np.float32)
    x[x >= np.float32(L)] = 0.0
    return x


def _workload(name, rng, parts, params, extra, bonds=None, bodies=None):
    """Particles from (xyz, type, class, state, pK) parts, in order."""
    n = sum(len(p[0]) for p in parts)
    col = lambda i, t: np.concatenate([np.broadcast_to(np.asarray(p[i], t), (len(p[0]),)) for p in parts]).copy()
    return W.Workload(name=name, xyz=np.concatenate([p[0] for p in parts]).astype(np.float32),
                      type=col(1, np.int32), cls=col(2, np.int32), state=col(3, np.int8), pK=col(4, np.float64),
                      bonds=np.zeros((0, 2), np.int32) if bonds is None else bonds,
                      vel=rng.normal(size=(n, 3)).astype(np.float32), params=params, capacity=n + extra,
                      meta=dict(bodies=bodies))


def _alternating(pairs):
    return np.where(np.arange(2 * pairs) % 2 == 0, W.XP, W.XM).astype(np.int32)


def _chains(rng, chains, beads, L, rc, pairs, pH, pK, pIS, trials, ionised=0.0):
    points, s, G = _walks(rng, L, chains, beads)
    n = chains * beads
    first = np.arange(n)[np.arange(n) % beads != beads - 1]
    bonds = np.stack([first, first + 1], 1).astype(np.int32)
    counter = int(ionised * n)  # that many acids have given their X+ away
    state = np.zeros(n, np.int8)
    state[rng.permutation(n)[:counter]] = 1
    ions = _coarse(rng, L, G, 2 * pairs + counter, beads=points)
    kinds = np.concatenate([_alternating(pairs), np.full(counter, W.XP, np.int32)])
    params = W.default_params(box_L=L, rc=rc, lB=2.0, pH=pH, pIS_plus=pIS, pIS_minus=pIS, trials_per_domain=trials)
    parts = [(_wrapped(points * s, L), W.ACID, 0, state, pK), (ions, kinds, 0, 0, 0.0)]
    return _workload("chains", rng, parts, params, n + 4096 + pairs, bonds=bonds)


def _nanoparticles(rng, sites, L, radius, gap, pIS, pH, trials):
    mid = np.full(3, L / 2)
    centres = [mid - (gap / 2, 0, 0), mid + (gap / 2, 0, 0)]
    parts = []
    for c, t in zip(centres, (W.ACID, W.BASE)):
        parts.append((_wrapped(c[None, :], L), W.CORE, 1, 0, 0.0))
        parts.append((_wrapped(c + W.fibonacci_sphere(sites, radius - 0.5), L), t, W.CLS_NONE, 0, 4.0))

    def clear(x):
        ok = np.ones(len(x), bool)
        for c in centres:
            d = x - c
            d -= L * np.round(d / L)
            ok &= (d * d).sum(1) > (radius + 0.7) ** 2
        return ok

    pairs = int(round(0.602214076 * (L * 0.355) ** 3 * 10 ** (-pIS)))
    parts.append((_coarse(rng, L, int(L / 0.97), 2 * pairs, clear=clear), _alternating(pairs), 0, 0, 0.0))
    delta = [0.0] * 16
    delta[1] = delta[4] = radius - 0.5
    delta[5] = 2 * radius - 1.0
    params = W.default_params(box_L=L, rc=12.0, lB=0.7, pH=pH, pIS_plus=pIS, pIS_minus=pIS, wca_del=delta,
                              trials_per_domain=trials)
    return _workload("nanoparticles", rng, parts, params, 4 * sites + 8192,
                     bodies=([0, 1 + sites], [1 + sites, 1 + sites]))


def _electrolyte(rng, acids, L, rc, trials, kmax):
    xyz = _coarse(rng, L, int(L / 0.97), acids)
    params = W.default_params(box_L=L, rc=rc, lB=2.0, alpha=0.15, pH=7.0, pIS_plus=2.0, pIS_minus=2.0, schedule=1,
                              trials_per_domain=trials, ewald_kmax=kmax)
    return _workload("electrolyte", rng, [(xyz, W.ACID, 0, 0, 6.5)], params, 4096)


def _beads(case, r):
    """Chain length of replica r: the middles of equal parts of the range's logarithm."""
    a, b = math.log(case["beads_lo"]), math.log(case["beads_hi"])
    return int(round(math.exp(a + (b - a) * (r + 0.5) / case["replicas"])))


def _replicas(case, rng):
    """The workloads of a batch, pH evenly spaced; in a ragged batch the chain lengths are spread over their
    logarithm and no pH goes with any length in particular."""
    R = case["replicas"]
    pHs = np.linspace(case["pH_lo"], case["pH_hi"], R).tolist()
    out = []
    for r in range(R):
        pH = pHs[r]
        if "beads_lo" in case:
            pH = pHs[(r * 29 + 7) % R]
            beads = _beads(case, r)
            L = (beads / 1e-3) ** (1.0 / 3.0)
            pairs = max(1, int(round(0.602214076 * (L * 0.355) ** 3 * 10 ** (-case["pIS"]))))
        else:
            beads, L, pairs = case["beads"], case["L"], case["pairs"]
        out.append(_chains(rng, case["chains"], beads, L, 12.0, pairs, pH, case["pK"], case["pIS"], case["trials"]))
    return out


# ---------------------------------------------------------------- what a program holds
class _Frames:
    """One array per quantity for all replicas of a batch, on the GPU or in pinned host memory."""

    def __init__(self, contexts, device):
        R, self.stride = len(contexts), max(c.capacity for c in contexts)
        make = lambda *shape, dtype: (torch.zeros(shape, dtype=dtype, device="cuda") if device else
                                      torch.zeros(shape, dtype=dtype).pin_memory())
        self.motion = make(2, R, self.stride, 3, dtype=torch.float32)   # positions, velocities
        self.id = make(R, self.stride, dtype=torch.int64)
        self.what = make(2, R, self.stride, dtype=torch.int32)          # type, class
        self.state = make(R, self.stride, dtype=torch.int8)
        self.n = torch.zeros(R, dtype=torch.int64).pin_memory()
        self.ptr = dict(xyz=self.motion[0].data_ptr(), vel=self.motion[1].data_ptr(), id=self.id.data_ptr(),
                        type=self.what[0].data_ptr(), cls=self.what[1].data_ptr(), state=self.state.data_ptr())

    def read(self, batch):
        batch.state_packed(self.stride, self.ptr, self.n.data_ptr())

    def load(self, batch):
        batch.load_packed(self.stride, {k: v for k, v in self.ptr.items() if k != "id"}, self.n.data_ptr())

    def arrays(self):
        """The program's own arrays; replica r's frame is their first n[r] entries."""
        return dict(motion=self.motion, id=self.id, what=self.what, state=self.state, n=self.n)


class _Sample:
    """Pinned host arrays that a program reads one context's configuration into."""

    def __init__(self, ctx):
        n = ctx.capacity
        make = lambda *shape, dtype: torch.zeros(shape, dtype=dtype).pin_memory()
        self.to = dict(xyz=make(n, 3, dtype=torch.float32), vel=make(n, 3, dtype=torch.float32),
                       id=make(n, dtype=torch.int64), type=make(n, dtype=torch.int32), cls=make(n, dtype=torch.int32),
                       state=make(n, dtype=torch.int8))
        self.ptr = {k: v.data_ptr() for k, v in self.to.items()}

    def read(self, ctx):
        """The arrays, the first n entries of each the frame, and the counts."""
        return dict(counts=ctx.state_into(**self.ptr), **self.to)


def _cycle(ctx, trials, k, gamma):
    ctx.md_begin(DT, gamma, 5000 + k)
    ctx.sweep(trials, 100 + k)
    ctx.md_end(DT, gamma, 5000 + k)


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s = dict(case=case, k=100)
    if kind == "cycle":
        gamma = GAMMA
        if case["system"] == "chains":
            w = _chains(rng, *(case[x] for x in ("chains", "beads", "L", "rc", "pairs", "pH", "pK", "pIS", "trials")))
        else:
            w = _nanoparticles(rng, *(case[x] for x in ("sites", "L", "radius", "gap", "pIS", "pH", "trials")))
            gamma = 0.05
        ctx = crmc.Context(w)
        if w.meta["bodies"]:
            ctx.set_rigid_bodies(*w.meta["bodies"])
        s.update(ctx=ctx, gamma=gamma, trials=ctx.trials_per_sweep, sample=_Sample(ctx))
        for k in range(CONTEXT_TUNING + 2):
            _cycle(ctx, s["trials"], k, gamma)
        ctx.check()
    elif kind in ("batch", "batch_io"):
        ctxs = [crmc.Context(w) for w in _replicas(case, rng)]
        if case["da"]:
            mlp = W.random_mlp(seed=int(rng.integers(1 << 30)), gain=0.7, out_gain=0.3)
            for c in ctxs:
                c.set_surrogate(mlp)
        b = crmc.Batch(ctxs)
        (b.sweep_da if case["da"] else b.sweep)(BATCH_TUNING // 2 if case["da"] else BATCH_TUNING, 3)
        for k in range(3):
            b.cycle(1, DT, GAMMA, 1 + k, 1000 + k, da=case["da"])
        frames = _Frames(ctxs, device=kind == "batch")
        frames.read(b)
        if kind == "batch_io":
            frames.load(b)
            b.cycle(1, DT, GAMMA, 50, 1050, da=case["da"])
            frames.read(b)
        s.update(ctxs=ctxs, batch=b, frames=frames)
    elif kind == "electrolyte":
        ctxs = [crmc.Context(_electrolyte(rng, *(case[x] for x in ("acids", "L", "rc", "trials", "kmax"))))
                for _ in range(case["replicas"])]
        b = crmc.Batch(ctxs)
        b.sweep(BATCH_TUNING, 3)
        frames = _Frames(ctxs, device=True)
        frames.read(b)
        s.update(ctxs=ctxs, batch=b, frames=frames)
    elif kind == "forces":
        w = _chains(rng, case["chains"], case["beads"], case["L"], case["rc"], case["pairs"], 4.5, 4.5, 1.066, 10,
                    ionised=case["ionised"])
        s.update(ctx=crmc.Context(w), n=w.n, force=torch.zeros((w.n, 3), dtype=torch.float32).pin_memory(),
                 id=torch.zeros(w.n, dtype=torch.int64).pin_memory())
    else:
        mlp, X, y = _training(case, rng)
        s.update(trainer=crmc.Trainer(mlp, max_batch=case["batch"], lr=1e-3, target_clip=20.0), X=X.cuda(), y=y.cuda())
    return s


def _training(case, rng):
    """Rows as the recorded trials give them: small whole numbers, most of them zero near the changed particles,
    and energies that grow with the charge around them."""
    rows = case["batch"] * case["steps"]
    width = np.tile(np.array([1, 2, 2, 2, 1, 3, 3, 4]), 6)
    X = np.rint(rng.normal(size=(rows, 48), scale=0.7) * width).astype(np.float32)
    pull = np.tile(np.array([3.0, 0.4, 0.25, 0.2, 0.15, 0.1, 0.08, 0.03]), 6) * np.repeat([1, 1, 0, 1, 1, 0], 8)
    y = (X @ (0.5 * pull) + 0.5 * rng.normal(size=rows)).astype(np.float32)
    return W.random_mlp(seed=int(rng.integers(1 << 30)), gain=0.5), torch.from_numpy(X), torch.from_numpy(y)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    s["k"] += 16
    k = s["k"]
    if kind == "cycle":
        for j in range(case["cycles"]):
            _cycle(s["ctx"], s["trials"], k + j, s["gamma"])
        out = s["sample"].read(s["ctx"])
        if case["system"] == "nanoparticles":
            out["bodies"] = s["ctx"].rigid_body_state()
        return out
    if kind == "batch":
        s["batch"].cycle(case["cycles"], DT, GAMMA, 100 + k, 5000 + k, da=case["da"])
        s["frames"].read(s["batch"])
        return s["frames"].arrays()
    if kind == "batch_io":
        s["frames"].load(s["batch"])
        s["batch"].cycle(1, DT, GAMMA, 100 + k, 5000 + k, da=case["da"])
        s["frames"].read(s["batch"])
        return s["frames"].arrays()
    if kind == "electrolyte":
        b = s["batch"]
        if case["md"]:
            for j in range(case["sweeps"]):
                b.md_begin(DT, GAMMA, 5000 + k + j)
                b.sweep(1, 100 + k + j)
                b.md_end(DT, GAMMA, 5000 + k + j)
        else:
            b.sweep(case["sweeps"], 100 + k)
        s["frames"].read(b)
        return s["frames"].arrays()
    if kind == "forces":
        s["ctx"].md_forces()
        s["ctx"].state_into(force=s["force"].data_ptr(), id=s["id"].data_ptr())
        return dict(force=s["force"], id=s["id"])
    B = case["batch"]
    for j in range(case["steps"]):
        loss = s["trainer"].step(s["X"][j * B:].data_ptr(), s["y"][j * B:].data_ptr(), B,
                                 want_loss=j == case["steps"] - 1)
    params, _ = s["trainer"].get()
    m, v = s["trainer"].moments()
    return dict(params=params, m=m, v=v, loss=np.float32(loss))


# ---------------------------------------------------------------- what a pass cannot do without
STATE_BYTES = 12 + 12 + 8 + 4 + 4 + 1  # position, velocity, id, type, class, state of a particle
PAIR_FLOPS, FORCE_FLOPS = 25, 40       # one damped-shifted Coulomb energy, one force with its three components
MODE_FLOPS = 16                        # one reciprocal vector's change of the structure factor and of the energy


def _box(L, rc, trials, n):
    """Particles, trials of a sweep, and pairs within the cutoff of a particle of a coloured box."""
    nc = int(2 * L / rc) // 4 * 4
    return n, (nc // 2) ** 3 * trials, n / L ** 3 * 4.0 / 3.0 * math.pi * rc ** 3


def work(case):
    kind = case["kind"]
    if kind == "train":
        rows = case["batch"] * case["steps"]
        return dict(bytes=rows * 49 * 4 + 4 * 6 * crmc.N_PARAMS, flops=rows * FLOPS_PER_ROW)
    if kind == "forces":
        n, _, pairs = _box(case["L"], case["rc"], 1, case["chains"] * case["beads"] * (1 + case["ionised"]) +
                           2 * case["pairs"])
        return dict(bytes=n * (12 + 4 + 4 + 12 + 8), flops=n * pairs / 2 * FORCE_FLOPS)
    if kind == "electrolyte":
        n = case["acids"] + 1.3 * case["acids"]  # the groups and about as many ions as they set free
        pairs = n / case["L"] ** 3 * 4.0 / 3.0 * math.pi * case["rc"] ** 3
        modes = 2.0 / 3.0 * math.pi * case["kmax"] ** 3
        flops = case["sweeps"] * (case["trials"] * 2 * (pairs * PAIR_FLOPS + modes * MODE_FLOPS) + n * modes * 8)
        if case["md"]:
            flops += case["sweeps"] * n * (pairs / 2 * FORCE_FLOPS + modes * MODE_FLOPS)
        return dict(bytes=case["replicas"] * n * 2 * STATE_BYTES, flops=case["replicas"] * flops)
    if kind == "cycle" and case["system"] == "nanoparticles":
        ions = 2 * 0.602214076 * (case["L"] * 0.355) ** 3 * 10 ** (-case["pIS"])
        boxes = [_box(case["L"], 12.0, case["trials"], 2 * case["sites"] + 2 + ions)]
    elif kind == "cycle":
        boxes = [_box(case["L"], case["rc"], case["trials"], case["chains"] * case["beads"] + 2 * case["pairs"])]
    elif "beads_lo" in case:
        beads = [_beads(case, r) for r in range(case["replicas"])]
        salt = 2 * 0.602214076 * 0.355 ** 3 * 10 ** (-case["pIS"]) / 1e-3
        boxes = [_box((x / 1e-3) ** (1.0 / 3.0), 12.0, case["trials"], x * (1 + salt)) for x in beads]
    else:
        boxes = [_box(case["L"], 12.0, case["trials"], case["chains"] * case["beads"] + 2 * case["pairs"])] * \
            case["replicas"]
    flops = sum(c * 2 * p * PAIR_FLOPS + n * p / 2 * FORCE_FLOPS for n, c, p in boxes) * case["cycles"]
    return dict(bytes=sum(n for n, _, _ in boxes) * 2 * STATE_BYTES, flops=flops)


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """Forces and training have one; a chain of accepted and rejected trials does not."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "forces":
        w = _chains(rng, case["chains"], case["beads"], case["L"], case["rc"], case["pairs"], 4.5, 4.5, 1.066, 10,
                    ionised=case["ionised"])
        return dict(force=_exact_forces(w), id=None)
    if case["kind"] == "train":
        mlp, X, y = _training(case, rng)
        return _exact_training(case, mlp, X, y)
    return None


def _exact_forces(w):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    p = w.params
    L, rc, lB, al = float(np.float32(p["box_L"])), p["rc"], p["lB"], p["alpha"]
    x = torch.from_numpy(w.xyz).to(dev, torch.float64)
    q = np.zeros(w.n)
    q[w.type == W.ACID] = -w.state[w.type == W.ACID]
    q[w.type == W.XP], q[w.type == W.XM] = 1.0, -1.0
    q = torch.from_numpy(q).to(dev)
    shift = math.erfc(al * rc) / rc ** 2 + 2 * al / math.sqrt(math.pi) * math.exp(-(al * rc) ** 2) / rc
    f = torch.zeros_like(x)
    for i in range(0, w.n, 1024):
        d = x[i:i + 1024, None, :] - x[None, :, :]
        d -= L * torch.round(d / L)
        r2 = (d * d).sum(2)
        a, b = torch.nonzero((r2 < rc * rc) & (r2 > 0), as_tuple=True)
        d, r = d[a, b], r2[a, b].sqrt()
        g = lB * q[i + a] * q[b] * (torch.erfc(al * r) / r ** 2 +
                                    2 * al / math.sqrt(math.pi) * torch.exp(-(al * r) ** 2) / r - shift) / r
        t6 = r ** -6
        g += torch.where(r < 2 ** (1 / 6), 24 * (2 * t6 * t6 - t6) / r ** 2, torch.zeros_like(r))
        f.index_add_(0, i + a, g[:, None] * d)
    bonds = torch.from_numpy(w.bonds.astype(np.int64)).to(dev)
    if len(bonds):
        d = x[bonds[:, 0]] - x[bonds[:, 1]]
        d -= L * torch.round(d / L)
        g = -p["fene_K"] / (1 - (d * d).sum(1) / p["fene_R0"] ** 2)
        f.index_add_(0, bonds[:, 0], g[:, None] * d)
        f.index_add_(0, bonds[:, 1], -g[:, None] * d)
    return f


def _exact_training(case, mlp, X, y):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    up = lambda a: torch.from_numpy(np.array(a, np.float64)).to(dev)
    names = ("W1", "b1", "W2", "b2", "W3", "b3", "w4", "b4")
    P = [up(W.bf16_to_f32(mlp[n]) if n[0] in "Ww" else mlp[n]) for n in names]
    for a in P:
        a.requires_grad_(True)
    m, v = [torch.zeros_like(a) for a in P], [torch.zeros_like(a) for a in P]
    X, y = X.to(dev), y.to(dev)
    B = case["batch"]
    for k in range(case["steps"]):
        x = X[k * B:(k + 1) * B].double()
        t = y[k * B:(k + 1) * B].double().clamp(-20.0, 20.0)
        h = torch.relu(x @ P[0].T + P[1])
        h = torch.relu(h @ P[2].T + P[3])
        h = torch.relu(h @ P[4].T + P[5])
        loss = 0.5 * ((h @ P[6] + P[7] - t) ** 2).mean()
        g = torch.autograd.grad(loss, P)
        with torch.no_grad():
            for a, da, ma, va in zip(P, g, m, v):
                ma.mul_(0.9).add_(da, alpha=0.1)
                va.mul_(0.999).add_(da * da, alpha=0.001)
                a -= 1e-3 * (ma / (1 - 0.9 ** (k + 1))) / ((va / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    flat = lambda arrays: torch.cat([a.detach().reshape(-1) for a in arrays])
    return dict(params=flat(P), m=flat(m), v=flat(v), loss=loss.detach())
