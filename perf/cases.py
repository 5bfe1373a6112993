"""What the performance of this library is measured on: the calls that a
program makes through the public entry points, over their real range.

A case is a plain dict; `kind` says which part of the library it calls:

  liquid    one Lennard-Jones system: System.step, then what a program reads
            at the end of a segment of a run (particles on the device,
            observables, every correlator)
  ensemble  a batch of replicas of uneven sizes, densities and temperatures
            in one handle: System.step and the readouts of all replicas
  ionic     a binary melt with Buckingham pairs and particle-mesh Ewald
  push      a free-standing correlator fed from device arrays
  forward   the learned tail's network on device rows
  train     the learned tail's training call on host rows

Inputs come from the seed alone.  A liquid starts from a small box that
plain torch code melts here, repeated periodically and given velocities of
its own; a system can lose a few atoms to vacancies, so sizes are odd as
well.  Runs are short segments (10 to 40 steps): rounding differences then
stay rounding differences.

Results come back in the type the form computes them in: FP64 for the FP64
form, FP32 for the mixed form.  Positions are returned as displacements since
the start of the run, which do not jump where an atom crosses the box edge.
Lennard-Jones forces and virials are returned by the FP64 form only: the
truncated pair force jumps by f(rc) at the cutoff, and of the millions of
pairs of a large system some lie within FP32 rounding of it, so two correct
FP32 results differ there; velocities and energies carry every force all the
same.  The ionic melt (whose screened force at its cutoff is 1e-5 of a typical
one) returns them in both forms, but its heat flux in FP64 only: near the
lattice it is a small difference of large sums, of which FP32 energies keep
four digits; F, W, epot and v hold all that it is made of.
"""
import math

import numpy as np
import torch

import paper_2503_07526_gb300 as md

RC, DT = 2.5, 0.005                        # Lennard-Jones units (sigma, tau)
LONG = (12, 16, 2, 1)                      # stress and heat-flux correlators: blocks, lags, averaging, interval
VACF = (8, 16, 2, 1)                       # per-atom velocity correlator
KB = 8.617333262e-5                        # eV / K
FS = 1.0 / 10.1805055                      # one femtosecond in Angstrom sqrt(amu / eV)
ION = dict(rho=0.031, T=1300.0 * KB, masses=(22.99, 35.45), A=1200.0, brho=0.32, C=10.0, rc=10.0, skin=1.0, alpha=0.3)
MESHES = (16, 24, 32, 48, 64, 96, 128)
N_IN = 132                                 # features of the learned tail


def listed():
    return [
        # the state point of the plain FP64 method's configuration, in the mixed form: a single
        # small box, where a step is a chain of short kernels
        dict(name="liquid_4k_mixed", kind="liquid", cells=5, tiles=2, drop=0, rho=0.8442, T=0.722, fp64=False,
             mode="tiles", skin=0.3, vacf=True, steps=40),
        # the same box in FP64, the method as the paper has it
        dict(name="liquid_4k_fp64", kind="liquid", cells=5, tiles=2, drop=0, rho=0.8442, T=0.722, fp64=True,
             mode="verlet", skin=0.3, vacf=True, steps=20),
        # a mid-size box with an odd number of atoms, denser and hotter
        dict(name="liquid_37k_mixed", kind="liquid", cells=7, tiles=3, drop=37, rho=0.88, T=1.3, fp64=False,
             mode="tiles", skin=0.3, vacf=True, steps=20),
        # a larger FP64 comparison run
        dict(name="liquid_108k_fp64", kind="liquid", cells=5, tiles=6, drop=0, rho=0.8442, T=0.722, fp64=True,
             mode="verlet", skin=0.3, vacf=True, steps=8),
        # the benchmark: 2,048,000 atoms, every correlator on, the benchmark's skin
        dict(name="liquid_2m_mixed", kind="liquid", cells=5, tiles=16, drop=0, rho=0.8442, T=0.722, fp64=False,
             mode="tiles", skin=0.4, vacf=True, steps=20),
        # the learned tail's training ensemble: 256 replicas of 500 to 32,000 atoms in one handle
        dict(name="ensemble_256_mixed", kind="ensemble", replicas=256, fp64=False, mode="tiles", skin=0.2, steps=20),
        # the ionic melt of the particle-mesh Ewald configuration
        dict(name="ionic_512k_mixed", kind="ionic", cells=40, mesh=128, order=8, fp64=False, steps=10),
        # its parity box in FP64
        dict(name="ionic_1728_fp64", kind="ionic", cells=6, mesh=32, order=8, fp64=True, steps=10),
        # "any pair of observables can be correlated": velocities of 512,000 atoms pushed by a caller's own loop
        dict(name="push_1m5_mixed", kind="push", series=1_536_000, groups=3, cross=False, fp64=False, b=8, p=16, m=2,
             pushes=32),
        # the learned tail applied to one ensemble of runs
        dict(name="forward_4096", kind="forward", rows=4096, n_in=N_IN, depth=3),
        # and to a large sweep
        dict(name="forward_1m", kind="forward", rows=1_000_000, n_in=N_IN, depth=3),
        # its training on 3,584 runs (4,096 less the validation runs), a few epochs
        dict(name="train_3584", kind="train", rows=3584, n_in=N_IN, depth=3, batch=128, epochs=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["liquid", "liquid", "liquid", "ensemble", "ionic", "push", "forward", "train"])
    if kind == "liquid":
        fp64 = rng.random() < 0.35
        cells = rng.choice([5, 6, 7])
        most = (110_000 if fp64 else 2_048_000) // (4 * cells ** 3)
        tiles = max(2, min(_log_int(rng, 2, 16), int(most ** (1.0 / 3.0) + 1e-9)))
        n = 4 * cells ** 3 * tiles ** 3
        return dict(kind=kind, cells=cells, tiles=tiles, drop=rng.choice([0, rng.randint(1, n // 200)]),
                    rho=round(rng.uniform(0.7, 0.9), 4), T=round(rng.uniform(0.7, 2.0), 3), fp64=fp64,
                    mode="verlet" if fp64 or rng.random() < 0.25 else "tiles", skin=rng.choice([0.2, 0.3, 0.4]),
                    vacf=rng.random() < 0.6, steps=rng.choice([8, 10]) if fp64 else rng.choice([10, 16, 20]))
    if kind == "ensemble":
        return dict(kind=kind, replicas=_log_int(rng, 8, 256), fp64=False, mode=rng.choice(["tiles", "tiles", "verlet"]),
                    skin=0.2, steps=rng.choice([10, 16, 20]))
    if kind == "ionic":
        fp64 = rng.random() < 0.4
        cells = _log_int(rng, 6, 10 if fp64 else 40)
        fine = rng.choice([2.8, 3.2, 4.0]) * cells
        mesh = min(MESHES, key=lambda k: abs(k - fine))
        return dict(kind=kind, cells=cells, mesh=mesh, order=rng.choice([4, 6, 8, 8]), fp64=fp64,
                    steps=rng.choice([5, 8, 10]))
    if kind == "push":
        fp64 = rng.random() < 0.4
        groups = rng.choice([1, 3, 3, 6])
        each = _log_int(rng, 1, (1_000_000 if fp64 else 2_000_000) // groups)
        return dict(kind=kind, series=groups * each, groups=groups, cross=rng.random() < 0.3, fp64=fp64,
                    b=rng.choice([4, 8]), p=rng.choice([8, 16]), m=2, pushes=rng.choice([9, 16, 32]))
    if kind == "forward":
        return dict(kind=kind, rows=_log_int(rng, 1, 1_000_000), n_in=rng.choice([N_IN, N_IN, rng.randint(16, 240)]),
                    depth=rng.choice([2, 3, 3, 4]))
    batch = rng.choice([128, 128, 256, 512])
    return dict(kind=kind, rows=_log_int(rng, batch, 4096), n_in=rng.choice([N_IN, N_IN, rng.randint(16, 240)]),
                depth=rng.choice([2, 3, 3]), batch=batch, epochs=rng.choice([1, 2]))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _velocities(n, T, mass, g):
    v = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64) * torch.sqrt(T / mass)
    v -= (v * mass).sum(1, keepdim=True) / mass.sum()
    return v * torch.sqrt((3.0 * n - 3.0) * T / (mass * v * v).sum())


def _melted(cells, rho, T, g, steps=250):
    """Small boxes [R, 3, 4 cells^3] of a Lennard-Jones liquid at the given densities and temperatures, by plain
    all-pairs velocity Verlet from an fcc start (heated to T = 2 first)."""
    k = torch.arange(cells, device="cuda", dtype=torch.float64)
    corner = torch.stack(torch.meshgrid(k, k, k, indexing="ij")).reshape(3, -1, 1)
    basis = torch.tensor([[0.0, 0.5, 0.5, 0.0], [0.0, 0.5, 0.0, 0.5], [0.0, 0.0, 0.5, 0.5]], device="cuda",
                         dtype=torch.float64)
    frac = (corner + basis[:, None, :] + 0.25).reshape(3, -1)
    n = frac.shape[1]
    rho = torch.tensor(rho, device="cuda", dtype=torch.float64)
    T = torch.tensor(T, device="cuda", dtype=torch.float64)
    L = cells * (4.0 / rho) ** (1.0 / 3.0)
    r = frac[None] * (L / cells)[:, None, None]
    v = torch.randn(rho.numel(), 3, n, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(2.0)
    v -= v.mean(2, keepdim=True)
    own = torch.eye(n, device="cuda", dtype=torch.bool)

    def force(r):
        d = r[:, :, :, None] - r[:, :, None, :]
        d = d - L[:, None, None, None] * torch.round(d / L[:, None, None, None])
        r2 = (d * d).sum(1).masked_fill(own, 1e9)
        i2 = torch.where(r2 < RC * RC, 1.0 / r2, 0.0)
        i6 = i2 * i2 * i2
        return ((24.0 * i6 * (2.0 * i6 - 1.0) * i2)[:, None] * d).sum(3)

    f = force(r)
    for s in range(steps):
        v = v + 0.5 * DT * f
        r = r + DT * v
        f = force(r)
        v = v + 0.5 * DT * f
        if s % 10 == 9:
            now = (v * v).sum((1, 2)) / (3.0 * n - 3.0)
            v = v * torch.sqrt((torch.full_like(T, 2.0) if s < 100 else T) / now)[:, None, None]
    return r - L[:, None, None] * torch.floor(r / L[:, None, None]), L


def _repeat(base, L, tiles, drop, g):
    """The periodic box of tiles^3 copies of a small one, less `drop` atoms."""
    k = torch.arange(tiles, device="cuda", dtype=torch.float64) * L
    corner = torch.stack(torch.meshgrid(k, k, k, indexing="ij")).reshape(3, -1, 1)
    r = (corner + base[:, None, :]).reshape(3, -1)
    if drop:
        keep = torch.randperm(r.shape[1], generator=g, device="cuda")[drop:].sort().values
        r = r[:, keep]
    return r.contiguous(), float(L) * tiles


def _liquid_inputs(c, seed):
    g = _gen(seed)
    base, L = _melted(c["cells"], [c["rho"]], [c["T"]], g)
    r, box = _repeat(base[0], L[0], c["tiles"], c["drop"], g)
    one = torch.ones(r.shape[1], device="cuda", dtype=torch.float64)
    return [dict(r=r, v=_velocities(r.shape[1], c["T"], one, g), box=box)]


def _ensemble_sizes(c):
    """Copies per side and missing atoms of each replica: 500 to 32,000 atoms, log-uniform."""
    out = []
    for k in range(c["replicas"]):
        u = ((k * 37) % c["replicas"] + 0.5) / c["replicas"]
        tiles = max(1, min(4, int(round(64.0 ** (u / 3.0)))))
        out.append((tiles, (k * 13) % (2 * tiles ** 3)))
    return out


def _ensemble_inputs(c, seed):
    g = _gen(seed)
    rho = [0.70 + 0.2 * k / 7 for k in range(8)]
    T = [0.7 + 1.3 * ((3 * k) % 8) / 7 for k in range(8)]
    base, L = _melted(5, rho, T, g)
    reps = []
    for k, (tiles, drop) in enumerate(_ensemble_sizes(c)):
        r, box = _repeat(base[k % 8], float(L[k % 8]), tiles, drop, g)
        one = torch.ones(r.shape[1], device="cuda", dtype=torch.float64)
        reps.append(dict(r=r, v=_velocities(r.shape[1], T[k % 8], one, g), box=box))
    return reps


def _ionic_inputs(c, seed):
    g = _gen(seed)
    a = (8.0 / ION["rho"]) ** (1.0 / 3.0)
    k = torch.arange(c["cells"], device="cuda", dtype=torch.float64)
    corner = torch.stack(torch.meshgrid(k, k, k, indexing="ij")).reshape(3, -1, 1)
    basis = torch.tensor([[0.0, 0.5, 0.5, 0.0], [0.0, 0.5, 0.0, 0.5], [0.0, 0.0, 0.5, 0.5]], device="cuda",
                         dtype=torch.float64)
    cat = (corner + basis[:, None, :] + 0.25).reshape(3, -1)
    ani = cat + torch.tensor([[0.5], [0.0], [0.0]], device="cuda", dtype=torch.float64)
    r = torch.cat([cat, ani], 1) * a
    n, box = r.shape[1], a * c["cells"]
    r = r + 0.2 * (2.0 * torch.rand(3, n, generator=g, device="cuda", dtype=torch.float64) - 1.0)
    types = (torch.arange(n, device="cuda") >= n // 2).to(torch.int32)
    mass = torch.tensor(ION["masses"], device="cuda", dtype=torch.float64)[types.long()]
    return [dict(r=r.contiguous(), v=_velocities(n, ION["T"], mass, g), box=box, types=types)]


def _push_inputs(c, seed):
    """Correlated samples (a first-order autoregression), as velocities are."""
    g = _gen(seed)

    def series():
        x = torch.empty(c["pushes"], c["series"], device="cuda", dtype=torch.float64)
        x[0].normal_(generator=g)
        for k in range(1, c["pushes"]):
            x[k] = 0.95 * x[k - 1] + 0.3122498999199199 * torch.randn(c["series"], generator=g, device="cuda",
                                                                     dtype=torch.float64)
        return x

    x = series()
    return x, 0.5 * x + series() if c["cross"] else None


def _net_inputs(c, seed, rows):
    """Glorot-uniform weights, standardisation and rows of the learned tail's network."""
    g = _gen(seed)
    dims = (c["n_in"],) + (128,) * c["depth"] + (2,)
    flat = []
    for i, o in zip(dims[:-1], dims[1:]):
        flat.append((2.0 * torch.rand(o * i, generator=g, device="cuda") - 1.0) * math.sqrt(6.0 / (i + o)))
        flat.append(0.1 * (2.0 * torch.rand(o, generator=g, device="cuda") - 1.0))
    mean = torch.randn(c["n_in"], generator=g, device="cuda")
    std = 0.5 + torch.rand(c["n_in"], generator=g, device="cuda")
    X = torch.randn(rows, c["n_in"], generator=g, device="cuda") * std + mean
    return dims, torch.cat(flat), mean, std, X


def _train_inputs(c, seed):
    dims, flat, mean, std, X = _net_inputs(c, seed, c["rows"])
    Z = (X - mean) / std
    T = torch.stack([1.2 + 0.4 * torch.tanh(Z[:, :8].sum(1)), 2.0 + 0.5 * torch.tanh(Z[:, 4:16].sum(1))], 1)
    return dims, flat, X.cpu().numpy(), T.cpu().numpy()


# ------------------------------------------------------------- the library

def _params(c, reps):
    prec = md.MD_PREC_FP64 if c["fp64"] else md.MD_PREC_MIXED
    if c["kind"] == "ionic":
        return md.make_params(reps[0]["r"].shape[1], reps[0]["box"], rc=ION["rc"], dt=FS, skin=ION["skin"],
                              precision=prec, masses=ION["masses"], potential=md.MD_POT_BUCK_EWALD,
                              charges=(1.0, -1.0), buckingham=(ION["A"], ION["brho"], ION["C"]),
                              ewald_alpha=ION["alpha"], mesh=c["mesh"], order=c["order"], stress=LONG, heatflux=LONG,
                              vacf=None)
    one = c["kind"] == "liquid"
    return md.make_params(reps[0]["r"].shape[1] if one else 1, reps[0]["box"] if one else 1.0, rc=RC, dt=DT,
                          skin=c["skin"], precision=prec,
                          pair_mode=md.MD_PAIR_TILES if c["mode"] == "tiles" else md.MD_PAIR_VERLET, stress=LONG,
                          heatflux=LONG, vacf=VACF if one and c["vacf"] else None)


def _inputs(c, seed):
    return {"liquid": _liquid_inputs, "ensemble": _ensemble_inputs, "ionic": _ionic_inputs}[c["kind"]](c, seed)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("liquid", "ensemble", "ionic"):
        reps = _inputs(c, seed)
        p = _params(c, reps)
        if kind == "ensemble":
            s = md.System(p, replicas=reps)
        else:
            s = md.System(p, reps[0]["r"], reps[0]["v"], types=reps[0].get("types"))
        n = s.n
        r0 = torch.cat([x["r"] for x in reps], 1)
        box = torch.cat([torch.full((x["r"].shape[1],), x["box"], device="cuda", dtype=torch.float64) for x in reps])
        new = lambda *shape: torch.zeros(*shape, device="cuda", dtype=torch.float64)
        bufs = dict(r=new(3, n), v=new(3, n), epot=new(n))
        if c["fp64"] or kind == "ionic":
            bufs.update(F=new(3, n), W=new(6, n))
        return dict(case=c, sys=s, r0=r0, box=box, bufs=bufs)
    if kind == "push":
        x, y = _push_inputs(c, seed)
        h = md.Corr.create(c["b"], c["p"], c["m"], c["series"], group_size=c["series"] // c["groups"], cross=c["cross"],
                           precision=md.MD_PREC_FP64 if c["fp64"] else md.MD_PREC_MIXED, dt_unit=DT)
        return dict(case=c, corr=h, x=list(x), y=list(y) if c["cross"] else [None] * c["pushes"])
    if kind == "forward":
        dims, flat, mean, std, X = _net_inputs(c, seed, c["rows"])
        net = md.MLP(c["n_in"], 2, depth=c["depth"], batch=128, seed=1)
        net.set_flat(flat.cpu().numpy())
        net.set_scaler(mean.cpu().numpy(), std.cpu().numpy(), [1.2, 2.0], [0.3, 0.4])
        return dict(case=c, net=net, X=X)
    dims, flat, X, T = _train_inputs(c, seed)
    net = md.MLP(c["n_in"], 2, depth=c["depth"], batch=c["batch"], lr=1e-3, weight_decay=1e-3, seed=1)
    net.set_flat(flat.cpu().numpy())
    net.fit_scaler(X, T)
    return dict(case=c, net=net, X=X, T=T, seed=int(seed))


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "forward":
        return {"Y": state["net"].forward(state["X"])}
    if kind == "train":
        loss = state["net"].train(state["X"], state["T"], c["epochs"], shuffle_seed=state["seed"])
        return {"loss": loss.astype(np.float32), "params": state["net"].get_flat()}
    if kind == "push":
        h = state["corr"]
        for x, y in zip(state["x"], state["y"]):
            h.push(x, y)
        vals, count, used = h.raw()
        return {"sums": vals if c["fp64"] else vals.astype(np.float32), "count": count, "blocks": used}
    s, bufs = state["sys"], state["bufs"]
    s.step(c["steps"])
    s.particles_device(**bufs)
    moved = bufs["r"] - state["r0"]
    moved = moved - state["box"] * torch.round(moved / state["box"])
    out = dict(moved=moved, v=bufs["v"], epot=bufs["epot"])
    if "F" in bufs:
        out.update(F=bufs["F"], W=bufs["W"])
    corr = dict(stress=md.MD_CORR_STRESS, heatflux=md.MD_CORR_HEATFLUX)
    if kind == "ensemble":
        o = s.replica_observables_all()
        read = {k: s.corr(which).read_rows(0, s.nrep, 3) for k, which in corr.items()}
        out["energies"] = np.stack([o["U"], o["K"], o["T"], o["T_mean"]], 1)
    else:
        o = s.observables()
        if c.get("vacf"):
            corr["vacf"] = md.MD_CORR_VACF
        read = {k: s.corr(which).read(-1) for k, which in corr.items()}
        out["energies"] = np.array([o["U"], o["K"], o["T"], o["T_mean"]])
    out["sigma"], out["q"] = o["sigma"], o["q"]
    for k, (t, x) in read.items():
        out[k + "_t"], out[k] = t, x
    if kind == "ionic" and not c["fp64"]:
        del out["q"], out["heatflux"]
    if not c["fp64"]:
        out = {k: x.float() if isinstance(x, torch.Tensor) else x.astype(np.float32) for k, x in out.items()}
    return out


# ------------------------------------------------------------ what it takes

def _corr_bytes(c, series, pushes, size):
    """A correlator's ring traffic per pass: each level stores its sample and reads the m samples below and the older
    samples that its lags pair it with."""
    b, p, m, total = c[0], c[1], c[2], 0.0
    for k in range(b):
        per = pushes / m ** k
        lags = p - 1 if k == 0 else p - p // m
        total += per * (1 + lags / 8.0 + (m if k else 0))  # pushes can share the older samples' reads, eight at a time
    return series * size * total


def work(case):
    c, kind = case, case["kind"]
    if kind == "forward":
        dims = (c["n_in"],) + (128,) * c["depth"] + (2,)
        macs = sum(i * o for i, o in zip(dims[:-1], dims[1:]))
        return {"bytes": 4 * c["rows"] * (c["n_in"] + 2) + 4 * macs, "flops": 2 * c["rows"] * macs}
    if kind == "train":
        dims = (c["n_in"],) + (128,) * c["depth"] + (2,)
        macs = sum(i * o for i, o in zip(dims[:-1], dims[1:]))
        rows = c["rows"] // c["batch"] * c["batch"] * c["epochs"]
        return {"bytes": 4 * c["rows"] * (c["n_in"] + 2) + 24 * macs, "flops": 6 * rows * macs}
    if kind == "push":
        n, size = c["series"] * c["pushes"] * (2 if c["cross"] else 1), 8 if c["fp64"] else 4
        ring = _corr_bytes((c["b"], c["p"], c["m"]), c["series"], c["pushes"], size) * (2 if c["cross"] else 1)
        return {"bytes": 8 * n + ring, "flops": 2 * n * c["p"]}
    # an MD step reads and writes every atom's position and velocity (48 + 48 bytes; systems past the L2 stream them
    # every step), evaluates every pair inside the cutoff once (about 50 operations for a Lennard-Jones pair with its
    # energy and virial, 100 with an exponential and erfc), and feeds the correlators
    if kind == "ionic":
        n, rho, rc, per = 8 * c["cells"] ** 3, ION["rho"], ION["rc"], 100.0
        K3 = c["mesh"] ** 3
        mesh_flops = n * c["order"] ** 3 * 24.0 + 3 * 2.5 * K3 * math.log2(K3)
        mesh_bytes = (8 if c["fp64"] else 4) * K3 * 10.0
    else:
        mesh_flops = mesh_bytes = 0.0
        rc, per = RC, 50.0
        if kind == "ensemble":
            n, rho = sum(500 * t ** 3 - d for t, d in _ensemble_sizes(c)), 0.8
        else:
            n, rho = 4 * c["cells"] ** 3 * c["tiles"] ** 3 - c["drop"], c["rho"]
    pairs = n * rho * (2.0 / 3.0) * math.pi * rc ** 3
    vacf = _corr_bytes(VACF, 3 * n, c["steps"], 8 if c["fp64"] else 4) if c.get("vacf") else 0.0
    out = 8 * n * (16 if c["fp64"] else 7)
    return {"bytes": c["steps"] * (96.0 * n + mesh_bytes) + vacf + out,
            "flops": c["steps"] * (per * pairs + mesh_flops + 60.0 * n)}


# --------------------------------------------------- the same in 64 bits

def _list(r, L, rl):
    """Padded neighbour table [n, K] of one periodic box (entry i itself where a row is short)."""
    n, dev = r.shape[1], r.device
    nc = int(L // rl)
    if n <= 4500 or nc < 3:
        cand, rows = None, max(1, 40_000_000 // n)
    else:
        e = L / nc
        cc = torch.clamp((torch.remainder(r, L) / e).long(), max=nc - 1)
        cell = (cc[2] * nc + cc[1]) * nc + cc[0]
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=nc ** 3)
        start = torch.cumsum(count, 0) - count
        cap = int(count.max())
        table = torch.full((nc ** 3, cap), -1, device=dev, dtype=torch.long)
        table[cell[order], torch.arange(n, device=dev) - start[cell[order]]] = order
        o = torch.arange(27, device=dev)
        off = torch.stack([o % 3 - 1, (o // 3) % 3 - 1, o // 9 - 1])
        cand, rows = (cc, off, nc, table), max(1, 40_000_000 // (27 * cap))
    ii, jj = [], []
    for a in range(0, n, rows):
        b = min(n, a + rows)
        i = torch.arange(a, b, device=dev)
        if cand is None:
            j = torch.arange(n, device=dev)[None, :].expand(b - a, n)
        else:
            cc, off, nc, table = cand
            q = torch.remainder(cc[:, a:b, None] + off[:, None, :], nc)
            j = table[(q[2] * nc + q[1]) * nc + q[0]].reshape(b - a, -1)
        jc = j.clamp(min=0)
        d = r[:, a:b, None] - r[:, jc]
        d = d - L * torch.round(d / L)
        ok = ((d * d).sum(0) < rl * rl) & (j >= 0) & (j != i[:, None])
        x, y = ok.nonzero(as_tuple=True)
        ii.append(x + a)
        jj.append(j[x, y])
    ii, jj = torch.cat(ii), torch.cat(jj)
    num = torch.bincount(ii, minlength=n)
    first = torch.cumsum(num, 0) - num
    out = torch.arange(n, device=dev)[:, None].repeat(1, int(num.max()))
    out[ii, torch.arange(ii.numel(), device=dev) - first[ii]] = jj
    return out


def _pair_sums(r, L, nb, pot, rc, q=None):
    """Forces, energies and virials of every atom (half of each pair's energy and virial)."""
    n = r.shape[1]
    F, E, W = torch.zeros_like(r), torch.zeros_like(r[0]), torch.zeros(6, n, device=r.device, dtype=r.dtype)
    step = max(1, 20_000_000 // max(1, nb.shape[1]))
    for a in range(0, n, step):
        b = min(n, a + step)
        j = nb[a:b]
        d = r[:, a:b, None] - r[:, j]
        d = d - L[a:b, None] * torch.round(d / L[a:b, None])
        r2 = (d * d).sum(0)
        on = (r2 < rc * rc) & (j != torch.arange(a, b, device=r.device)[:, None])
        r2 = torch.where(on, r2, 1.0)
        u, fs = pot(r2, None if q is None else q[a:b, None] * q[j])
        u, fs = torch.where(on, u, 0.0), torch.where(on, fs, 0.0)
        f = fs * d
        F[:, a:b], E[a:b] = f.sum(2), 0.5 * u.sum(1)
        for k, (x, y) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            W[k, a:b] = 0.5 * (d[x] * f[y]).sum(1)
    return F, E, W


def _lj(r2, qq):
    i6 = 1.0 / r2 ** 3
    s6 = RC ** -6.0
    return 4.0 * i6 * (i6 - 1.0) - 4.0 * s6 * (s6 - 1.0), 24.0 * i6 * (2.0 * i6 - 1.0) / r2


def _buck(r2, qq):
    r = torch.sqrt(r2)
    ex, i6 = ION["A"] * torch.exp(-r / ION["brho"]), 1.0 / r2 ** 3
    k, al = md.KE_EV_ANGSTROM * qq, ION["alpha"]
    ec = torch.erfc(al * r)
    u = ex - ION["C"] * i6 + k * ec / r
    du = ex / ION["brho"] - 6.0 * ION["C"] * i6 / r + k * (ec / r2 + 2.0 * al / math.sqrt(math.pi) *
                                                            torch.exp(-(al * r) ** 2) / r)
    return u, du / r


def _splines(w, n):
    """M_n(w + t) for t = 0 .. n-1 with first and second derivatives, stacked [3, n, N]."""
    m = {2: [w, 1.0 - w]}
    for p in range(3, n + 1):
        prev = m[p - 1] + [torch.zeros_like(w)]
        m[p] = [((w + t) * prev[t] + (p - w - t) * (prev[t - 1] if t else torch.zeros_like(w))) / (p - 1)
                for t in range(p)]
    at = lambda p, t: m[p][t] if 0 <= t < p else torch.zeros_like(w)
    return torch.stack([torch.stack(m[n]), torch.stack([at(n - 1, t) - at(n - 1, t - 1) for t in range(n)]),
                        torch.stack([at(n - 2, t) - 2.0 * at(n - 2, t - 1) + at(n - 2, t - 2) for t in range(n)])])


def _mesh_sums(r, L, q, K, n):
    """Smooth particle-mesh Ewald: forces, energies and virials of every ion (self term included)."""
    dev, al, ke = r.device, ION["alpha"], md.KE_EV_ANGSTROM
    u = torch.remainder(r, L) * (K / L)
    base = torch.floor(u).long()
    sp = [_splines((u - base)[a], n) for a in range(3)]
    t = torch.arange(n, device=dev)
    idx = [torch.remainder(base[a][None] - t[:, None], K) for a in range(3)]
    N, mesh = r.shape[1], torch.zeros(K ** 3, device=dev, dtype=torch.float64)
    for tx in range(n):
        for ty in range(n):
            row = (idx[0][tx] * K + idx[1][ty]) * K
            w = (q * sp[0][0, tx] * sp[1][0, ty])[None] * sp[2][0]
            mesh.index_add_(0, (row[None] + idx[2]).reshape(-1), w.reshape(-1))
    at = _splines(torch.zeros(1, device=dev, dtype=torch.float64), n)[0, :, 0]  # M_n at 0 .. n-1
    ang = 2.0 * math.pi / K * torch.arange(K, device=dev, dtype=torch.float64)
    s = sum(torch.polar(at[k + 1], ang * k) for k in range(n - 1))
    bm = 1.0 / s.abs() ** 2
    m = torch.arange(K, device=dev, dtype=torch.float64)
    m = torch.where(m <= K // 2, m, m - K) / L
    m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2
    m2[0, 0, 0] = 1.0
    tt = math.pi ** 2 / al ** 2 * m2
    BC = bm[:, None, None] * bm[None, :, None] * bm[None, None, :] * torch.exp(-tt) / m2 / (math.pi * L ** 3)
    BC[0, 0, 0] = 0.0
    G = torch.fft.fftn(mesh.reshape(K, K, K))
    phi = (torch.fft.ifftn(G * BC).real * K ** 3).reshape(-1)
    psi = (torch.fft.ifftn(G * BC * 2.0 * (1.0 + tt) / m2).real * K ** 3).reshape(-1)
    acc = torch.zeros(10, N, device=dev, dtype=torch.float64)
    for tx in range(n):
        for ty in range(n):
            at_ = ((idx[0][tx] * K + idx[1][ty]) * K)[None] + idx[2]
            x, y, z = sp[0][:, tx], sp[1][:, ty], sp[2]
            p, s = [(phi[at_] * z[k]).sum(0) for k in range(2)], [(psi[at_] * z[k]).sum(0) for k in range(3)]
            acc += torch.stack([x[0] * y[0] * p[0], x[1] * y[0] * p[0], x[0] * y[1] * p[0], x[0] * y[0] * p[1],
                                x[2] * y[0] * s[0], x[0] * y[2] * s[0], x[0] * y[0] * s[2], x[1] * y[1] * s[0],
                                x[1] * y[0] * s[1], x[0] * y[1] * s[1]])
    E = 0.5 * ke * q * acc[0]
    W = ke * q * (K / L) ** 2 / (8.0 * math.pi ** 2) * acc[4:]
    W[:3] += E
    return -ke * q * (K / L) * acc[1:4], E - ke * al / math.sqrt(math.pi) * q * q, W


def _readout(x, spec, unit):
    """The multiple-tau readout grid of series x [samples, series]: times, and products averaged over the series."""
    b, p, m = spec[:3]
    ts, cs = [], []
    for k in range(b):
        if k:
            if x.shape[0] < m:
                break
            x = x[:x.shape[0] // m * m].reshape(x.shape[0] // m, m, -1).mean(1)
        for lag in range(p // m if k else 0, p):
            if x.shape[0] > lag:
                ts.append(lag * m ** k * unit)
                cs.append((x[:x.shape[0] - lag] * x[lag:]).mean().reshape(1))
    return torch.tensor(ts, dtype=torch.float64), torch.cat(cs).cpu()


def _exact_md(c, seed):
    reps = _inputs(c, seed)
    ionic, one = c["kind"] == "ionic", c["kind"] != "ensemble"
    rc, dt, pot, skin = (ION["rc"], FS, _buck, 0.6) if ionic else (RC, DT, _lj, 0.7)
    r0 = torch.cat([x["r"] for x in reps], 1)
    v = torch.cat([x["v"] for x in reps], 1)
    n, dev = r0.shape[1], r0.device
    sizes = [x["r"].shape[1] for x in reps]
    rep = torch.repeat_interleave(torch.arange(len(reps), device=dev), torch.tensor(sizes, device=dev))
    box = torch.tensor([x["box"] for x in reps], device=dev, dtype=torch.float64)
    L, V = box[rep], box ** 3
    mass, q = torch.ones(n, device=dev, dtype=torch.float64), None
    if ionic:
        mass = torch.tensor(ION["masses"], device=dev, dtype=torch.float64)[reps[0]["types"].long()]
        q = 1.0 - 2.0 * reps[0]["types"].double()
    add = lambda x: torch.zeros(x.shape[0], len(reps), device=dev, dtype=torch.float64).index_add_(1, rep, x)
    r, nb, r_nb = r0.clone(), None, None

    def forces():
        nonlocal nb, r_nb
        if nb is None or float(((r - r_nb) ** 2).sum(0).max()) > (0.5 * skin) ** 2:
            nb = None
            parts, at = [], 0
            for x in reps:
                k = x["r"].shape[1]
                parts.append(_list(r[:, at:at + k], x["box"], rc + skin) + at)
                at += k
            most = max(x.shape[1] for x in parts)
            nb = torch.arange(n, device=dev)[:, None].repeat(1, most)
            at = 0
            for x in parts:
                nb[at:at + x.shape[0], :x.shape[1]] = x
                at += x.shape[0]
            r_nb = r.clone()
        out = _pair_sums(r, L, nb, pot, rc, q)
        if ionic:
            out = tuple(x + y for x, y in zip(out, _mesh_sums(r, float(box[0]), q, c["mesh"], c["order"])))
        return out

    F, E, W = forces()
    stress, heat, vel, Ts = [], [], [], []
    row = ((0, 3, 4), (3, 1, 5), (4, 5, 2))
    dof = 3.0 * torch.tensor(sizes, device=dev, dtype=torch.float64) - 3.0
    for _ in range(c["steps"]):
        v = v + 0.5 * dt / mass * F
        r = r + dt * v
        F, E, W = forces()
        v = v + 0.5 * dt / mass * F
        ke = 0.5 * mass * (v * v).sum(0)
        vv = torch.stack([v[0] * v[0], v[1] * v[1], v[2] * v[2], v[0] * v[1], v[0] * v[2], v[1] * v[2]])
        sig = add(mass * vv + W) / V
        flux = add(torch.stack([(ke + E) * v[a] + sum(W[row[a][k]] * v[k] for k in range(3)) for a in range(3)])) / V
        U, K = add(E[None])[0], add(ke[None])[0]
        Ts.append(2.0 * K / dof)
        stress.append(sig[3:])
        heat.append(flux)
        if c.get("vacf"):
            vel.append(v.reshape(-1))
    out = dict(moved=r - r0, v=v, epot=E)
    if c["fp64"] or ionic:
        out.update(F=F, W=W)
    en = torch.stack([U, K, Ts[-1], torch.stack(Ts).mean(0)], 1)
    out["energies"], out["sigma"], out["q"] = (en[0], sig[:, 0], flux[:, 0]) if one else (en, sig.T, flux.T)
    for name, x in (("stress", stress), ("heatflux", heat)):
        x = torch.stack(x)  # [steps, 3, replicas]
        rows = [_readout(x[:, :, k], LONG, dt) for k in range(len(reps))]
        out[name + "_t"], out[name] = rows[0][0], rows[0][1] if one else torch.stack([y[1] for y in rows])
    if vel:
        out["vacf_t"], out["vacf"] = _readout(torch.stack(vel), VACF, dt)
    if ionic and not c["fp64"]:
        del out["q"], out["heatflux"]
    return out


def _exact_push(c, seed):
    x, y = _push_inputs(c, seed)
    y = x if y is None else y
    b, p, m, G = c["b"], c["p"], c["m"], c["groups"]
    sums = torch.zeros(G, b, p, dtype=torch.float64)
    for k in range(b):
        if k:
            if x.shape[0] < m:
                break
            x, y = (z[:z.shape[0] // m * m].reshape(z.shape[0] // m, m, -1).mean(1) for z in (x, y))
        for lag in range(p // m if k else 0, min(p, x.shape[0])):
            sums[:, k, lag] = (x[:x.shape[0] - lag] * y[lag:]).reshape(x.shape[0] - lag, G, -1).sum((0, 2)).cpu()
    return {"sums": sums, "count": None, "blocks": None}


def _b16(x):
    return x.to(torch.bfloat16).double()


def _layers(dims, flat):
    out, k = [], 0
    for i, o in zip(dims[:-1], dims[1:]):
        W = flat[k:k + i * o].reshape(o, i)
        k += i * o
        out.append([W, flat[k:k + o]])
        k += o
    return out


def _exact_forward(c, seed):
    dims, flat, mean, std, X = _net_inputs(c, seed, c["rows"])
    h = _b16((X.double() - mean.double()) / std.double())
    lay = _layers(dims, flat.double())
    for k, (W, b) in enumerate(lay):
        h = h @ _b16(W).T + b
        if k < len(lay) - 1:
            h = _b16(torch.tanh(h))
    scale = torch.tensor([[0.3, 0.4], [1.2, 2.0]], device="cuda", dtype=torch.float32).double()
    return {"Y": h * scale[0] + scale[1]}


def _shuffled(seed, rows):
    """Order of one epoch: rows sorted by their SplitMix64 keys."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, rows + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return np.argsort(z, kind="stable")


def _exact_train(c, seed):
    """Adam on the mean squared error, with bfloat16 rounding where include/gk_tail.h has it."""
    dims, flat, X, T = _train_inputs(c, seed)
    X, T = (torch.from_numpy(a).cuda().double() for a in (X, T))
    X, T = ((a - a.mean(0).float().double()) / a.std(0, correction=0).float().double() for a in (X, T))
    lay = _layers(dims, flat.double())
    m1, m2 = [[torch.zeros_like(a) for a in p] for p in lay], [[torch.zeros_like(a) for a in p] for p in lay]
    f32 = lambda a: float(np.float32(a))
    b1, b2, lr, wd, eps = f32(0.9), f32(0.999), f32(1e-3), f32(1e-3), f32(1e-8)
    t, hist = 0, []
    for e in range(c["epochs"]):
        order = torch.from_numpy(_shuffled(int(seed) + e, c["rows"])).cuda()
        losses = []
        for k in range(c["rows"] // c["batch"]):
            at = order[k * c["batch"]:(k + 1) * c["batch"]]
            h = [_b16(X[at])]
            for l, (W, b) in enumerate(lay):
                z = h[-1] @ _b16(W).T + b
                h.append(_b16(torch.tanh(z)) if l < len(lay) - 1 else z)
            d = h[-1] - T[at]
            losses.append((d * d).mean())
            dz = _b16(2.0 / d.numel() * d)
            grads = []
            for l in range(len(lay) - 1, -1, -1):
                grads.append((dz.T @ h[l], dz.sum(0)))
                if l:
                    dz = _b16((dz @ _b16(lay[l][0])) * (1.0 - h[l] * h[l]))
            t += 1
            c1, c2 = 1.0 - b1 ** t, 1.0 - b2 ** t
            for l, g in enumerate(reversed(grads)):
                for w in range(2):
                    m1[l][w] = b1 * m1[l][w] + (1.0 - b1) * g[w]
                    m2[l][w] = b2 * m2[l][w] + (1.0 - b2) * g[w] ** 2
                    step = (m1[l][w] / c1) / (torch.sqrt(m2[l][w] / c2) + eps)
                    lay[l][w] = lay[l][w] - lr * (step + wd * lay[l][w] if w == 0 else step)
        hist.append(torch.stack(losses).mean())
    return {"loss": torch.stack(hist), "params": torch.cat([a.reshape(-1) for p in lay for a in p])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "push":
        return _exact_push(case, seed)
    if kind == "forward":
        return _exact_forward(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return _exact_md(case, seed)
