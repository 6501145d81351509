"""What a program that uses this framework has it do, as measurable cases.

Almost every case is the call sequence of a molecular-dynamics program: load a
state, advance it some velocity-Verlet steps, read the energies, export a
frame.  The systems are those of the framework's own benchmark and tests (fcc
crystal, porous solid, liquid, Sutton-Chen metal, embedded-atom bcc metal,
two-species alloy, batch of replicas), from 864 atoms, where launches and
latency are the cost, to the 9.8 million atoms of the porous solid.  One case
is an iteration of the learned cost model's training.

A pass starts from the same state each time (md_set_state, as after reading a
restart file), so it holds one forced list build; the others come from the
half-skin rule while it steps.  Frames of the mixed-precision path are kept
in float32, as trajectory files are; the float64 path's in float64.
"""
from __future__ import annotations

import math

import torch

from paper_1611_00075_gb300 import inputs, md

FCC = ((0.0, 0.0, 0.0), (0.5, 0.5, 0.0), (0.5, 0.0, 0.5), (0.0, 0.5, 0.5))
BCC = ((0.0, 0.0, 0.0), (0.5, 0.5, 0.5))
VARIANT = {"full": md.MD_FORCE_FULL, "paired": md.MD_FORCE_PAIRED}
SCHED = {"grid": md.MD_SCHED_GRID, "paircount": md.MD_SCHED_PAIRCOUNT, "mlp": md.MD_SCHED_MLP}
EAM_KEYS = ("phi_r", "phi_a", "psi_r", "psi_a", "F_sqrt", "F_quad")


def _md(system, nx, ny, nz, **over):
    c = dict(system=system, nx=nx, ny=ny, nz=nz, T=0.72, precision="mixed", variant="full",
             sched="grid", stream=True, rebuild_every=0, steps=50)
    c.update(over)
    return c


def listed():
    named = [
        # a first script: a small crystal, every default, the default stream;
        # launches and latency are all it costs
        ("lj_fcc_864_default", _md("fcc", 6, 6, 6, stream=False)),
        # the plain float64 run of 4,000 atoms that every MD code starts with
        ("lj_fcc_4000_fp64", _md("fcc", 10, 10, 10, precision="fp64")),
        # a porous sample as in the README: two atoms per thread, learned partition
        ("lj_porous_150k_mlp", _md("porous", 40, 40, 40, T=0.3, variant="paired", sched="mlp")),
        # float64 production run of a medium sample under the pair-count partition
        ("lj_porous_112k_fp64", _md("porous", 36, 36, 36, T=0.3, precision="fp64",
                                    sched="paircount", steps=20)),
        # per-atom lists on a ragged orthorhombic box, rebuilt every 10 steps
        ("lj_fcc_ragged_331k_full", _md("fcc", 47, 61, 29, T=0.3, rebuild_every=10)),
        # the melted liquid of 1,048,576 atoms, whose lists last five steps
        ("lj_liquid_1m", _md("liquid", 64, 64, 64, T=1.2, variant="paired", steps=25)),
        # the largest: the porous solid of 16.4 million sites under the learned partition
        ("lj_porous_9.8m_mlp", _md("porous", 160, 160, 160, T=0.3, variant="paired",
                                   sched="mlp", steps=40)),
        # many-body metals: density pass and force pass
        ("sc_fcc_1m", _md("sc", 64, 64, 64, T=2.088, variant="paired")),
        ("eam_bcc_986k", _md("eam", 79, 79, 79, T=0.018)),
        # two species in one box
        ("alloy_1.15m", _md("alloy", 66, 66, 66, T=0.063, variant="paired")),
        # replicas of uneven size advanced together
        ("batch_64", dict(system="batch", count=64, nmin=1000, nmax=200000, variant="paired",
                          precision="mixed", sched="grid", stream=True, rebuild_every=0,
                          steps=25, T=1.0)),
        # one training iteration of the cost model at the porous solid's sample count
        ("cost_model_train_541k", dict(system="train", ns=541199)),
    ]
    return [dict(c, name=n) for n, c in named]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("fcc", "fcc", "porous", "porous", "liquid", "fp64", "sc", "eam", "alloy",
                       "batch", "train"))
    if kind == "train":
        return dict(system="train", ns=_logint(rng, 500, 541199))
    if kind == "batch":
        return dict(system="batch", count=_logint(rng, 3, 64), nmin=1000,
                    nmax=_logint(rng, 4000, 200000), variant=rng.choice(("full", "paired")),
                    precision="mixed", sched="grid", stream=rng.random() < 0.7, rebuild_every=0,
                    steps=25, T=1.0)
    top = {"fcc": 72, "porous": 120, "liquid": 64, "fp64": 36, "sc": 56, "eam": 72, "alloy": 66}[kind]
    edge = math.exp(rng.uniform(math.log(8 if kind in ("sc", "eam") else 6), math.log(top)))
    lo = {"sc": 7, "eam": 6}.get(kind, 6)

    def cells():
        return min(top, max(lo, int(round(edge * rng.uniform(0.8, 1.25)))))

    over = dict(stream=rng.random() < 0.7)
    if kind != "liquid" and rng.random() < 0.25:  # a fixed interval is for cold systems
        over["rebuild_every"] = 10
    if kind == "liquid":
        k = max(1, int(round(edge / 8)))
        nx, ny, nz = 8 * k, 8 * k, 8 * max(1, k - rng.randint(0, 1))
        return _md("liquid", nx, ny, nz, T=rng.choice((0.9, 1.2)), steps=25,
                   variant=rng.choice(("full", "paired")), **over)
    nx, ny, nz = cells(), cells(), cells()
    if kind == "porous":
        return _md("porous", nx, nx, nx, T=0.3, variant=rng.choice(("full", "paired", "paired")),
                   sched=rng.choice(("grid", "mlp", "paircount")), steps=40, **over)
    if kind == "fp64":
        return _md(rng.choice(("fcc", "fcc", "sc", "alloy")), max(nx, 7), max(ny, 7), max(nz, 7),
                   T=0.3, precision="fp64", steps=20, **over)
    if kind == "fcc":
        return _md("fcc", nx, ny, nz, T=0.3 if "rebuild_every" in over else round(rng.uniform(0.3, 0.8), 2),
                   variant=rng.choice(("full", "paired")), **over)
    T = {"sc": 2.088, "eam": 0.018, "alloy": 0.063}[kind]
    variant = "full" if kind == "eam" else rng.choice(("full", "paired", "paired"))
    return _md(kind, nx, ny, nz, T=T, variant=variant, **over)


# ---- inputs, made on the GPU from the seed -----------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, n):
    return torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)


def _thermal(g, n, u):
    """Displacements of rms u per component, without the tail that would put
    two atoms on top of each other (a repulsive pair never gets there)."""
    return u * _randn(g, n).clamp_(-2.2, 2.2)


def _lattice(nx, ny, nz, a0, basis):
    ax = [torch.arange(k, device="cuda", dtype=torch.float64) for k in (nx, ny, nz)]
    cell = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 1, 3)
    b = torch.tensor(basis, device="cuda", dtype=torch.float64)
    # a quarter cell off the faces of the box, so that no lattice plane lies on one
    return (a0 * (cell + b + 0.25 - 0.125 * (len(basis) == 4))).reshape(-1, 3)


def _velocities(g, n, T, mass=None):
    """Maxwell-Boltzmann, no net momentum, exactly T over 3n - 3 degrees of freedom."""
    m = torch.ones(n, 1, device="cuda", dtype=torch.float64) if mass is None else mass[:, None]
    v = _randn(g, n) * torch.sqrt(T / m)
    v -= (m * v).sum(0) / m.sum()
    ke = 0.5 * float((m * v * v).sum())
    return (v * math.sqrt(0.5 * (3 * n - 3) * T / ke)).contiguous()


def _wrap(x, box):
    b = torch.tensor(box, device="cuda", dtype=torch.float64)
    x = torch.remainder(x, b)
    return torch.where(x >= b, x - b, x).contiguous()


def _voids(seed, nc, a0):
    """Sites of an nc^3 fcc block that spherical voids of radius U(3, 15) (up
    to 0.45 box sides) leave: 60 % of them, the 40 % deepest inside removed."""
    L = nc * a0
    rmax = min(15.0, 0.45 * L)
    mean_v = math.pi * (rmax ** 4 - 3.0 ** 4) / (3.0 * (rmax - 3.0))
    count = max(2, int(round(-math.log(0.56) * L ** 3 / mean_v)))
    g = torch.Generator().manual_seed(int(seed))
    u = torch.rand(count, 4, generator=g, dtype=torch.float64).tolist()
    site = _lattice(nc, nc, nc, a0, FCC).float().reshape(nc, nc, nc, 4, 3)
    depth = torch.full((nc, nc, nc, 4), float(L * L), device="cuda")  # d^2 - r^2
    for ux, uy, uz, ur in u:
        r, sl = 3.0 + (rmax - 3.0) * ur, []
        for q in (ux, uy, uz):
            lo = int(math.floor((q * L - r) / a0)) - 2
            span = min(int(math.ceil(2 * r / a0)) + 4, nc)
            sl.append(torch.arange(lo, lo + span, device="cuda") % nc)
        ix, iy, iz = torch.meshgrid(*sl, indexing="ij")
        d = site[ix, iy, iz] - torch.tensor((ux * L, uy * L, uz * L), device="cuda")
        d -= L * torch.round(d / L)
        depth[ix, iy, iz] = torch.minimum(depth[ix, iy, iz], (d * d).sum(-1) - r * r)
    order = torch.argsort(depth.reshape(-1), stable=True)
    return order[int(round(0.4 * len(order))):].sort().values


def _liquid_box(g, nb, a0):
    """A disordered box at the liquid's density: fcc sites moved by 0.35 sigma,
    then a short descent along capped Lennard-Jones forces."""
    L = nb * a0
    x = _lattice(nb, nb, nb, a0, FCC)
    x = torch.remainder(x + 0.35 * _randn(g, len(x)), L)
    eye = torch.eye(len(x), device="cuda", dtype=torch.bool)
    for _ in range(60):
        d = x[None, :, :] - x[:, None, :]
        d -= L * torch.round(d / L)
        r2 = (d * d).sum(-1).clamp_(min=0.49)
        r2 = torch.where(eye | (r2 >= 6.25), 1e12, r2)
        s6 = r2.reciprocal().pow(3)
        f = -((48 * s6 * (s6 - 0.5) / r2)[:, :, None] * d).sum(1)
        x = torch.remainder(x + (0.0015 * f).clamp_(-0.05, 0.05), L)
    return x


def _batch_sizes(case, seed):
    """Replicas of the batch: (cells per side, rho, T)."""
    g = torch.Generator().manual_seed(int(seed))
    u = torch.rand(case["count"], 2, generator=g, dtype=torch.float64).tolist()
    # sizes are the batch's own (the same for every seed), evenly spread over the logarithm
    out = []
    for r, (ur, ut) in enumerate(u):
        t = (r * 0.6180339887498949) % 1.0
        nstar = case["nmin"] * (case["nmax"] / case["nmin"]) ** t
        out.append((max(6, int(round((nstar / 4.0) ** (1 / 3)))), 0.7 + 0.2 * ur, 0.5 + ut))
    return out


def _crystal(g, nx, ny, nz, a0, basis, u):
    x = _lattice(nx, ny, nz, a0, basis)
    box = [nx * a0, ny * a0, nz * a0]
    return _wrap(x + _thermal(g, len(x), u), box), box


def _lj_params(dt=0.005, mass=1.0):
    return dict(potential="lj", eps=1.0, sigma=1.0, rc=2.5, skin=0.3, dt=dt, mass=mass)


def _system(case, seed):
    """[(pos, vel, box)] (one per replica), potential parameters, species types."""
    g, kind, T = _gen(seed), case["system"], case["T"]
    if kind == "batch":
        out = []
        for nb, rho, t in _batch_sizes(case, seed):
            pos, box = _crystal(g, nb, nb, nb, (4 / rho) ** (1 / 3), FCC, 0.05 * math.sqrt(t))
            out.append((pos, _velocities(g, len(pos), t), box))
        return out, _lj_params(), None
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    types, mass = None, None
    if kind in ("fcc", "porous", "liquid"):
        a0, par = (4 / 0.8442) ** (1 / 3), _lj_params()
        if kind == "liquid":
            nb = 8
            base, kx, ky, kz = _liquid_box(g, nb, a0), nx // nb, ny // nb, nz // nb
            off = _lattice(kx, ky, kz, nb * a0, ((0.0, 0.0, 0.0),)) - 0.25 * nb * a0
            box = [nx * a0, ny * a0, nz * a0]
            pos = (base[None, :, :] + off[:, None, :]).reshape(-1, 3)
            pos = _wrap(pos + _thermal(g, len(pos), 0.04), box)
        else:
            pos, box = _crystal(g, nx, ny, nz, a0, FCC, 0.055 * math.sqrt(T))
            if kind == "porous":
                pos = pos[_voids(seed, nx, a0)].contiguous()
    elif kind == "sc":
        p = inputs.SC_DEFAULT
        pos, box = _crystal(g, nx, ny, nz, 1.0, FCC, 0.02)
        par = dict(potential="sc", eps=p["eps"], sigma=p["a"], c=p["c"], n_exp=p["n_exp"],
                   m_exp=p["m_exp"], rc=p["rc"], skin=p["skin"], dt=p["dt"], mass=p["mass"])
    elif kind == "eam":
        p = inputs.EAM_FE_LIKE
        pos, box = _crystal(g, nx, ny, nz, 1.0, BCC, 0.02)
        par = dict(potential="eam", rc=p["rc"], skin=p["skin"], dt=p["dt"], mass=p["mass"],
                   eam={k: p[k] for k in EAM_KEYS})
    else:  # alloy
        p = inputs.LJ_CUAU
        pos, box = _crystal(g, nx, ny, nz, p["a0"], FCC, 0.02)
        types = (torch.rand(len(pos), generator=g, device="cuda") < 0.25).to(torch.int32)
        mass = torch.tensor(p["mass"], device="cuda", dtype=torch.float64)[types.long()]
        t_eps, t_sigma = inputs.mixing_rules(p["eps"], p["sigma"])
        par = dict(_lj_params(dt=p["dt"]), types=types, t_eps=t_eps, t_sigma=t_sigma,
                   t_mass=p["mass"])
    return [(pos, _velocities(g, len(pos), T, mass), box)], par, types


def _train_inputs(case, seed):
    """Samples as the cost model sees them (log-scaled atom, neighbour and
    stencil counts of cells) with their log cycles, weights after a few
    iterations, and Adam's moments."""
    g, ns = _gen(seed), case["ns"]
    r = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    occ = 1 + torch.floor(24 * r(ns).sqrt())
    X = torch.stack([occ / 16, occ * (30 + 50 * r(ns)) / 1024, (100 + 450 * r(ns)) / 512], 1)
    y = (0.6 + 0.4 * torch.log1p(X[:, 1]) + 0.1 * X[:, 2]
         + 0.01 * torch.randn(ns, generator=g, device="cuda"))
    P = torch.cat([(2 * r(96) - 1) * math.sqrt(2.0), 0.1 * (r(32) - 0.5),
                   (2 * r(1024) - 1) * math.sqrt(6 / 32), 0.1 * (r(32) - 0.5),
                   (2 * r(32) - 1) * math.sqrt(6 / 32), 0.1 * (r(1) - 0.5)])
    m = 1e-3 * (r(md.MLP_NPARAMS) - 0.5)
    v = 1e-6 * r(md.MLP_NPARAMS)
    return [t.float().contiguous() for t in (X, y, P, m, v)]


# ---- the framework's calls -----------------------------------------------------

def prepare(case, seed):
    if case["system"] == "train":
        X, y, P, m, v = _train_inputs(case, seed)
        return dict(case=case, X=X, y=y, P=P, m=m, v=v, G=torch.empty_like(P),
                    loss=torch.empty(1, device="cuda"))
    reps, par, types = _system(case, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if case["stream"] else torch.cuda.current_stream()
    kw = dict(precision=case["precision"], force_variant=VARIANT[case["variant"]],
              scheduler=SCHED[case["sched"]], rebuild_every=case["rebuild_every"], stream=stream)
    with torch.cuda.stream(stream):
        if case["system"] == "batch":
            sy = md.Batch(reps, **kw, **par)
        elif types is not None:
            sp = (types, par.pop("t_eps"), par.pop("t_sigma"), par.pop("t_mass"))
            par.pop("types")
            sy = md.System(*reps[0], species=sp, **kw, **par)
        else:
            sy = md.System(*reps[0], **kw, **par)
        if case["sched"] == "mlp":
            md.md_cost_model(sy.h, md.MD_COST_SAMPLE)
            md.md_cost_model(sy.h, md.MD_COST_TRAIN)
        pos = torch.cat([r[0] for r in reps])
        vel = torch.cat([r[1] for r in reps])
    torch.cuda.synchronize()
    return dict(case=case, sy=sy, stream=stream, pos=pos, vel=vel, x=torch.empty_like(pos),
                w=torch.empty_like(vel))


def run(s):
    case = s["case"]
    if case["system"] == "train":
        # gradient and Adam step; the weights and moments of the pass are new tensors
        P, m, v = s["P"].clone(), s["m"].clone(), s["v"].clone()
        md.md_mlp_loss_grad(s["X"], s["y"], P, s["G"], s["loss"])
        md.md_mlp_adam(P, s["G"], m, v, 5, lr=3e-3)
        return {"G": s["G"], "loss": s["loss"], "P": P, "m": m, "v": v}
    h = s["sy"].h
    with torch.cuda.stream(s["stream"]):
        md.md_set_state(h, s["pos"], s["vel"])
        md.md_step(h, case["steps"])
        if case["system"] == "batch":
            ke, pe = s["sy"].energies()
            ke, pe = torch.tensor(ke), torch.tensor(pe)
        else:
            ke, pe = s["sy"].energy()
        md.md_get_state(h, s["x"], s["w"], None)
        if case["precision"] == "fp64":
            return {"pos": s["x"], "vel": s["w"], "ke": ke, "pe": pe}
        return {"pos": s["x"].float(), "vel": s["w"].float(), "ke": ke, "pe": pe}


# pairs inside the cutoff per atom, each once, and operations per pair
_PAIRS = {"fcc": 27.5, "porous": 25.0, "liquid": 27.5, "batch": 26.0, "alloy": 30.5, "sc": 82.0,
          "eam": 29.0}
_FLOPS = {"fcc": 25, "porous": 25, "liquid": 25, "batch": 25, "alloy": 25, "sc": 45, "eam": 90}


def work(case):
    if case["system"] == "train":
        ns = case["ns"]
        return {"bytes": 16.0 * ns + 36.0 * md.MLP_NPARAMS, "flops": 6.0 * 1152 * ns}
    if case["system"] == "batch":
        n = sum(4 * r[0] ** 3 for r in _batch_sizes(case, 1))
    else:
        n = (2 if case["system"] == "eam" else 4) * case["nx"] * case["ny"] * case["nz"]
        if case["system"] == "porous":
            n *= 0.6
    out = 48 if case["precision"] == "fp64" else 24
    # the loaded and the exported state, then per step positions and velocities
    # read and written (float64)
    return {"bytes": n * (48.0 + out + 96.0 * case["steps"]),
            "flops": n * (case["steps"] + 2.0) * (_PAIRS[case["system"]] * _FLOPS[case["system"]] + 12)}


# ---- the same in float64 with plain torch --------------------------------------

def _neighbours(x, box, rl):
    """Neighbour table (n x K, padded with n) of all pairs within rl."""
    n = len(x)
    nd = [int(b // rl) for b in box]
    bx = torch.tensor(box, device="cuda", dtype=torch.float64)
    ndt = torch.tensor(nd, device="cuda")
    xw = torch.remainder(x, bx)
    c = torch.minimum((xw / bx * ndt).long(), ndt - 1)
    lin = (c[:, 2] * nd[1] + c[:, 1]) * nd[0] + c[:, 0]
    ncell = nd[0] * nd[1] * nd[2]
    order = torch.argsort(lin, stable=True)
    count = torch.bincount(lin, minlength=ncell)
    cap = int(count.max())
    start = torch.cumsum(count, 0) - count
    table = torch.full((ncell, cap), n, device="cuda", dtype=torch.int32)
    ls = lin[order]
    table[ls, torch.arange(n, device="cuda") - start[ls]] = order.int()
    off = torch.tensor([(a, b, d) for a in sorted({o % nd[0] for o in (-1, 0, 1)})
                        for b in sorted({o % nd[1] for o in (-1, 0, 1)})
                        for d in sorted({o % nd[2] for o in (-1, 0, 1)})], device="cuda")
    xe = torch.cat([x, torch.zeros(1, 3, device="cuda", dtype=torch.float64)])
    rows, K = [], 0
    for b in range(0, n, 40000):
        i = torch.arange(b, min(n, b + 40000), device="cuda")
        cc = (c[i, None, :] + off[None]) % ndt
        cand = table[(cc[..., 2] * nd[1] + cc[..., 1]) * nd[0] + cc[..., 0]].reshape(len(i), -1)
        r2 = torch.zeros(cand.shape, device="cuda", dtype=torch.float64)
        for k in range(3):
            d = xe[:, k][cand] - x[i, k][:, None]
            d -= box[k] * torch.round(d / box[k])
            r2 += d * d
        ok = (r2 < rl * rl) & (cand != i[:, None]) & (cand != n)
        rank = torch.cumsum(ok, 1, dtype=torch.int32) - 1
        w = int(rank[:, -1].max()) + 1
        row = torch.full((len(i), w), n, device="cuda", dtype=torch.int32)
        at = ok.nonzero(as_tuple=True)
        row[at[0], rank[at].long()] = cand[at]
        rows.append(row)
        K = max(K, w)
    return rows, K


def _exact_md(case, x, v, box, par, types, steps):
    """Velocity-Verlet steps, then kinetic and potential energy, in float64."""
    n = len(x)
    pot, rc, dt = par["potential"], par["rc"], par["dt"]
    skin = max(0.05, min(0.6, min(box) / 3.0 - rc - 1e-9))
    bt = [float(b) for b in box]
    if types is not None:
        eps = torch.as_tensor(par["t_eps"], device="cuda", dtype=torch.float64).reshape(-1)
        sig2 = torch.as_tensor(par["t_sigma"], device="cuda", dtype=torch.float64).reshape(-1) ** 2
        ty = torch.cat([types.long(), torch.zeros(1, device="cuda", dtype=torch.long)])
        mass = torch.tensor(par["t_mass"], device="cuda", dtype=torch.float64)[types.long()][:, None]
    else:
        mass = torch.full((n, 1), float(par["mass"]), device="cuda", dtype=torch.float64)
    if pot == "eam":
        e = par["eam"]

    def cubes(r, knots, coef):
        f, df = torch.zeros_like(r), torch.zeros_like(r)
        for rk, a in zip(knots, coef):
            t = (rk - r).clamp(min=0)
            f += a * t ** 3
            df -= 3 * a * t * t
        return f, df

    def chunks(x, rows):
        xe = torch.cat([x, torch.zeros(1, 3, device="cuda", dtype=torch.float64)])
        b = 0
        for row in rows:
            i = slice(b, b + len(row))
            ds = []
            r2 = torch.zeros(row.shape, device="cuda", dtype=torch.float64)
            for k in range(3):
                d = xe[:, k][row] - x[i, k][:, None]
                d -= bt[k] * torch.round(d / bt[k])
                ds.append(d)
                r2 += d * d
            ok = (row != n) & (r2 < rc * rc)
            r2 = torch.where(ok, r2, 1.0)
            yield i, row, ds, r2, ok
            b += len(row)

    def forces(x, rows):
        f = torch.empty_like(x)
        U = 0.0
        if pot != "lj":
            rho = torch.empty(n, device="cuda", dtype=torch.float64)
            for i, row, ds, r2, ok in chunks(x, rows):
                if pot == "sc":
                    psi = (par["sigma"] ** 2 / r2) ** (par["m_exp"] / 2)
                else:
                    psi = cubes(r2.sqrt(), e["psi_r"], e["psi_a"])[0]
                rho[i] = (psi * ok).sum(1)
            if pot == "sc":
                ec = par["eps"] * par["c"]
                U += float(-ec * rho.sqrt().sum())
                dF = -0.5 * ec / rho.sqrt()
            else:
                U += float((-e["F_sqrt"] * rho.sqrt() + e["F_quad"] * rho * rho).sum())
                dF = -0.5 * e["F_sqrt"] / rho.sqrt() + 2 * e["F_quad"] * rho
            dFe = torch.cat([dF, torch.zeros(1, device="cuda", dtype=torch.float64)])
        for i, row, ds, r2, ok in chunks(x, rows):
            if pot == "lj":
                if types is None:
                    s2, ep = par["sigma"] ** 2, par["eps"]
                else:
                    t = ty[i][:, None] * len(par["t_mass"]) + ty[row]
                    s2, ep = sig2[t], eps[t]
                s6 = (s2 / r2) ** 3
                sc6 = (s2 / (rc * rc)) ** 3
                fs = 48 * ep * s6 * (s6 - 0.5) / r2
                phi = 4 * ep * (s6 * (s6 - 1) - sc6 * (sc6 - 1))
            elif pot == "sc":
                q = par["sigma"] ** 2 / r2
                phi = par["eps"] * q ** (par["n_exp"] / 2)
                psi = q ** (par["m_exp"] / 2)
                fs = (par["n_exp"] * phi + par["m_exp"] * (dF[i][:, None] + dFe[row]) * psi) / r2
            else:
                r = r2.sqrt()
                phi, dphi = cubes(r, e["phi_r"], e["phi_a"])
                dpsi = cubes(r, e["psi_r"], e["psi_a"])[1]
                fs = -(dphi + (dF[i][:, None] + dFe[row]) * dpsi) / r
            fs = fs * ok
            U += 0.5 * float((phi * ok).sum())
            for k in range(3):
                f[i, k] = -(fs * ds[k]).sum(1)
        return f, U

    x0 = x.clone()
    rows, _ = _neighbours(x, bt, rc + skin)
    f, U = forces(x, rows)
    for _ in range(steps):
        v = v + 0.5 * dt * f / mass
        x = x + dt * v
        if float(((x - x0) ** 2).sum(1).max()) > 0.25 * skin * skin * 0.99:
            rows, _ = _neighbours(x, bt, rc + skin)
            x0 = x.clone()
        f, U = forces(x, rows)
        v = v + 0.5 * dt * f / mass
    return _wrap(x, bt), v, 0.5 * float((mass * v * v).sum()), U


def _exact_train(case, seed):
    X, y, P, m, v = [t.double() for t in _train_inputs(case, seed)]
    Q = P.clone().requires_grad_(True)
    W1, b1, W2, b2 = Q[:96].view(32, 3), Q[96:128], Q[128:1152].view(32, 32), Q[1152:1184]
    a = torch.relu(X @ W1.T + b1)
    out = torch.relu(a @ W2.T + b2) @ Q[1184:1216] + Q[1216]
    loss = ((out - y) ** 2).mean()
    loss.backward()
    G = Q.grad
    m = 0.9 * m + 0.1 * G
    v = 0.999 * v + 0.001 * G * G
    P = P - 3e-3 * (m / (1 - 0.9 ** 5)) / ((v / (1 - 0.999 ** 5)).sqrt() + 1e-8)
    return {"G": G, "loss": loss.detach().reshape(1), "P": P, "m": m, "v": v}


def exact(case, seed):
    if case["system"] == "train":
        return _exact_train(case, seed)
    reps, par, types = _system(case, seed)
    got = [_exact_md(case, x, v, box, par, types, case["steps"]) for x, v, box in reps]
    pos, vel = torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    if case["system"] == "batch":
        ke = torch.tensor([g[2] for g in got], dtype=torch.float64)
        pe = torch.tensor([g[3] for g in got], dtype=torch.float64)
    else:
        ke, pe = (torch.tensor(t, dtype=torch.float64) for t in got[0][2:])
    return {"pos": pos, "vel": vel, "ke": ke, "pe": pe}
