"""Performance cases: the library's work as a user's program calls it.

A case is a dict of plain values.  `listed()` gives the named ones, `draw(rng)`
one more of the same ranges, `prepare(case, seed)` what a program holds before
the call (a context, the crystal's sites, a thermal state made from the seed),
`run(state)` one pass through the public entry points, `work(case)` the bytes
and operations the pass cannot do without, and `exact(case, seed)` the pass's
outputs in FP64 from plain torch.

Sizes and conditions are those of the repository's configurations and tests:
the bcc 4^3 reference run, the 20-replica Frenkel-Ladd campaign at 1400 K, the
256 uneven replicas, reversible scaling of bcc 16^3, and the gradient cells of
65,536 and 70,304 atoms.
"""
import math

import numpy as np
import torch

from paper_2201_04622_gb300 import ne
from paper_2201_04622_gb300 import workloads as W

KB = 8.617333262e-5  # eV / K
AMU = 1.0364269656262175e-4  # eV ps^2 / A^2
MASS = W.MASS_FE_AMU * AMU
DT, DAMP = 1e-3, 0.1
BETA_T, TAU_P = 1.2, 0.5  # barostat coupling (A^3 / eV, ps)
LATTICE = {"bcc": W.BCC, "fcc": W.FCC, "hcp": W.HCP}
EDGE = {"bcc": W.A_BCC, "fcc": W.A_FCC, "hcp": W.A_HCP}
BASIS = {"bcc": [[0, 0, 0], [0.5, 0.5, 0.5]],
         "fcc": [[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]],
         "hcp": [[0, 0, 0], [0.5, 0.5, 0], [0, 1 / 3, 0.5], [0.5, 5 / 6, 0.5]]}
PAIRS = {"bcc": 58, "fcc": 54, "hcp": 56}  # neighbours inside r_c
# two species as in an iron-aluminium B2 cell: masses and springs
SPECIES_MASS = (MASS, 26.98 * AMU)
SPECIES_K = (4.2, 3.1)
STREAM_FL, STREAM_RS, STREAM_MSD, STREAM_BARO = 0, 2, 3, 5


# ------------------------------------------------------------------- cases
def listed():
    return [
        # single point on the smallest cell: latency of one call
        dict(name="energy_bcc4_mixed", kind="energy", cells="bcc 4 4 4", T=300.0, prec="mixed"),
        # single point on the largest cell, FP64 (a reference energy with rho)
        dict(name="energy_fcc26_fp64", kind="energy", cells="fcc 26 26 26", T=300.0, prec="fp64"),
        # one step of a potential fit: U and its gradients by positions and knots
        dict(name="autograd_bcc32_mixed", kind="autograd", cells="bcc 32 32 32", T=300.0, prec="mixed"),
        # the spring-constant fit that precedes every campaign
        dict(name="fit_bcc10_mixed", kind="fit", cells="bcc 10 10 10", T=1400.0, prec="mixed", n_eq=50,
             n_samples=15, stride=10, skin=1.0),
        # a whole forward/backward switch of the small reference cell
        dict(name="switch_bcc4_fp64", kind="switch", cells="bcc 4 4 4", T=100.0, prec="fp64", t_eq=100, t_s=200,
             skin=0.3),
        # the Frenkel-Ladd campaign: ten bcc and ten fcc seeds in one batch
        dict(name="fl20_runner", kind="runner", cells="10*bcc 10 10 10, 10*fcc 8 8 8", T=1400.0, path="fl",
             begin=30000, steps=100),
        # the uneven 256-replica batch, 300-1600 K
        dict(name="fl256_runner", kind="runner", uneven=256, set_seed=1, path="fl", begin=30000, steps=20),
        # reversible scaling of four seeds of bcc 16^3 with cumulative works
        dict(name="rs16x4_runner", kind="runner", cells="4*bcc 16 16 16", T=100.0, path="rs", begin=30000, steps=100),
        # the largest single cell
        dict(name="fl32_runner", kind="runner", cells="bcc 32 32 32", T=300.0, path="fl", begin=30000, steps=50),
        # reversible scaling at zero pressure (barostat)
        dict(name="rs12x4_npt_runner", kind="runner", cells="4*bcc 12 12 12", T=100.0, path="rs", begin=20000,
             steps=100, npt=1),
        # the same campaign in FP64: the precision reference
        dict(name="fl20_fp64", kind="general", cells="10*bcc 10 10 10, 10*fcc 8 8 8", T=1400.0, prec="fp64",
             path="fl", begin=30000, steps=160, skin=2.6),
        # parameter gradient along a run of the 65,536-atom cell
        dict(name="grad32_mixed", kind="general", cells="bcc 32 32 32", T=300.0, prec="mixed", path="fl",
             begin=30000, steps=160, skin=1.0, grad=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_cells(rng, lo, hi, lmin, lattices=("bcc", "fcc", "hcp")):
    """A cell of about lo..hi atoms (spread over the logarithm) with edges
    above lmin and unequal cell counts."""
    lat = rng.choice(lattices)
    nb, edge = len(BASIS[lat]), _cell(lat)
    for _ in range(100):
        m = (_log_int(rng, lo, hi) / nb) ** (1 / 3) * (edge[0] * edge[1] * edge[2]) ** (1 / 3)
        n = [max(3, math.ceil(lmin / edge[d] + 1e-6), int(round(m / edge[d] * rng.uniform(0.85, 1.18)))) for d in
             range(3)]
        if nb * n[0] * n[1] * n[2] <= hi:
            break
        lo = max(64, lo // 2)
    return "%s %d %d %d" % (lat, *n)


def draw(rng):
    kind = rng.choice(["energy", "autograd", "fit", "switch", "runner", "runner", "runner", "general", "general"])
    T = round(rng.uniform(100.0, 1500.0), 1)
    if kind == "energy":
        return dict(kind=kind, cells=_draw_cells(rng, 128, 70000, 10.9), T=T, prec=rng.choice(["mixed", "fp64"]))
    if kind == "autograd":
        return dict(kind=kind, cells=_draw_cells(rng, 128, 65536, 10.9, ("bcc", "fcc")), T=min(T, 600.0),
                    prec=rng.choice(["mixed", "mixed", "fp64"]))
    if kind == "fit":
        c = _draw_cells(rng, 250, 4000, 13.0)
        return dict(kind=kind, cells="%d*%s" % (rng.choice([1, 1, 2, 5]), c), T=T,
                    prec=rng.choice(["mixed", "mixed", "fp64"]), n_eq=rng.randint(20, 60),
                    n_samples=rng.randint(5, 15), stride=rng.choice([5, 10]), skin=1.0)
    if kind == "switch":
        return dict(kind=kind, cells=_draw_cells(rng, 128, 1500, 11.4), T=min(T, 800.0),
                    prec=rng.choice(["mixed", "fp64"]), t_eq=rng.randint(40, 110), t_s=rng.randint(80, 210),
                    skin=0.3)
    if kind == "runner":
        how = rng.choice(["fl", "fl", "rs", "npt", "uneven", "brick", "brick"])
        if how == "uneven":
            return dict(kind=kind, uneven=_log_int(rng, 6, 220), set_seed=rng.randint(2, 999), path="fl",
                        begin=rng.randint(15000, 45000), steps=rng.randint(10, 20))
        path = "fl" if how in ("fl", "brick") else "rs"
        if how == "brick":
            c, n_rep = _draw_cells(rng, 4200, 60000, 14.0), 1
        else:
            c = _draw_cells(rng, 400, 4000, 14.0)
            n_rep = _log_int(rng, 1, 24)
        d = dict(kind=kind, cells="%d*%s" % (n_rep, c), T=T if path == "fl" else round(rng.uniform(60.0, 150.0), 1),
                 path=path, begin=rng.randint(15000, 30000), steps=rng.randint(20, 100))
        if how == "npt":
            d["npt"] = 2 if c.startswith("hcp") else rng.choice([1, 2])
        return d
    prec = rng.choice(["mixed", "mixed", "fp64"])
    how = rng.choice(["fl", "rs", "npt", "species", "grad"])
    n_rep = 1 if how == "grad" else _log_int(rng, 1, 12)
    hi = 16000 if how == "grad" else (2000 if prec == "fp64" else 4000)
    c = _draw_cells(rng, 400, hi, 16.0, ("bcc", "fcc") if how in ("grad", "species") else ("bcc", "fcc", "hcp"))
    rs = how in ("rs", "npt")
    d = dict(kind="general", cells="%d*%s" % (n_rep, c), T=round(rng.uniform(60.0, 150.0), 1) if rs else T, prec=prec,
             path="rs" if rs else "fl", begin=rng.randint(15000, 30000), steps=rng.randint(130, 200),
             skin=rng.choice([1.0, 2.4]))
    if how == "npt":
        d["npt"] = 2 if c.startswith("hcp") else rng.choice([1, 2])
    if how == "species":
        d["species"], d["T"] = True, min(T, 900.0)
    if how == "grad":
        d["grad"], d["T"] = True, min(T, 600.0)
    return d


def _cell(lat):
    a = EDGE[lat]
    return [a, math.sqrt(3.0) * a, math.sqrt(8.0 / 3.0) * a] if lat == "hcp" else [a, a, a]


def _replicas(case):
    """One dict per replica of the batch: lattice, cells, temperature, spring."""
    if case.get("uneven"):
        spec = [("bcc" if r["lattice"] == W.BCC else "fcc", [r["n"]] * 3, r["T"])
                for r in W.batched_replicas(case["uneven"], seed=case["set_seed"])]
    else:
        spec = []
        for part in case["cells"].split(","):
            count, _, cell = part.strip().rpartition("*")
            lat, *n = cell.split()
            spec += [(lat, [int(q) for q in n], case["T"])] * int(count or 1)
    out = []
    for r, (lat, n, T) in enumerate(spec):
        # springs of eq. msd for this potential: 4.2 eV/A^2 at 100 K, 2.4 at 1400 K (bcc)
        k = 4.3 - 1.37e-3 * T + (0.0 if lat == "bcc" else 0.3)
        out.append(dict(lat=lat, n=n, T=T, k=k, id=r, atoms=len(BASIS[lat]) * n[0] * n[1] * n[2]))
    return out


def _schedule(case):
    """(t_eq, t_s, first step, steps, lambda_f) of the case's run."""
    if case["kind"] == "switch":
        return case["t_eq"], case["t_s"], 0, 2 * (case["t_eq"] + case["t_s"]), 0.0625
    if case.get("path") == "rs":
        return 10000, 100000, case["begin"], case["steps"], 0.25 if case.get("npt") else 0.0625
    return 10000, 50000, case.get("begin", 0), case.get("steps", 0), 0.0625


def _lambda(case, s):
    """Lambda in force at the start of step s of the four-phase schedule."""
    t_eq, t_s, _, _, lf = _schedule(case)
    fl = case.get("path", "fl") == "fl"

    def f(t):
        return t ** 5 * (126 + t * (-420 + t * (540 + t * (-315 + t * 70)))) if fl else 1 / (1 + t * (1 / lf - 1))
    if s <= t_eq:
        return f(0.0)
    if s <= t_eq + t_s:
        return f((s - t_eq) / t_s)
    if s <= 2 * t_eq + t_s:
        return f(1.0)
    t = (s - 2 * t_eq - t_s) / t_s
    return (1 - f(t)) if fl else f(1 - t)


# -------------------------------------------------------------- thermal state
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _sites(rep, dev):
    """Sites [cells, basis, 3] of one replica, in the library's atom order."""
    n, edge = rep["n"], _cell(rep["lat"])
    g = torch.meshgrid(*[torch.arange(m, dtype=torch.float64, device=dev) for m in n], indexing="ij")
    c = torch.stack(g, -1).reshape(-1, 1, 3) + torch.tensor(BASIS[rep["lat"]], dtype=torch.float64, device=dev)
    return c * torch.tensor(edge, dtype=torch.float64, device=dev)


def _thermal(case, seed):
    """Displacements and velocities of the batch, [atoms, 3] each: the mean
    square displacement of eq. msd at the replica's temperature (T / lambda
    on the reversible-scaling path), three quarters of it in waves with the
    1 / omega^2 weight of a crystal's phonons, so that neighbours move
    together as in a real state, and Maxwell-Boltzmann velocities."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    us, vs = [], []
    for rep in _replicas(case):
        n, nb = rep["n"], len(BASIS[rep["lat"]])
        T_eff = rep["T"] / (_lambda(case, _schedule(case)[2]) if case.get("path") == "rs" else 1.0)
        k = max(1.8, rep["k"] if case.get("path") != "rs" else 4.3 - 1.37e-3 * T_eff)
        sd = math.sqrt(KB * T_eff / k)
        q = torch.meshgrid(*[2 * math.pi * torch.fft.fftfreq(m, dtype=torch.float64, device=dev) for m in n],
                           indexing="ij")
        amp = (sum(2 - 2 * torch.cos(p) for p in q) + 0.3).rsqrt()
        noise = torch.randn(3, *n, generator=gen, dtype=torch.float64, device=dev)
        white = torch.randn(nb, *n, 3, generator=gen, dtype=torch.float64, device=dev)
        wave = torch.fft.fftn(noise, dim=(1, 2, 3)) * amp
        u = torch.stack([torch.fft.ifftn(wave * torch.exp(1j * sum(t * p for t, p in zip(b, q))), dim=(1, 2, 3)).real
                         .permute(1, 2, 3, 0) for b in BASIS[rep["lat"]]])
        u = math.sqrt(0.75) * u / u.std() + 0.5 * white
        u = u.permute(1, 2, 3, 0, 4).reshape(-1, 3)
        v = torch.randn(len(u), 3, generator=gen, dtype=torch.float64, device=dev) * math.sqrt(KB * rep["T"] / MASS)
        us.append(sd * (u - u.mean(0)))
        vs.append(v - v.mean(0))
    return torch.cat(us), torch.cat(vs)


def _knots(case, seed):
    """Knot parameters at one point of a potential fit, [3 * n_knots * 2]: phi,
    f and F each scaled by a few per cent."""
    th = torch.from_numpy(_theta()).to(_device()).reshape(3, -1)
    g = np.random.Generator(np.random.PCG64(seed + 7)).normal(1.0, 0.02, size=(3, 1))
    return (th * torch.from_numpy(g).to(th.device)).reshape(-1)


def _species(n, dev):
    return torch.arange(n, device=dev).remainder(2)


# ---------------------------------------------------------------- the passes
class State:
    """What a program holds before the call; the context goes with it."""

    ctx = None

    def __del__(self):
        if self.ctx is not None:
            ne.ne_ctx_destroy(self.ctx)


def prepare(case, seed):
    s = State()
    s.case, reps = case, _replicas(case)
    s.prec = ne.NE_FP64 if case.get("prec") == "fp64" else ne.NE_MIXED
    dev = _device()
    s.x0 = torch.cat([_sites(r, dev).reshape(-1, 3) for r in reps])
    u, s.v = _thermal(case, seed)
    s.x = s.x0 + u
    s.offs = [0]
    for r in reps:
        s.offs.append(s.offs[-1] + r["atoms"])
    s.boxes = [[m * c for m, c in zip(r["n"], _cell(r["lat"]))] for r in reps]
    t_eq, t_s, s.begin, s.steps, lf = _schedule(case)
    path = ne.NE_PATH_RS if case.get("path") == "rs" else ne.NE_PATH_FL
    s.sp = _species(max(r["atoms"] for r in reps), dev).to(torch.uint8) if case.get("species") else None
    s.mds = [ne.md_params(dt=DT, T=r["T"], damp=DAMP, mass=MASS, k_spring=r["k"], skin=case.get("skin", 1.0),
                          path=path, t_eq=t_eq, t_s=t_s, lambda_f=lf, seed=seed + 1, replica=r["id"], prec=s.prec,
                          npt=case.get("npt", 0), beta_T=BETA_T if case.get("npt") else 0.0,
                          tau_p=TAU_P if case.get("npt") else 0.0,
                          **(dict(species=s.sp, mass_s=SPECIES_MASS, k_s=SPECIES_K) if case.get("species") else {}))
             for r in reps]
    s.ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(s.x), len(reps))
    if case["kind"] == "autograd":
        s.energy = ne.eam_energy_function()
        s.theta = _knots(case, seed).requires_grad_()
        s.x.requires_grad_()
    if case["kind"] == "runner":
        s.batch = [(LATTICE[r["lat"]], EDGE[r["lat"]], *r["n"]) for r in reps]
    if case.get("grad"):
        s.w = torch.full((s.steps + 1,), 1.0 / (s.steps + 1), dtype=torch.float64, device=dev)
    return s


def _out(s, **kw):
    """The outputs in the type of the arithmetic behind them: mixed runs pair,
    kick and draw in FP32, so they are handed on in FP32."""
    if s.prec == ne.NE_FP64:
        return kw
    return {k: v.detach().float() if isinstance(v, torch.Tensor) else v for k, v in kw.items()}


def run(s):
    kind, case = s.case["kind"], s.case
    new = lambda *n: torch.empty(n, dtype=torch.float64, device=s.x.device)  # noqa: E731
    if kind == "energy":
        f, e, rho = torch.empty_like(s.x), new(1), new(len(s.x))
        ne.ne_eam_energy_forces(s.ctx, s.prec, s.x, s.boxes[0], f=f, e=e, rho=rho)
        return _out(s, f=f, e=e, rho=rho)
    if kind == "autograd":
        U = s.energy.apply(s.x, s.theta, s.ctx, s.boxes[0], s.prec)
        gx, gth = torch.autograd.grad(U, (s.x, s.theta))
        return _out(s, U=U.detach(), gx=gx, gtheta=gth)
    # a run starts from the stored state and leaves it in place
    x, v = s.x.clone(), s.v.clone()
    if kind == "fit":
        n = (case["n_eq"], case["n_samples"], case["stride"])
        if len(s.mds) == 1:
            msd, k = ne.ne_msd_fit(s.ctx, s.mds[0], x, v, s.x0, s.boxes[0], *n)
        else:
            msd, k = ne.ne_msd_fit_batched(s.ctx, s.mds, s.offs, x, v, s.x0, s.boxes, *n)
        k = torch.from_numpy(np.atleast_1d(np.asarray(k, dtype=np.float64)))
        return _out(s, x=x, v=v, msd=torch.from_numpy(np.atleast_1d(np.asarray(msd, dtype=np.float64))), k=k)
    if kind == "switch":
        wf, wb = new(s.mds[0].t_s + 1), new(s.mds[0].t_s + 1)
        W2 = new(2)
        ne.ne_switch_run(s.ctx, s.mds[0], x, v, s.x0, s.boxes[0], W2[:1], W2[1:], Wcum_fwd=wf, Wcum_bwd=wb)
        return _out(s, x=x, v=v, W=W2, Wcum_f=wf, Wcum_b=wb)
    Wd = torch.zeros((len(s.mds), 2), dtype=torch.float64, device=x.device)
    if kind == "runner":
        if case["path"] == "rs":
            t_s = s.mds[0].t_s
            wc = new(len(s.mds), 2, t_s + 1)
            ne.ne_crystal_run_segment_cum(s.ctx, s.mds, s.batch, x, v, Wd, wc, s.begin, s.steps)
            k0 = s.begin - s.mds[0].t_eq
            out = dict(x=x, v=v, W=Wd, Wcum=wc[:, 0, k0 + 1:k0 + 1 + s.steps])  # the entries this segment writes
        else:
            ne.ne_crystal_run_segment(s.ctx, s.mds, s.batch, x, v, Wd, s.begin, s.steps)
            out = dict(x=x, v=v, W=Wd)
    elif case.get("grad"):
        g = torch.zeros(6 * W.EAM_FE_LIKE["n_knots"], dtype=torch.float64, device=x.device)
        ne.ne_switch_run_segment_grad(s.ctx, s.mds, s.offs, x, v, s.x0, s.boxes, Wd, s.begin, s.steps, s.w, g)
        out = dict(x=x, v=v, W=Wd, gtheta=g)
    else:
        ne.ne_switch_run_segment(s.ctx, s.mds, s.offs, x, v, s.x0, s.boxes, Wd, s.begin, s.steps)
        out = dict(x=x, v=v, W=Wd)
    if case.get("npt"):  # the boxes the next segment starts from
        out["boxes"] = torch.from_numpy(ne.ne_ctx_boxes(s.ctx, len(s.mds)))
    return _out(s, **out)


def work(case):
    """State in and out once; per force evaluation every pair inside r_c once
    (distance, two cubics with their slopes, two force updates: about 60
    operations) and about 80 an atom (embedding, Langevin step, normals)."""
    reps = _replicas(case)
    n = sum(r["atoms"] for r in reps)
    per_eval = sum(r["atoms"] * (0.5 * PAIRS[r["lat"]] * 60 + 80) for r in reps)
    theta = 8 * 6 * W.EAM_FE_LIKE["n_knots"]
    if case["kind"] == "energy":
        return {"bytes": 8 * 7 * n, "flops": per_eval}
    if case["kind"] == "autograd":
        return {"bytes": 8 * 6 * n + 2 * theta, "flops": per_eval + sum(r["atoms"] * 0.5 * PAIRS[r["lat"]] * 30
                                                                       for r in reps)}
    if case["kind"] == "fit":
        return {"bytes": 8 * 15 * n, "flops": (case["n_eq"] + case["n_samples"] * case["stride"]) * per_eval}
    steps = _schedule(case)[3]
    extra = theta if case.get("grad") else 0
    grad = sum(r["atoms"] * 0.5 * PAIRS[r["lat"]] * 30 for r in reps) if case.get("grad") else 0
    return {"bytes": 8 * 12 * n + extra, "flops": steps * (per_eval + grad)}


# ------------------------------------------------------------ exact, in FP64
def _theta():
    """Knot values and slopes of the analytic potential, [3 * n_knots * 2]."""
    p = W.EAM_FE_LIKE
    nk = p["n_knots"]
    r = np.arange(nk) * (p["r_c"] / (nk - 1))
    w = p["r_c"] - p["r_s"]
    x = np.clip((r - p["r_s"]) / w, 0.0, 1.0)
    s = (1 - x) ** 3 * (1 + x * (3 + 6 * x))
    ds = -30 * x ** 2 * (1 - x) ** 2 / w
    th = np.zeros((3, nk, 2))
    for fn, (a, c) in enumerate(((p["A"], p["alpha"]), (1.0, p["beta"]))):
        e = a * np.exp(-c * (r / p["r_e"] - 1))
        th[fn, :, 0], th[fn, :, 1] = e * s, e * (ds - c / p["r_e"] * s)
    rho = np.arange(1, nk) * (p["rho_max"] / (nk - 1))
    th[2, 1:, 0], th[2, 1:, 1] = -p["B"] * np.sqrt(rho), -0.5 * p["B"] / np.sqrt(rho)
    th[2, 0, 1] = th[2, 1, 0] / rho[0]
    return th.reshape(-1)


def _basis(x, h, nk):
    """Interval, the four Hermite weights on it and their derivatives."""
    t = x / h
    k = t.long().clamp(0, nk - 2)
    u = t - k
    u2, u3 = u * u, u * u * u
    w = torch.stack([2 * u3 - 3 * u2 + 1, h * (u3 - 2 * u2 + u), 3 * u2 - 2 * u3, h * (u3 - u2)], -1)
    dw = torch.stack([6 * (u2 - u) / h, 3 * u2 - 4 * u + 1, 6 * (u - u2) / h, 3 * u2 - 2 * u], -1)
    return k, w, dw


def _knots4(th, k):
    return torch.cat([th[k], th[k + 1]], -1)


class _Crystal:
    """FP64 EAM of a stack of replicas of one crystal, from their
    displacements u [R, atoms, 3] off sites scaled by mu [R, 3]."""

    def __init__(self, rep, theta, dev):
        self.rep, self.theta, self.dev = rep, theta.reshape(3, -1, 2), dev
        self.nk = self.theta.shape[1]
        self.hr, self.hF = W.EAM_FE_LIKE["r_c"] / (self.nk - 1), W.EAM_FE_LIKE["rho_max"] / (self.nk - 1)
        self.reach = 0.0

    def _neighbours(self, reach):
        n, edge, basis = self.rep["n"], np.array(_cell(self.rep["lat"])), np.array(BASIS[self.rep["lat"]])
        nb, m = len(basis), [int(math.ceil(reach / e)) + 1 for e in edge]
        d = np.stack(np.meshgrid(*[np.arange(-q, q + 1) for q in m], indexing="ij"), -1).reshape(-1, 1, 3)
        cell = torch.stack(torch.meshgrid(*[torch.arange(q, device=self.dev) for q in n], indexing="ij"),
                           -1).reshape(-1, 1, 3)
        nt = torch.tensor(n, device=self.dev)
        idx, vec = [], []
        for b in range(nb):
            R = (d + basis[None] - basis[b]) * edge
            r2 = (R ** 2).sum(-1)
            at, b2 = np.nonzero((r2 < reach ** 2) & (r2 > 1e-12))
            vec.append(torch.from_numpy(R[at, b2]).to(self.dev))
            c = torch.remainder(cell + torch.from_numpy(d[at, 0])[None].to(self.dev), nt)
            idx.append(((c[..., 0] * n[1] + c[..., 1]) * n[2] + c[..., 2]) * nb + torch.from_numpy(b2).to(self.dev))
        self.idx = torch.stack(idx, 1).reshape(self.rep["atoms"], -1)  # [atoms, K]
        self.vec = torch.stack(vec).repeat(self.rep["atoms"] // nb, 1, 1)  # [atoms, K, 3]
        self.reach = reach

    def pairs(self, u, mu):
        rc = W.EAM_FE_LIKE["r_c"]
        need = (rc + 2 * float(u.norm(dim=-1).max())) / float(mu.min())
        if need > self.reach:
            self._neighbours(need + 0.6)
        R, n = u.shape[:2]
        part = []
        for r in range(R):  # one replica at a time bounds the memory
            d = self.vec * mu[r] + u[r][self.idx] - u[r][:, None]
            r2 = (d * d).sum(-1)
            i, k = torch.nonzero(r2 < rc * rc, as_tuple=True)
            part.append((i + r * n, self.idx[i, k] + r * n, d[i, k], r2[i, k].sqrt()))
        return [torch.cat(p) for p in zip(*part)]

    def eval(self, u, mu, grad=False):
        """U [R], forces, rho, diagonal virial [R, 3] and, with grad, the
        gradient of U by the knots (summed over the replicas)."""
        R, n = u.shape[:2]
        i, j, d, r = self.pairs(u, mu)
        k, w, dw = _basis(r, self.hr, self.nk)
        phi4, f4 = _knots4(self.theta[0], k), _knots4(self.theta[1], k)
        rho = torch.zeros(R * n, dtype=u.dtype, device=u.device).index_add_(0, i, (w * f4).sum(-1))
        kF, wF, dwF = _basis(rho, self.hF, self.nk)
        F4 = _knots4(self.theta[2], kF)
        dF = (dwF * F4).sum(-1)
        rep = torch.div(i, n, rounding_mode="floor")
        U = torch.zeros(R, dtype=u.dtype, device=u.device).index_add_(0, rep, 0.5 * (w * phi4).sum(-1))
        U = U + (wF * F4).sum(-1).reshape(R, n).sum(1)
        s = ((dw * phi4).sum(-1) + (dF[i] + dF[j]) * (dw * f4).sum(-1)) / r
        f = torch.zeros(R * n, 3, dtype=u.dtype, device=u.device).index_add_(0, i, s[:, None] * d)
        vir = torch.zeros(R, 3, dtype=u.dtype, device=u.device).index_add_(0, rep, -0.5 * s[:, None] * d * d)
        if not grad:
            return U, f.reshape(R, n, 3), rho.reshape(R, n), vir, None
        g = torch.zeros(3, self.nk * 2, dtype=u.dtype, device=u.device)
        for fn, kk, ww in ((0, k, 0.5 * w), (1, k, dF[i][:, None] * w), (2, kF, wF)):
            for c in range(4):
                g[fn].index_add_(0, 2 * kk + c, ww[:, c])
        return U, f.reshape(R, n, 3), rho.reshape(R, n), vir, g.reshape(-1)


def _philox(c, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF
    k0, k1 = key & M, (key >> 32) & M
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _normals(seed, ids, stream, step, n, mixed, dev):
    """Three normals per atom, [R, n, 3]; the mixed runs draw from 24 bits."""
    atom = torch.arange(n, device=dev).expand(len(ids), n)
    rep = (torch.tensor(ids, device=dev)[:, None] * 16 + stream).expand(len(ids), n)
    c = _philox([atom, torch.full_like(atom, step & 0xFFFFFFFF), torch.full_like(atom, step >> 32), rep], seed)
    w = [((q >> 8).double() + 0.5) * 2.0 ** -24 if mixed else (q.double() + 0.5) * 2.0 ** -32 for q in c]
    r0, r1 = torch.sqrt(-2 * torch.log(w[0])), torch.sqrt(-2 * torch.log(w[2]))
    a0, a1 = 2 * math.pi * w[1], 2 * math.pi * w[3]
    return torch.stack([r0 * torch.cos(a0), r0 * torch.sin(a0), r1 * torch.cos(a1)], -1)


def _exact_run(case, seed, group, u, v, theta, dev):
    """The Langevin run of a stack of replicas of one crystal, step by step."""
    reps, n = [r for r, _ in group], group[0][0]["atoms"]
    ids = [r["id"] for r in reps]
    C = _Crystal(reps[0], theta, dev)
    col = lambda q: torch.tensor(q, dtype=torch.float64, device=dev).reshape(-1, 1, 1)  # noqa: E731
    kT, k, m = col([KB * r["T"] for r in reps]), col([r["k"] for r in reps]), col([MASS] * len(reps))
    if case.get("species"):
        sp = _species(n, dev)
        k = torch.tensor(SPECIES_K, dtype=torch.float64, device=dev)[sp].reshape(1, n, 1)
        m = torch.tensor(SPECIES_MASS, dtype=torch.float64, device=dev)[sp].reshape(1, n, 1)
    m = m.expand(len(reps), n, 1)
    M = m.sum(1, keepdim=True)
    centred = lambda q, wt: q - wt * q.sum(1, keepdim=True) / M  # noqa: E731  (weight m_i / M of the sum)
    fl, mixed = case.get("path", "fl") == "fl", case.get("prec") != "fp64"
    t_eq, t_s, s0, steps, _ = _schedule(case)
    fit = case["kind"] == "fit"
    if fit:
        s0, steps = 0, case["n_eq"] + case["n_samples"] * case["stride"]
    stream = STREAM_MSD if fit else (STREAM_FL if fl else STREAM_RS)
    lam = (lambda s: 0.0) if fit else (lambda s: _lambda(case, s))  # noqa: E731
    c1 = math.exp(-DT / DAMP)
    c2 = torch.sqrt((1 - c1 * c1) * kT / m)
    mu = torch.ones(len(reps), 3, dtype=torch.float64, device=dev)
    box = torch.tensor([[q * e for q, e in zip(reps[0]["n"], _cell(reps[0]["lat"]))]] * len(reps),
                       dtype=torch.float64, device=dev)
    Wsum = torch.zeros(len(reps), 2, dtype=torch.float64, device=dev)
    cum = [[], []]
    gth = torch.zeros_like(theta) if case.get("grad") else None
    msd = torch.zeros(len(reps), dtype=torch.float64, device=dev)

    def kick(v, F, u, lm):
        FE = centred(-k * u, m)
        return v + 0.5 * DT / m * ((1 - lm) * centred(F, m) + lm * FE if fl else lm * centred(F, m))

    for q in range(steps + 1):
        s = s0 + q
        U, F, _, vir, g = C.eval(u, mu, grad=gth is not None)
        if gth is not None:
            gth += g / (steps + 1)
        if q > 0:
            v = kick(v, F, u, lam(s))
        if q == steps:
            break
        ln = lam(s + 1)
        UE = 0.5 * (k * u * u).sum((1, 2))
        slot = 0 if t_eq <= s < t_eq + t_s else 1 if 2 * t_eq + t_s <= s < 2 * t_eq + 2 * t_s else None
        if slot is not None and not fit:
            Wsum[:, slot] += (ln - lam(s)) * (U - UE if fl else U)
            cum[slot].append(Wsum[:, slot].clone())
        v = kick(v, F, u, ln)
        u = u + 0.5 * DT * v
        dv = c2 * _normals(seed + 1, ids, stream, s, n, mixed, dev)
        v = c1 * v + dv - (m * dv).sum(1, keepdim=True) / M
        u = u + 0.5 * DT * v
        if case.get("npt"):
            V, kTr, mob = (mu * box).prod(1), kT[:, 0, 0], BETA_T / TAU_P
            z = _normals(seed + 1, ids, STREAM_BARO, s, 1, False, dev)[:, 0]
            amp = torch.sqrt(2 * kTr * mob * DT / V)[:, None]
            dof = 3 * n - 3
            if case["npt"] == 2:
                e = mob * DT * (dof / 3 * kTr[:, None] + ln * vir) / V[:, None] + amp * z
            else:
                e = ((mob * DT * (dof * kTr + ln * vir.sum(1)) / (3 * V))[:, None] + amp * z[:, :1]) / 3
                e = e.expand(-1, 3)
            mu, u = mu * e.exp(), u * e.exp()[:, None]
        if fit and q + 1 > case["n_eq"] and (q + 1 - case["n_eq"]) % case["stride"] == 0:
            d = u - u.mean(1, keepdim=True)
            msd += (d * d).sum((1, 2)) / n
    return u, v, mu, Wsum, cum, gth, msd, box * mu


def exact(case, seed):
    dev, reps = _device(), _replicas(case)
    th = torch.from_numpy(_theta()).to(dev)
    u, v = _thermal(case, seed)
    offs = np.concatenate([[0], np.cumsum([r["atoms"] for r in reps])])
    x0 = torch.cat([_sites(r, dev).reshape(-1, 3) for r in reps])
    # the positions as the run holds them
    u = (x0 + u) - x0
    if case["kind"] in ("energy", "autograd"):
        grad = case["kind"] == "autograd"
        C = _Crystal(reps[0], _knots(case, seed) if grad else th, dev)
        U, f, rho, _, g = C.eval(u[None], torch.ones(1, 3, dtype=torch.float64, device=dev), grad=grad)
        if grad:
            return dict(U=U[0], gx=-f[0], gtheta=g)
        return dict(f=f[0], e=U, rho=rho[0])
    groups = {}
    for q, r in enumerate(reps):
        groups.setdefault((r["lat"], *r["n"]), []).append((r, q))
    x, vo = torch.empty_like(x0), torch.empty_like(x0)
    Wd = torch.zeros(len(reps), 2, dtype=torch.float64, device=dev)
    wc = torch.zeros(len(reps), max(1, _schedule(case)[3]), dtype=torch.float64, device=dev)
    boxes = torch.zeros(len(reps), 3, dtype=torch.float64, device=dev)
    msd = torch.zeros(len(reps), dtype=torch.float64, device=dev)
    gth, cum = None, None
    for group in groups.values():
        at = [slice(offs[q], offs[q + 1]) for _, q in group]
        ug, vg, mu, Wg, cum, gth, md, bx = _exact_run(case, seed, group, torch.stack([u[a] for a in at]),
                                                      torch.stack([v[a] for a in at]), th, dev)
        for e, ((_, q), a) in enumerate(zip(group, at)):
            x[a], vo[a], Wd[q], boxes[q], msd[q] = x0[a] * mu[e] + ug[e], vg[e], Wg[e], bx[e], md[e]
            if cum[0] and case["kind"] == "runner":
                wc[q] = torch.stack(cum[0])[:, e]
    if case["kind"] == "fit":
        msd = msd / case["n_samples"]
        return dict(x=x, v=vo, msd=msd, k=3 * KB * torch.tensor([r["T"] for r in reps], dtype=torch.float64, device=dev) / msd)
    out = dict(x=x, v=vo, W=Wd)
    if case["kind"] == "switch":
        z = torch.zeros(1, dtype=torch.float64, device=dev)
        return dict(x=x, v=vo, W=Wd[0], Wcum_f=torch.cat([z, torch.stack(cum[0])[:, 0]]),
                    Wcum_b=torch.cat([z, torch.stack(cum[1])[:, 0]]))
    if case["kind"] == "runner" and case["path"] == "rs":
        out["Wcum"] = wc
    if case.get("grad"):
        out["gtheta"] = gth
    if case.get("npt"):
        out["boxes"] = boxes
    return out
