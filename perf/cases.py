"""Measured cases of the dose engine: what its users run, through the public entry points of
paper_1109_3266_gb300.ctd.

A case names a form of the engine and a problem of `inputs`:
  run     a dose calculation on a loaded phantom: ctd_run, then dose, standard error and stats
  call    the whole call from host arrays: phantom upload, set-up, run, read-back, release
  range   a shard of a problem's histories: ctd_run_range and the raw energy tally
  batch   several requests in one ctd_run_batch
  served  several requests through the served form, each stopped at its avg RSD
  noalloc the precision measures of device-resident dose arrays (ctd_avg_rsd_noalloc)
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_1109_3266_gb300 import ctd, inputs as I

COUNTS = ("pe", "compton", "rayleigh", "fictitious", "escaped", "missed", "cutoff", "terminated", "aborted", "steps",
          "histories")
TOTALS = ("e_emitted_kev", "e_escaped_kev", "e_deposited_kev", "avg_rsd", "paper_sigma_bar", "d_max")


def listed():
    return [
        # the smallest calculation: a quality check on a water cube, 1e5 photons of one energy
        dict(name="water_check", form="run", phantom="water", nx=32, ny=32, nz=32, d=0.5, source="static",
             histories=100_000, batches=10),
        # a quick low-precision look at a coarse head, sizes that divide nothing
        dict(name="head_preview", form="run", phantom="head", nx=51, ny=51, nz=32, d=0.5, source="arc", kvp=100,
             histories=1_000_003, batches=7),
        # the paper's head-and-neck scan: a new patient from host arrays, 200 degree arc, 2.5e8 photons
        dict(name="head_scan_call", form="call", phantom="head", nx=128, ny=128, nz=60, d=0.4, source="arc200",
             kvp=125, histories=250_000_000, batches=10),
        # the benchmark's two workloads at their full sizes
        dict(name="cbct_water", form="run", phantom="water", nx=256, ny=256, nz=128, d=0.2, source="cbct", kvp=120,
             histories=1_000_000_000, batches=10),
        dict(name="head_full", form="run", phantom="head", nx=256, ny=256, nz=160, d=0.1, source="halffan", kvp=100,
             histories=2_000_000_000, batches=10),
        # a measured (bowtie) fluence map in front of the water phantom
        dict(name="cbct_bowtie", form="run", phantom="water", nx=256, ny=256, nz=128, d=0.2, source="bowtie",
             kvp=120, histories=100_000_000, batches=10),
        # the paper's default physics: Waller-Hartree Compton, independent-atom Rayleigh
        dict(name="head_wh_iaa", form="run", phantom="head", nx=64, ny=64, nz=40, d=0.4, source="halffan", kvp=100,
             compton="wh", rayleigh="iaa", histories=50_000_000, batches=10),
        # helical CT, continuous rotation
        dict(name="helical_ct", form="run", phantom="head", nx=48, ny=48, nz=40, d=0.5, source="helix", kvp=120,
             histories=10_000_000, batches=10),
        # one worker's ragged share of a primary-only calculation
        dict(name="primary_share", form="range", phantom="water", nx=256, ny=256, nz=128, d=0.2, source="cbct",
             kvp=120, mode="max_real", histories=100_000_000, batches=10, begin=12_345_678, end=45_678_901),
        # a planning queue: uneven water and head requests in one call
        dict(name="batch_of_requests", form="batch", requests=16, side_max=128, lo=1e6, hi=1e7, batches=10),
        # online requests on coarse heads, each until 1 % avg RSD
        dict(name="served_requests", form="served", requests=8, nx=26, ny=26, nz=16, d=1.0, kvp=100,
             batch=4_000_000, target=0.01),
        # the precision measures alone, on arrays of the full head's size
        dict(name="precision_of_dose", form="noalloc", phantom="head", nx=256, ny=256, nz=160, d=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(("run", "run", "run", "call", "range", "batch", "served", "noalloc"))
    if form == "batch":
        return dict(form=form, requests=rng.randint(4, 24), side_max=rng.choice((96, 128, 160)), lo=1e6,
                    hi=float(_log(rng, 2e6, 3e7)), batches=rng.randint(2, 12))
    if form == "served":
        nx = rng.randint(20, 52)
        return dict(form=form, requests=rng.randint(2, 10), nx=nx, ny=nx, nz=rng.randint(12, 33), d=26.0 / nx,
                    kvp=rng.randint(80, 125), batch=_log(rng, 1e6, 2e7), target=round(rng.uniform(0.01, 0.03), 4))
    phantom = rng.choice(("water", "head"))
    big = form == "noalloc" or rng.random() < 0.3
    nx, ny = (rng.randint(120, 256) for _ in range(2)) if big else (rng.randint(24, 120) for _ in range(2))
    nz = rng.randint(60, 160) if big else rng.randint(16, 70)
    c = dict(form=form, phantom=phantom, nx=nx, ny=ny, nz=nz, d=round(25.6 / max(nx, ny), 3))
    if form == "noalloc":
        return dict(c, phantom="head")
    if form == "run" and rng.random() < 0.2:
        # a small monoenergetic check
        n = rng.randint(16, 48)
        return dict(form="run", phantom="water", nx=n, ny=rng.randint(16, 48), nz=n, d=0.5, source="static",
                    histories=_log(rng, 2e4, 2e5), batches=rng.randint(2, 12))
    c["source"] = rng.choice(("arc", "arc200", "cbct", "halffan", "helix", "bowtie"))
    c["kvp"] = rng.randint(80, 140)
    c["batches"] = rng.randint(2, 20)
    c["histories"] = _log(rng, 2e5, 3e8)
    if rng.random() < 0.3:
        c.update(compton="wh", rayleigh="iaa")
    if form == "range":
        c["begin"] = rng.randint(0, c["histories"] // 3)
        c["end"] = rng.randint(c["histories"] // 2, c["histories"])
        if rng.random() < 0.5:
            c["mode"] = "max_real"
    return c


# ----------------------------------------------------------------------- problems
def _phantom(c, seed):
    if c["phantom"] == "water":
        return I.uniform_box(c["nx"], c["ny"], c["nz"], c["d"], I.thomson(I.WATER) if c["source"] == "static" else I.WATER)
    return I.head_phantom(c["nx"], c["ny"], c["nz"], c["d"], seed)


def _source(c, seed):
    hu, hv = 0.4 * c["nx"] * c["d"], 0.4 * c["nz"] * c["d"]
    kind = c["source"]
    if kind == "static":
        return I.static_source(50.0, 5.0, 5.0)
    if kind == "arc":
        return I.arc_source(100.0, -hu, hu, -hv, hv, n_proj=360)
    if kind == "arc200":
        return I.arc_source(100.0, -hu, hu, -hv, hv, n_proj=200, arc0=0.0, arc1=math.radians(200.0))
    if kind == "halffan":
        return I.arc_source(100.0, -1.0, 13.5, -8.0, 8.0, n_proj=360)
    if kind == "helix":
        return I.helical_source(100.0, -hu, hu, -1.0, 1.0, 2.5, -hv, hv, continuous=True)
    src = I.arc_source(100.0, -10.0, 10.0, -10.0, 10.0, n_proj=360)
    return replace(src, fluence=I.bowtie_fluence(128, 32, seed=seed)) if kind == "bowtie" else src


def _problem(c, seed):
    line = c["source"] == "static"
    mode = c.get("mode", "full")
    phys = I.Physics(e_min=10 if line else 1, e_max=150, mode=mode, max_real=1 if mode == "max_real" else 0,
                     compton=c.get("compton", "kn"), rayleigh=c.get("rayleigh", "gauss"))
    spec = I.spectrum_line(60.0) if line else I.spectrum_kramers(c["kvp"], 2.5)
    return I.Problem(c.get("name", "case"), _phantom(c, seed), _source(c, seed), spec, phys, c["histories"],
                     c["batches"], seed)


def _requests(c, seed):
    """The requests' kinds, sizes and histories are the case's; densities and histories' keys the seed's."""
    sides = tuple(range(64, c["side_max"] + 1, 32))
    out = []
    for k, p in enumerate(I.batched_requests(c["requests"], 4, c["lo"], c["hi"], sides)):
        ph = p.phantom
        if p.meta["kind"] == "head":
            ph = I.head_phantom(ph.nx, ph.ny, ph.nz, ph.dx, seed + k, size_ref=(25.6, 25.6, 25.6))
        out.append(replace(p, phantom=ph, n_batches=c["batches"], seed=seed + k))
    return out


class _State:
    """A context and what a program holds beside it; the context goes with it."""

    def __init__(self, case, **held):
        self.case = case
        self.__dict__.update(held)

    def __del__(self):
        if getattr(self, "ctx", None):
            ctd.ctd_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    form = case["form"]
    if form == "noalloc":
        return _State(case, **_dose_arrays(case, seed))
    ctx = ctd.ctd_create(device=0, stream=torch.cuda.current_stream().cuda_stream,
                         serve_round_histories=1e9 if form == "served" else 0.0)
    if form == "batch":
        ps = _requests(case, seed)
        return _State(case, ctx=ctx, problems=ps, handles=[ctd.load_problem(ctx, p) for p in ps])
    if form == "served":
        ps = [I.head_request(I.head_phantom(case["nx"], case["ny"], case["nz"], case["d"], seed + r), seed + 100 + r,
                             kvp=case["kvp"]) for r in range(case["requests"])]
        return _State(case, ctx=ctx, problems=ps, handles=[ctd.load_problem(ctx, p) for p in ps])
    p = _problem(case, seed)
    return _State(case, ctx=ctx, problem=p, handle=None if form == "call" else ctd.load_problem(ctx, p))


def _outputs(dose, sd, st):
    return {"dose": dose, "stddev": sd, "counts": np.array([st[k] for k in COUNTS], dtype=np.int64),
            "totals": np.array([st[k] for k in TOTALS])}


def run(state):
    c, form = state.case, state.case["form"]
    if form == "run":
        dose, sd, st, _ = ctd.run_problem(state.ctx, state.problem, state.handle)
        return _outputs(dose, sd, st)
    if form == "call":
        dose, sd, st, h = ctd.run_problem(state.ctx, state.problem)
        ctd.ctd_destroy_phantom(state.ctx, h)
        return _outputs(dose, sd, st)
    if form == "range":
        p = state.problem
        ctd.ctd_run_range(state.ctx, state.handle, p.n_hist, p.seed, p.n_batches, c["begin"], c["end"])
        edep = ctd.ctd_get_edep(state.ctx, state.handle, p.phantom.nvox)
        _, _, st = ctd.ctd_get_dose_and_stddev(state.ctx, state.handle, 0, want_arrays=False)
        return {"edep": edep, "counts": np.array([st[k] for k in COUNTS], dtype=np.int64),
                "totals": np.array([st[k] for k in TOTALS[:3]])}
    if form == "batch":
        ps = state.problems
        ctd.ctd_run_batch(state.ctx, state.handles, [p.n_hist for p in ps], [p.seed for p in ps], c["batches"])
    elif form == "served":
        for h, p in zip(state.handles, state.problems):
            ctd.ctd_submit(state.ctx, h, c["batch"], c["target"], p.seed, n_histories_max=200 * c["batch"])
        while ctd.ctd_serve_wait(state.ctx, 0.01):
            pass
    else:
        ctd.ctd_avg_rsd_noalloc(state.dose.data_ptr(), state.sd.data_ptr(), state.rho.data_ptr(), state.dose.numel(),
                                state.result.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state.result
    return [_outputs(*ctd.ctd_get_dose_and_stddev(state.ctx, h, p.phantom.nvox))
            for h, p in zip(state.handles, state.problems)]


# Woodcock steps of a history in each kind of phantom, about; a step is some forty operations
# (free path, move, two interpolations, the choice), a scatter eighty more, a source photon a hundred
STEPS = {"water": (5.0, 4.0), "head": (16.0, 2.0)}


def work(case):
    if case["form"] == "noalloc":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 20 * n + 24, "flops": 4 * n}
    if case["form"] == "batch":
        ps = _sizes(case)
    elif case["form"] == "served":
        # batches until the target: ten at least, about 1.06e8 histories to 1 % on 1 cm voxels
        need = 1.06e8 * (0.01 / case["target"]) ** 2 / case["d"] ** 3
        ps = [("head", case["nx"] * case["ny"] * case["nz"], max(10 * case["batch"], min(need, 200 * case["batch"])))
              ] * case["requests"]
    else:
        n = case["histories"] if case["form"] != "range" else case["end"] - case["begin"]
        ps = [(case["phantom"], case["nx"] * case["ny"] * case["nz"], n)]
    out = {"bytes": 0, "flops": 0}
    for kind, nvox, n in ps:
        steps, scatters = STEPS[kind]
        # material and density read once, dose and standard error (or the tally) written once
        out["bytes"] += nvox * (5 + (8 if case["form"] == "range" else 16))
        out["flops"] += n * (100 + 40 * steps + 80 * (1 if case.get("mode") == "max_real" else scatters))
    return out


def _sizes(case):
    """(kind, voxels, histories) of a batch's requests, about: the middle of their ranges."""
    mid = math.exp(0.5 * (math.log(case["lo"]) + math.log(case["hi"])))
    side = (64 + case["side_max"]) // 2
    return [("water" if r % 2 == 0 else "head", side ** 3, mid) for r in range(case["requests"])]


# ----------------------------------------------------------------------- precision arrays
def _dose_arrays(case, seed):
    """A dose falling off from the surface with its standard error, and the phantom's densities."""
    ph = I.head_phantom(case["nx"], case["ny"], case["nz"], case["d"], seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    rho = torch.from_numpy(ph.rho.ravel()).cuda()
    r = torch.rand(rho.numel(), generator=g, device="cuda", dtype=torch.float64)
    dose = 1e-15 * torch.exp(-3.0 * r) * (rho.double() + 0.05)
    sd = dose * (0.01 + 0.02 * torch.rand(rho.numel(), generator=g, device="cuda", dtype=torch.float64))
    return {"rho": rho, "dose": dose, "sd": sd, "result": torch.zeros(3, device="cuda", dtype=torch.float64)}


def _exact_precision(case, seed):
    a = _dose_arrays(case, seed)
    m = a["rho"] >= 0.1
    d, s = a["dose"][m], a["sd"][m]
    dmax = d.max()
    k1, k2 = d > 0.1 * dmax, d > 0.2 * dmax
    return torch.stack([(s[k1] / d[k1]).mean(), s[k2].mean() / dmax, dmax])


# ----------------------------------------------------------------------- the method in 64 bits
# Mono-energetic photons from a static source into a water box, history by history with the same
# counter-based random numbers (Philox4x32-10), in numpy float64.
MEC2, R0, NA = 510.99895, 2.8179403262e-13, 6.02214076e23


def _philox(h, step, stream, seed):
    u32, mask = np.uint64(32), np.uint64(0xFFFFFFFF)
    c = [h & mask, h >> u32, np.broadcast_to(np.uint64(step), h.shape), np.broadcast_to(np.uint64(stream), h.shape)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> u32) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> u32) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(2.0 * (x >> np.uint64(9)).astype(np.float64) + 1.0) * 2.0 ** -24 for x in c]


def _water_tables(e):
    """Cumulative mass attenuation (cm^2/g) of water at node energies e, in the engine's closed forms."""
    m = I.WATER
    k = e / MEC2
    kn = 2 * np.pi * R0 ** 2 * ((1 + k) / k ** 2 * (2 * (1 + k) / (1 + 2 * k) - np.log1p(2 * k) / k)
                                + np.log1p(2 * k) / (2 * k) - (1 + 3 * k) / (1 + 2 * k) ** 2)
    pe = 1e-2 * m.z_eff ** 4 / (e * 1e-3) ** 3 * 1e-30 * NA / m.a_mol
    ray = 1.565e-5 * m.z_eff ** 2 / (e * 1e-3) ** 2 * 1e-24 * NA / m.a_mol
    return np.cumsum([pe, NA * m.z_over_a * kn, ray], axis=0)


def _surface(pdf, n_zeta=1024):
    mu = np.linspace(-1.0, 1.0, 20001)
    zeta = np.arange(n_zeta) / (n_zeta - 1.0)
    rows = []
    for p in pdf(mu):
        cdf = np.concatenate([[0.0], np.cumsum(0.5 * (p[1:] + p[:-1]))])
        rows.append(np.interp(zeta, cdf / cdf[-1], mu))
    return np.array(rows)


def _exact_water(case, seed):
    p = _problem(case, seed)
    ph, n, nb, e_min, e_max = p.phantom, p.n_hist, p.n_batches, p.physics.e_min, p.physics.e_max
    e_node = np.arange(e_min, e_max + 1, dtype=np.float64)
    cum = _water_tables(e_node)
    kk = (e_node / MEC2)[:, None]

    def klein_nishina(mu):
        r = 1.0 / (1.0 + kk * (1.0 - mu))
        return r * r * (r + 1.0 / r - 1.0 + mu * mu)

    S = {1: _surface(klein_nishina), 2: _surface(lambda mu: np.broadcast_to(1.0 + mu * mu, (e_node.size, mu.size)))}
    half = 0.5 * ph.dx * np.array([ph.nx, ph.ny, ph.nz])
    dims = np.array([ph.nx, ph.ny, ph.nz])
    src = p.source
    h = np.arange(n, dtype=np.uint64)
    e = np.full(n, 60.0)
    uu, vv = np.zeros(n), np.zeros(n)
    todo, t = np.arange(n), 1
    while todo.size:
        a, b, c, _ = _philox(h[todo], t, 1, seed)
        uu[todo], vv[todo] = src.u_lo + (src.u_hi - src.u_lo) * a, src.v_lo + (src.v_hi - src.v_lo) * b
        c2 = src.sad ** 2 / (uu[todo] ** 2 + vv[todo] ** 2 + src.sad ** 2)
        todo, t = todo[c >= c2 * np.sqrt(c2)], t + 1
    u = np.stack([uu, vv, np.full(n, src.sad)], axis=1)
    u /= np.linalg.norm(u, axis=1)[:, None]
    r0 = np.array([0.0, 0.0, -src.sad])
    with np.errstate(divide="ignore"):
        t0, t1 = (-half - r0) / u, (half - r0) / u
    tn, tf = np.minimum(t0, t1).max(axis=1), np.maximum(t0, t1).min(axis=1)
    live = np.flatnonzero((tn < tf) & (tf > 0.0))
    g = np.clip((r0 + np.maximum(tn, 0.0)[:, None] * u + half) / ph.dx, 0.0, dims * (1.0 - 1e-16))
    size = np.array([n // nb + (b < n % nb) for b in range(nb)])
    batch = np.repeat(np.arange(nb), size)
    edep = np.zeros((nb, ph.nvox))
    emitted, escaped = float(e.sum()), float(e.sum() - e[live].sum())
    step = 0
    while live.size:
        x = _philox(h[live], step, 0, seed)
        step += 1
        j = np.clip((e[live] - e_min).astype(int), 0, e_node.size - 2)
        te = e[live] - e_node[j]
        c1, c2, c3 = cum[:, j] + te * (cum[:, j + 1] - cum[:, j])
        g[live] += (-np.log(x[0]) / c3 / ph.dx)[:, None] * u[live]
        out = ((g[live] < 0.0) | (g[live] >= dims)).any(axis=1)
        escaped += float(e[live[out]].sum())
        real = ~out & (x[1] < 1.0)
        i = g[live].astype(int) @ np.array([1, ph.nx, ph.nx * ph.ny])
        kind = np.where(x[1] * c3 < c1, 0, np.where(x[1] * c3 < c2, 1, 2))
        z = x[2] * 1023.0
        iz = np.minimum(z.astype(int), 1022)
        a = z - iz
        mu = np.zeros(live.size)
        for k in (1, 2):
            lo = S[k][j, iz] + a * (S[k][j, iz + 1] - S[k][j, iz])
            hi = S[k][j + 1, iz] + a * (S[k][j + 1, iz + 1] - S[k][j + 1, iz])
            mu = np.where(kind == k, np.clip(lo + te * (hi - lo), -1.0, 1.0), mu)
        ep = np.where(kind == 1, e[live] / (1.0 + e[live] / MEC2 * (1.0 - mu)), e[live])
        end = real & ((kind == 0) | (ep < e_min))
        dep = np.where(end, e[live], e[live] - ep)
        np.add.at(edep, (batch[live[real]], i[real]), dep[real])
        e[live] = ep
        # rotation by mu and azimuth 2 pi x3 about the flight direction
        st, cp, sp = np.sqrt(np.maximum(1.0 - mu * mu, 0.0)), np.cos(2 * np.pi * x[3]), np.sin(2 * np.pi * x[3])
        ux, uy, uz = u[live].T
        s = np.sqrt(ux * ux + uy * uy)
        axis = s * s < 1e-12
        q = st / np.where(axis, 1.0, s)
        v = np.stack([np.where(axis, st * cp, q * (ux * uz * cp - uy * sp) + ux * mu),
                      np.where(axis, st * sp, q * (uy * uz * cp + ux * sp) + uy * mu),
                      np.where(axis, np.sign(uz) * mu, -s * st * cp + uz * mu)], axis=1)
        u[live] = v / np.linalg.norm(v, axis=1)[:, None]
        live = live[real & ~end]
    d = edep * (1.602176634e-13 / (ph.dx ** 3 * size[:, None]))
    dose, sd = d.mean(axis=0), d.std(axis=0, ddof=1) / math.sqrt(nb)
    dmax = dose.max()
    k1, k2 = dose > 0.1 * dmax, dose > 0.2 * dmax
    totals = [emitted, escaped, edep.sum(), (sd[k1] / dose[k1]).mean(), sd[k2].mean() / dmax, dmax]
    return {"dose": dose, "stddev": sd, "counts": None, "totals": np.array(totals)}


def exact(case, seed):
    if case["form"] == "noalloc":
        return _exact_precision(case, seed)
    if case.get("source") == "static":
        return _exact_water(case, seed)
    # the other calculations take hours in plain numpy
    return None
