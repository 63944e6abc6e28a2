"""The work that users of this solver have it do, as cases that can be timed and compared.

A pass is what a user's program does between two looks at its simulation: advance it a number of
steps, ask for the diagnostics it records (tip, sums) and read the fields.  The grids, lattices,
parameters and storage types are those of the repository's workloads, benchmark and tests: the
isothermal alloy dendrites, the coupled heat and solute runs, the two-harmonic runs, the batched
parameter sweep, the 2D pure-substance benchmark and the isotropic sphere of the grid-anisotropy
test.  Fields are read into pinned host arrays that the program keeps (the library hands out FP64 in
every storage type); a program keeps its fields in the type that it chose to store the distributions
in, and the sums of a run that computes in 32 bits in 32 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1602_07483_gb300 import lbpf

STORED = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
KEPT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}

# Physical set-ups: parameters, undercooling or supersaturation range, frozen or initial theta.
SETUPS = {
    # isothermal alloy, cubic anisotropy: the single dendrites and the parameter sweep
    "alloy": dict(W0=1.0, tau0=1.0, D=2.0, kappa=1.0, lam=2.0 / 0.6267, Mc_inf=1.0, k=0.15, aniso=0, eps1=0.05,
                  eps2=0.0, dx=0.8, dt=0.05, antitrapping=1, grad2_min=1e-12),
    # heat and solute coupled, Lewis number 50
    "heat": dict(W0=1.0, tau0=1.0, D=2.0, kappa=100.0, lam=2.0 / 0.6267, Mc_inf=1.0, k=0.15, aniso=0, eps1=0.05,
                 eps2=0.0, dx=0.8, dt=0.05, antitrapping=1, grad2_min=1e-12),
    # the two-harmonic anisotropy of the large runs
    "harmonic": dict(W0=1.0, tau0=1.0, D=2.0, kappa=100.0, lam=2.0 / 0.6267, Mc_inf=1.0, k=0.15, aniso=1, eps1=-0.02,
                     eps2=0.015, dx=0.8, dt=0.01, antitrapping=1, grad2_min=1e-12),
    # pure substance, anisotropic (2D benchmark)
    "pure": dict(W0=1.0, tau0=1.0, D=1.0, kappa=4.0, lam=6.3826, Mc_inf=0.0, k=1.0, aniso=0, eps1=0.05, eps2=0.0,
                 dx=0.4, dt=0.008, antitrapping=0, grad2_min=1e-12),
    # pure substance, isotropic (grid-anisotropy test)
    "sphere": dict(W0=0.01, tau0=1e-4, D=1.0, kappa=0.7, lam=10.0, Mc_inf=0.0, k=1.0, aniso=0, eps1=0.0, eps2=0.0,
                   dx=0.01, dt=1.5e-5, antitrapping=0, grad2_min=1e-12),
}


def _case(name, setup, grid, lattices, storage, steps, nuclei=1, sums_every=0, tip=True, reseed=False):
    return {"name": name, "kind": "run", "setup": setup, "nx": grid[0], "ny": grid[1], "nz": grid[2],
            "q_phi": lattices[0], "q_u": lattices[1], "q_theta": lattices[2], "storage": storage, "steps": steps,
            "nuclei": nuclei, "sums_every": sums_every, "tip": tip, "reseed": reseed}


def listed():
    return [
        # the smallest call: a small box watched after every step
        _case("watch32_f64", "alloy", (32, 32, 32), (15, 19, 0), "f64", 1),
        # a whole short study of the small box: seeded, advanced 500 steps, read
        _case("study32_f64", "alloy", (32, 32, 32), (15, 19, 0), "f64", 500, reseed=True),
        # the single dendrite in plain FP64, its tip recorded every 100 steps
        _case("dendrite128_f64", "alloy", (128, 128, 128), (19, 19, 0), "f64", 100),
        # an ordinary single-precision run of a size that one look at a parameter takes
        _case("heat96_f32", "heat", (96, 96, 96), (19, 19, 7), "f32", 200),
        # the coupled run in single and in half precision storage
        _case("heat256_f32", "heat", (256, 256, 256), (19, 19, 7), "f32", 50),
        _case("heat256_f16", "heat", (256, 256, 256), (19, 19, 7), "f16", 50),
        # an uneven box in bfloat16 storage, its conservation sums watched after every step
        _case("box200_bf16", "harmonic", (200, 168, 117), (19, 19, 19), "bf16", 24, nuclei=2, sums_every=1),
        # the largest run: four nuclei in 512^3
        _case("large512_f32", "harmonic", (512, 512, 512), (19, 19, 19), "f32", 80, nuclei=4, sums_every=80),
        # the isotropic sphere on D3Q15, an odd edge
        _case("sphere301_f32", "sphere", (301, 301, 301), (15, 7, 7), "f32", 60),
        # the 2D benchmark, its tip recorded every 625 steps, and a large 2D plane
        _case("plane500_f32", "pure", (500, 500, 1), (9, 5, 5), "f32", 625, reseed=True),
        _case("plane8192_f32", "pure", (8192, 8192, 1), (9, 5, 5), "f32", 60),
        # the parameter sweep: 64 uneven boxes advanced together
        {"name": "sweep64_f16", "kind": "batch", "setup": "alloy", "members": 64, "sizes": 11, "q_phi": 19, "q_u": 19,
         "q_theta": 0, "storage": "f16", "steps": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _site_ns(case):
    """Rough device nanoseconds of a site-update, to give a drawn case a number of steps."""
    q = case["q_phi"] + case["q_u"] + case["q_theta"]
    return q * {"f64": 0.025, "f32": 0.0025, "f16": 0.0025, "bf16": 0.0025}[case["storage"]]


def draw(rng):
    kind = rng.choice(["run", "run", "run", "plane", "plane", "batch"])
    if kind == "batch":
        c = {"kind": "batch", "setup": "alloy", "members": _log_int(rng, 2, 64), "sizes": rng.randrange(1, 1000),
             "q_phi": 19, "q_u": 19, "q_theta": 0, "storage": rng.choice(["f16", "f16", "bf16", "f32", "f64"])}
        sites = sum(e ** 3 for e in _edges(c))
    elif kind == "plane":
        c = _case("", "pure", (_log_int(rng, 40, 6000), _log_int(rng, 40, 6000), 1),
                  (rng.choice([9, 9, 5]), rng.choice([5, 9]), rng.choice([5, 5, 9, 0])),
                  rng.choice(["f32", "f32", "f64", "f16", "bf16"]), 1, nuclei=rng.randrange(1, 4))
        sites = c["nx"] * c["ny"]
    else:
        setup = rng.choice(["alloy", "heat", "harmonic", "sphere"])
        lattices = (rng.choice([19, 19, 15, 7]), rng.choice([19, 19, 15, 7]),
                    0 if setup == "alloy" else rng.choice([7, 7, 15, 19]))
        storage = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
        while True:
            grid = tuple(_log_int(rng, 16, 400) for _ in range(3))
            sites = grid[0] * grid[1] * grid[2]
            if sites <= (6e6 if storage == "f64" else 3e7):
                break
        c = _case("", setup, grid, lattices, storage, 1, nuclei=rng.randrange(1, 5),
                  sums_every=rng.choice([0, 0, 1]), reseed=rng.random() < 0.25)
    if c["kind"] == "run":
        del c["name"]
    each = max(20e-6, sites * _site_ns(c) * 1e-9)
    span = math.exp(rng.uniform(math.log(2e-3), math.log(0.2)))
    c["steps"] = max(1, min(400, int(span / each)))
    return c


def _edges(case):
    """Edges of the batch's boxes, uneven as in the sweep."""
    r = np.random.default_rng(case["sizes"])
    return [int(e) for e in r.choice([48, 64, 80, 96], size=case["members"])]


def _inputs(case, seed):
    """Per simulation: grid, parameters, nuclei and initial values, from the seed alone."""
    r = np.random.default_rng(seed)
    grids = ([(e, e, e) for e in _edges(case)] if case["kind"] == "batch" else [(case["nx"], case["ny"], case["nz"])])
    out = []
    for grid in grids:
        p = dict(SETUPS[case["setup"]])
        if case["setup"] in ("alloy", "heat"):
            p["eps1"] = float(r.uniform(0.03, 0.07))
            p["k"] = float(r.choice([0.1, 0.15, 0.3]))
        n = case.get("nuclei", 1)
        centres = np.zeros((n, 3))
        for a in range(3):
            if grid[a] > 1:  # off the walls where the box has room
                m = min(14, (grid[a] - 1) // 3)
                centres[:, a] = r.integers(m, grid[a] - m, size=n)
        radii = r.uniform(5.0, 9.0, size=n) * (2.0 if case["setup"] == "pure" else 1.0)
        drive = float(r.uniform(0.3, 0.65))
        if case["setup"] in ("alloy", "heat", "harmonic"):
            U0, th0 = -drive, (0.0 if case["setup"] == "alloy" else -0.3)
        else:
            U0, th0 = 0.0, -drive
        out.append((grid, p, centres, radii, U0, th0))
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.inputs = case, _inputs(case, seed)
    lat = (case["q_phi"], case["q_u"], case["q_theta"])
    if case["kind"] == "batch":
        s.batch = lbpf.Batch.create([i[0] for i in s.inputs], lat,
                                    [lbpf.make_params(case["storage"], **i[1]) for i in s.inputs])
        s.sims = s.batch.sims
    else:
        s.sims = [lbpf.Sim(s.inputs[0][0], lat, storage=case["storage"], **s.inputs[0][1])]
    s.mask = lbpf.LBPF_PHI | lbpf.LBPF_U | (lbpf.LBPF_THETA if lat[2] else 0)
    nf = 3 if lat[2] else 2
    # the program's host arrays: one pinned FP64 block read into, one in the type it keeps
    sizes = [nf * sim.nx * sim.ny * sim.nz for sim in s.sims]
    s.read = torch.empty(sum(sizes), dtype=torch.float64, pin_memory=True)
    s.keep = s.read if case["storage"] == "f64" else torch.empty(sum(sizes), dtype=KEPT[case["storage"]])
    s.read.zero_(), s.keep.zero_()
    s.into, s.fields, at = [], [], 0
    for sim, size in zip(s.sims, sizes):
        view = s.read[at:at + size].view((nf,) + sim.shape3).numpy()
        s.into.append([view[f] if f < nf else None for f in range(3)])
        s.fields.append(s.keep[at:at + size].view((nf,) + sim.shape3))
        at += size
    for sim, (_, _, centres, radii, U0, th0) in zip(s.sims, s.inputs):
        sim.init_seed(centres, radii, U0, th0)
    return s


def run(s):
    c = s.case
    out = {}
    if c["kind"] == "batch":
        s.batch.step(c["steps"])
    else:
        sim = s.sims[0]
        _, _, centres, radii, U0, th0 = s.inputs[0]
        if c["reseed"]:
            sim.init_seed(centres, radii, U0, th0)
        left, sums = c["steps"], []
        while left:
            n = min(left, c["sums_every"] or left)
            sim.step(n)
            left -= n
            if c["sums_every"]:
                sums.append(sim.sums())
        if sums:
            out["sums"] = torch.tensor(np.array(sums), dtype=torch.float64 if c["storage"] == "f64" else torch.float32)
        if c["tip"]:
            out["tip"] = torch.tensor(sim.tip(centres[0]), dtype=s.keep.dtype)
    for sim, into in zip(s.sims, s.into):
        sim.read_fields(s.mask, out=into)
    if s.keep is not s.read:
        s.keep.copy_(s.read)
    out["fields"] = s.fields if c["kind"] == "batch" else s.fields[0]
    return out


def work(case):
    """Each population read once and written once per step, and the fields handed to the host;
    the arithmetic of the three collisions per node (about 10 operations per population and 250
    for the gradients, the anisotropy, the solute fluxes and the sources)."""
    sites = sum(e ** 3 for e in _edges(case)) if case["kind"] == "batch" else case["nx"] * case["ny"] * case["nz"]
    q = case["q_phi"] + case["q_u"] + case["q_theta"]
    b = STORED[case["storage"]]
    fields = 3 if case["q_theta"] else 2
    return {"bytes": case["steps"] * sites * 2 * q * b + fields * sites * b,
            "flops": case["steps"] * sites * (10.0 * q + 250.0)}


# ---------------------------------------------------------------- the same in plain 64-bit torch


def _lattice(q):
    """Links, weights, sound speed squared; the rest link first."""
    axes3 = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    if q == 7:
        e, w, e2 = axes3, [1 / 4] + [1 / 8] * 6, 1 / 4
    elif q == 15:
        e = axes3 + [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
        w, e2 = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8, 1 / 3
    elif q == 19:
        e = axes3 + [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if abs(a) + abs(b) + abs(c) == 2]
        w, e2 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 1 / 3
    elif q == 5:
        e, w, e2 = axes3[:4], [1 / 3] + [1 / 6] * 4, 1 / 3
    else:
        e = axes3[:4] + [(a, b, 0) for a in (1, -1) for b in (1, -1)]
        w, e2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 1 / 3
    e = [(0, 0, 0)] + e
    opp = [e.index((-a, -b, -c)) for a, b, c in e]
    return e, w, e2, opp


def _part(a, o):
    """Slices (to, from) along an axis for to[x] = from[x - o]."""
    return ((slice(max(o, 0), a + min(o, 0)), slice(max(-o, 0), a + min(-o, 0))))


def _stream(post, e, opp):
    new = []
    for i, (ex, ey, ez) in enumerate(e):
        nz, ny, nx = post[i].shape
        t = post[opp[i]].clone()  # links from outside come back
        (tz, fz), (ty, fy), (tx, fx) = _part(nz, ez), _part(ny, ey), _part(nx, ex)
        t[tz, ty, tx] = post[i][fz, fy, fx]
        new.append(t)
    return new


def _next(a, axis, d):
    """a at the neighbour d along the axis, walls mirrored."""
    n = a.shape[axis]
    at = torch.clamp(torch.arange(n, device=a.device) + d, 0, n - 1)
    return a.index_select(axis, at)


def _grad(a, dx):
    return [(_next(a, ax, 1) - _next(a, ax, -1)) / (2 * dx) for ax in (2, 1, 0)]


def _plain_step(st, p, lat, planar):
    Lp, Lu, Lt = lat
    g, h, f, phi, U, th = st
    dx, dt = p["dx"], p["dt"]
    e, w, e2, opp = Lp
    # phase field
    gr = _grad(phi, dx)
    G2 = gr[0] ** 2 + gr[1] ** 2 + gr[2] ** 2
    some = G2 >= p["grad2_min"]
    G = torch.sqrt(torch.where(some, G2, torch.ones_like(G2)))
    n = [x / G for x in gr]
    s4 = n[0] ** 4 + n[1] ** 4 + n[2] ** 4
    if p["aniso"] == 0:
        a = 1 - 3 * p["eps1"] + 4 * p["eps1"] * s4
        da = [16 * p["eps1"] * x * (x * x - s4) for x in n]
    else:
        sq = [x * x for x in n]
        a = 1 + p["eps1"] * (s4 - 0.6) + p["eps2"] * (3 * s4 + 66 * sq[0] * sq[1] * sq[2] - 17 / 7)
        da = [4 * (p["eps1"] + 3 * p["eps2"]) * n[i] * (sq[i] - s4)
              + 132 * p["eps2"] * n[i] * sq[(i + 1) % 3] * sq[(i + 2) % 3] * (1 - 3 * sq[i]) for i in range(3)]
    N = [torch.where(some, G * a * x, torch.zeros_like(x)) for x in da]
    a = torch.where(some, a, torch.ones_like(a))
    W2t = p["W0"] ** 2 / p["tau0"]
    eta = a * a * W2t * dt / (dx * dx) / e2 + 0.5
    one = 1 - phi * phi
    Q = (phi - p["lam"] * (p["Mc_inf"] * U + th) * one) * one
    wall = torch.zeros_like(phi, dtype=torch.bool)
    for ax in ((1, 2) if planar else (0, 1, 2)):
        wall.index_fill_(ax, torch.tensor([0, phi.shape[ax] - 1], device=phi.device), True)
    a2 = torch.where(wall, torch.ones_like(a), a * a)
    post = []
    for i, (ex, ey, ez) in enumerate(e):
        eq = w[i] * (phi - (ex * N[0] + ey * N[1] + ez * N[2]) * (dt / dx * W2t / e2))
        far = torch.roll(g[i], (-ez, -ey, -ex), (0, 1, 2))
        post.append((g[i] - (1 - a2) * far - (g[i] - eq) / eta + w[i] * Q * dt / p["tau0"]) / a2)
    g = _stream(post, e, opp)
    new = sum(g)
    # supersaturation
    e, w, e2, opp = Lu
    q = 0.5 * (1 - new)
    iz = 2 / ((1 + p["k"]) - (1 - p["k"]) * new)
    gp, gq, F = _grad(new, dx), _grad(q * iz, dx), _grad(iz, dx)
    div = 0
    for ax in (0, 1, 2):
        for d in (1, -1):
            div = div + 0.5 * (q + _next(q, ax, d)) * (_next(iz, ax, d) - iz)
    div = div * p["D"] / (dx * dx)
    rate = (new - phi) / dt
    c = 1 + (1 - p["k"]) * U
    G2 = gp[0] ** 2 + gp[1] ** 2 + gp[2] ** 2
    some = (G2 >= p["grad2_min"]) if p["antitrapping"] else torch.zeros_like(G2, dtype=torch.bool)
    amp = torch.where(some, -p["W0"] / (2 * math.sqrt(2)) * c * rate / torch.sqrt(torch.where(some, G2, torch.ones_like(G2))),
                      torch.zeros_like(G2))
    j = [amp * x for x in gp]
    J = [p["D"] * (gq[i] + q * F[i]) * U + j[i] * iz for i in range(3)]
    src = U * div + j[0] * F[0] + j[1] * F[1] + j[2] * F[2] + c * 0.5 * rate * iz
    eta = p["D"] * dt / (dx * dx) / e2 + 0.5
    post = []
    for i, (ex, ey, ez) in enumerate(e):
        b = w[i] - 1 if i == 0 else w[i]
        eq = (U if i == 0 else 0) + b * (q * iz * U + (ex * J[0] + ey * J[1] + ez * J[2]) * (dt / dx / e2))
        post.append(h[i] - (h[i] - eq) / eta + w[i] * src * dt)
    h = _stream(post, e, opp)
    # temperature
    if f is not None:
        e, w, e2, opp = Lt
        eta = p["kappa"] * dt / (dx * dx) / e2 + 0.5
        f = _stream([f[i] - (f[i] - w[i] * th) / eta + w[i] * 0.5 * rate * dt for i in range(len(e))], e, opp)
        th = sum(f)
    return g, h, f, new, sum(h), th


def _plain_run(case, inputs, sums_every=0):
    grid, p, centres, radii, U0, th0 = inputs
    planar = case["q_phi"] in (5, 9)
    qs = (case["q_phi"], case["q_u"], case["q_theta"])
    lat = [_lattice(q) if q else None for q in qs]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    z, y, x = torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device=dev) for n in grid[::-1]], indexing="ij")
    arg = None
    for c, r in zip(centres, radii):
        v = (float(r) - torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)) * p["dx"] / (math.sqrt(2) * p["W0"])
        arg = v if arg is None else torch.maximum(arg, v)
    phi = torch.tanh(arg)
    del x, y, z, arg
    g = [w * phi for w in lat[0][1]]
    qz = 0.5 * (1 - phi) * 2 / ((1 + p["k"]) - (1 - p["k"]) * phi)
    h = [((1.0 if i == 0 else 0.0) + (w - 1 if i == 0 else w) * qz) * U0 for i, w in enumerate(lat[1][1])]
    f = [torch.full_like(phi, w * th0) for w in lat[2][1]] if qs[2] else None
    st = (g, h, f, phi, torch.full_like(phi, U0), torch.full_like(phi, th0))
    sums = []
    for n in range(1, case["steps"] + 1):
        st = _plain_step(st, p, lat, planar)
        if sums_every and (n % sums_every == 0 or n == case["steps"]):
            _, _, _, a, U, th = st
            zeta = 0.5 * ((1 + p["k"]) - (1 - p["k"]) * a)
            sums.append([float(v.sum()) for v in (a, U, th, zeta * (1 + (1 - p["k"]) * U))])
    return torch.stack(st[3:6] if qs[2] else st[3:5]).cpu(), sums


def exact(case, seed):
    sims = _inputs(case, seed)
    q = case["q_phi"] + case["q_u"] + case["q_theta"]
    # seconds this takes: the launches of some 30 operations per population, and their passes over the fields
    if sum(case["steps"] * (30 * q + 300) * (5e-6 + math.prod(i[0]) * 4e-12) for i in sims) > 18:
        return None
    out = {}
    got = [_plain_run(case, i, case.get("sums_every", 0)) for i in sims]
    if case["kind"] == "batch":
        return {"fields": [f for f, _ in got]}
    if case["sums_every"]:
        out["sums"] = torch.tensor(got[0][1], dtype=torch.float64)
    if case["tip"]:
        out["tip"] = None
    out["fields"] = got[0][0]
    return out
