"""The work a user of this library has it do, as cases that can be timed and checked.

A case is a configuration (water-like cube, four-type monolayer, atom-and-bead
nanowire, two-type mixture with per-pair cutoffs), a precision form and the entry
point that a program calls on it:

  md       steps of velocity-Verlet MD in one call (nep_md_step, nep_md_step_hnemd)
  compute  energy, forces and per-particle virials of one configuration
           (nep_compute on device arrays, Model.compute on host arrays,
           nep_compute_static without allocation)
  batch    the same for many configurations of two models at once (nep_compute_batch)

The sizes are those of the repository's benchmark configurations and tests.

Outputs.  The FP64 form's outputs are returned as they are.  The FP32 and BF16 forms
widen FP32 numbers into the interface's FP64 arrays; a program that runs them keeps
the results (training labels, trajectory frames) in FP32, and so do these cases, with
one conversion of all outputs together.
"""
import math

import numpy as np
import torch

from paper_2603_01234_gb300 import binding, inputs

KB = 8.617333262e-5        # eV/K
ACC = 9.648533212e-3       # 1 eV/(A amu) in A/fs^2

# Per system: types, hidden width, cutoffs and MD step as in the benchmark's configurations.
SYSTEMS = {
    "water": dict(n_types=1, hidden=30, rc_radial=8.0, rc_angular=5.0, dt=10.0),
    "monolayer": dict(n_types=4, hidden=50, rc_radial=15.0, rc_angular=11.0, dt=20.0),
    "nanowire": dict(n_types=3, hidden=40, rc_radial=7.0, rc_angular=5.0, dt=5.0),
    "mixture": dict(n_types=2, hidden=30, rc_radial=((6.0, 7.0), (7.0, 8.0)), rc_angular=((5.0, 6.0), (6.0, 7.0)),
                    dt=5.0),
}


def listed():
    return [
        # the benchmark's first configuration: a 512-bead box, everything in FP64
        dict(name="md_water512_fp64", kind="md", system="water", n=512, form="fp64", steps=10, drive=False),
        # the same box in the FP32 form: the smallest MD, bound by latency and launches
        dict(name="md_water512_fp32", kind="md", system="water", n=512, form="fp32", steps=16, drive=False),
        # the headline workload: NVE of 100,000-bead water
        dict(name="md_water100k_fp32", kind="md", system="water", n=100_000, form="fp32", steps=20, drive=False),
        # four types, few neighbours, long cutoffs
        dict(name="md_monolayer200k_fp32", kind="md", system="monolayer", n=200_000, form="fp32", steps=20,
             drive=False),
        # the largest system: three types, uneven neighbour counts, open axes
        dict(name="md_nanowire1m_fp32", kind="md", system="nanowire", n=1_000_000, form="fp32", steps=10,
             drive=False),
        # thermal conductivity: HNEMD driving force, thermostat, heat current (per-particle virials every step)
        dict(name="hnemd_nanowire60k_fp32", kind="md", system="nanowire", n=60_001, form="fp32", steps=10,
             drive=True),
        # labels of one large configuration in FP64 (the accuracy reference of the FP32 form)
        dict(name="compute_water100k_fp64", kind="compute", system="water", n=100_000, form="fp64",
             many_body=False, mem="device"),
        # one mid-sized configuration with the four- and five-body descriptors, ragged size
        dict(name="compute_water2999_manybody", kind="compute", system="water", n=2999, form="fp32",
             many_body=True, mem="device"),
        # the smallest call: one small configuration from and to host arrays
        dict(name="compute_water64_host", kind="compute", system="water", n=64, form="fp32", many_body=False,
             mem="host"),
        # two types with per-pair cutoffs through the allocation-free entry point
        dict(name="static_mixture1500", kind="compute", system="mixture", n=1500, form="fp32", many_body=False,
             mem="static"),
        # BF16 hidden-layer weights on a four-type monolayer
        dict(name="compute_monolayer50k_bf16", kind="compute", system="monolayer", n=50_000, form="bf16",
             many_body=False, mem="device"),
        # a served batch: 64 configurations of 64 to 4,096 beads, two models
        dict(name="batch64_mixed_fp32", kind="batch", requests=64, n_max=4096, mix=1004, form="fp32"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "compute", "compute", "batch"])
    if kind == "batch":
        form = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind="batch", requests=_log_uniform(rng, 2, 96 if form == "fp32" else 24),
                    n_max=_log_uniform(rng, 128, 4096), mix=rng.randrange(1 << 20), form=form)
    system = rng.choice(sorted(SYSTEMS))
    if kind == "md":
        form = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp64"])
        top = {"water": 120_000, "mixture": 60_000, "monolayer": 240_000, "nanowire": 800_000}[system]
        n = _log_uniform(rng, 512, top if form != "fp64" else top // 40)
        steps = max(2, min(10, int(4e5 / n))) if form != "fp64" else 4
        return dict(kind="md", system=system, n=n, form=form, steps=steps, drive=rng.random() < 0.25)
    form = rng.choice(["fp32", "fp32", "bf16", "fp64"])
    mem = rng.choice(["device", "device", "host", "static"])
    top = {"device": 200_000 if form != "fp64" else 40_000, "host": 20_000, "static": 4000}[mem]
    return dict(kind="compute", system=system, n=_log_uniform(rng, 64, top), form=form,
                many_body=rng.random() < 0.3, mem=mem)


# ---- inputs --------------------------------------------------------------------------
def _model(system, seed, many_body=False):
    s = SYSTEMS[system]
    return inputs.random_model(n_types=s["n_types"], hidden=s["hidden"], rc_radial=s["rc_radial"],
                               rc_angular=s["rc_angular"], seed=seed, l_max_4b=2 if many_body else 0,
                               l_max_5b=1 if many_body else 0)


def _system(system, n, seed):
    """A configuration of about n particles (the monolayer comes in cells of four)."""
    if system == "monolayer":
        cells = max(6, n // 4)
        nx = max(2, int(round(math.sqrt(cells))))
        return inputs.monolayer(nx, max(2, int(round(cells / nx))), seed=seed)
    if system == "nanowire":
        # long wires where there are particles enough, the benchmark's 196 cells at most;
        # the shortest holds its atomistic core and a sheath
        n = max(n, 1500)
        return inputs.nanowire(n, seed=seed, n_cells_x=max(6, min(196, n // 250)))
    s = inputs.water_box(n, seed=seed)
    if system == "mixture":
        s.types = np.random.default_rng(seed + 1).integers(0, 2, size=n).astype(np.int32)
        s.masses = np.array([12.0, 40.0])
    return s


def _requests(case, seed):
    """(model, system) of each request: sizes log-uniform from 64 on, a coin picks the
    system.  The mix of sizes is the case's, the configurations are the seed's."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for r in range(case["requests"]):
        n = int(round(math.exp(rng.uniform(math.log(64), math.log(case["n_max"])))))
        m = int(rng.uniform() < 0.5)
        out.append((m, _system(("water", "monolayer")[m], n, seed + 7919 * (r + 1))))
    return out


def _md_inputs(case, seed):
    s = _system(case["system"], case["n"], seed)
    vel = inputs.maxwell_boltzmann(s, 300.0, seed=seed + 2)
    noise = binding.bussi_noise(case["steps"], s.n, seed=seed + 3) if case["drive"] else None
    return s, vel, noise


FIELD, TEMPERATURE, TAU = (0.0, 0.0, 1e-3), 300.0, 100.0  # of the driven runs


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        reqs = _requests(case, seed)
        models = [binding.Model(_model("water", seed), case["form"]),
                  binding.Model(_model("monolayer", seed), case["form"])]
        req_n, box, pbc, types, pos = binding.pack_requests([s for _, s in reqs])
        n, k = int(req_n.sum()), len(reqs)
        return dict(case=case, models=models, which=np.array([m for m, _ in reqs], np.int32), req_n=req_n, box=box,
                    pbc=pbc, types=torch.from_numpy(types).to(dev), pos=torch.from_numpy(pos).to(dev),
                    out=_out_buffer(n, k, dev), n=n, k=k)
    model = binding.Model(_model(case["system"], seed, case.get("many_body", False)), case["form"])
    if case["kind"] == "compute":
        s = _system(case["system"], case["n"], seed)
        if case["mem"] == "host":
            return dict(case=case, model=model, system=s)
        return dict(case=case, model=model, n=s.n, box=s.box, pbc=s.pbc, types=torch.from_numpy(s.types).to(dev),
                    pos=torch.from_numpy(s.pos).to(dev), out=_out_buffer(s.n, 1, dev))
    s, vel, noise = _md_inputs(case, seed)
    types = torch.from_numpy(s.types).to(dev)
    start = torch.zeros(3, 3, s.n, dtype=torch.float64, device=dev)  # positions, velocities, forces
    start[0] = torch.from_numpy(s.pos)
    start[1] = torch.from_numpy(vel)
    if not case["drive"]:  # a driven call forms its own first forces, which hold the driving force
        binding.nep_compute(model.h, types, start[0], s.box, s.pbc, force=start[2])
    return dict(case=case, model=model, system=s, types=types, start=start, now=torch.empty_like(start), noise=noise,
                thermo=np.zeros((1, 12)), heat=np.zeros((1, 6)))


def _out_buffer(n, k, dev):
    """All outputs of an evaluation behind one another, so that one conversion covers them."""
    return torch.zeros(10 * k + 13 * n, dtype=torch.float64, device=dev)


def _views(flat, n, k):
    cut = [0, k, 10 * k, 10 * k + n, 10 * k + 4 * n, 10 * k + 13 * n]
    names = ("energy", "virial_total", "site_energy", "force", "virial")
    return {name: flat[a:b] for name, a, b in zip(names, cut, cut[1:])}


def _kept(x, form):
    """FP64 results as they are, those of the reduced forms in FP32 (see above)."""
    if form == "fp64":
        return x
    return x.astype(np.float32) if isinstance(x, np.ndarray) else x.to(torch.float32)


# ---- one pass -------------------------------------------------------------------------
def run(state):
    case = state["case"]
    form = case["form"]
    if case["kind"] == "md":
        s, now, steps = state["system"], state["now"], case["steps"]
        now.copy_(state["start"])  # every pass runs the same steps
        dt = SYSTEMS[case["system"]]["dt"]
        pos, vel, force = now[0], now[1], now[2]
        out = {}
        if case["drive"]:
            binding.nep_md_step_hnemd(state["model"].h, state["types"], s.masses, s.box, s.pbc, pos, vel, force, 0,
                                      steps, dt, np.array(FIELD), TEMPERATURE, TAU, state["noise"], steps,
                                      state["thermo"], state["heat"])
            out["heat"] = _kept(state["heat"], form)
        else:
            binding.nep_md_step(state["model"].h, state["types"], s.masses, s.box, s.pbc, pos, vel, force, 1, steps,
                                dt, steps, state["thermo"])
        frame = _kept(now, form)
        out.update(pos=frame[0], vel=frame[1], force=frame[2], thermo=_kept(state["thermo"], form))
        return out
    if case["kind"] == "batch":
        v = _views(state["out"], state["n"], state["k"])
        binding.nep_compute_batch([m.h for m in state["models"]], state["req_n"], state["which"], state["box"],
                                  state["pbc"], state["types"], state["pos"], v["energy"], v["virial_total"],
                                  v["site_energy"], v["force"], v["virial"])
        return _views(_kept(state["out"], form), state["n"], state["k"])
    if case["mem"] == "host":
        got = state["model"].compute(state["system"])
        got["energy"] = np.array([got["energy"]])
        return {k: _kept(x, form) for k, x in got.items()}
    v = _views(state["out"], state["n"], 1)
    call = binding.nep_compute if case["mem"] == "device" else binding.nep_compute_static
    call(state["model"].h, state["types"], state["pos"], state["box"], state["pbc"], v["energy"], v["virial_total"],
         v["site_energy"], v["force"], v["virial"])
    return _views(_kept(state["out"], form), state["n"], 1)


# ---- what a pass cannot do without -------------------------------------------------------
# Ordered pairs per particle within the radial and the angular cutoff of these
# configurations (mean, counted on them).
PAIRS = {"water": (76.6, 18.0), "monolayer": (6.0, 5.9), "mixture": (49.0, 29.5)}


def _pairs(system, n):
    if system != "nanowire":
        return PAIRS[system]
    core = min(1.0, 172.0 * max(6, min(196, n // 250)) / n)  # the dense atomistic core's share of the particles
    return 19.2 + 52.4 * core, 6.0 + 22.4 * core


def _flops(system, n, many_body=False):
    """The evaluation's formulas, every ordered pair's terms and gradient once."""
    pr, pa = _pairs(system, n)
    s = SYSTEMS[system]
    T, H, nr, na, k = s["n_types"], s["hidden"], 5, 4, 8
    nd = nr + na * (6 if many_body else 4)
    radial = 13 + 40 + k + 13 + 80 + 2 * k + 24
    angular = 16 + 40 + 2 * na * k + 60 + 48 * na + 16 + 80 + 4 * na * k + 150 + 24 * (4 * na + 10) + 30
    bead = 4 * T * nr * k + 96 * na + H * (4 * nd + 6) + (130 * na if many_body else 0)
    return n * (pr * radial + pa * angular + bead)


def work(case):
    if case["kind"] == "batch":
        # sizes are log-uniform, half of the requests of each system
        n = case["requests"] * (case["n_max"] - 64) / math.log(case["n_max"] / 64)
        return {"bytes": n * (4 + 24 + 13 * 8), "flops": _flops("water", n / 2) + _flops("monolayer", n / 2)}
    n = case["n"]
    once = _flops(case["system"], n, case.get("many_body", False))
    if case["kind"] == "md":  # positions, velocities and forces in and out of every step
        evals = case["steps"] + (1 if case["drive"] else 0)
        return {"bytes": case["steps"] * n * (4 + 6 * 24), "flops": evals * once}
    return {"bytes": n * (4 + 24 + 13 * 8), "flops": once}


# ---- the same in 64 bits, plain torch ------------------------------------------------------
def _neighbours(pos, box, pbc, rc):
    """Ordered pairs (i, j, r_j - r_i) within rc, periodic images included, by cells."""
    dev = pos.device
    n = pos.shape[1]
    box = np.asarray(box, np.float64)
    nc = np.maximum(1, np.floor(box / rc)).astype(int)
    side = box / nc
    reach = [int(math.ceil(rc / side[a] - 1e-12)) if pbc[a] else 1 for a in range(3)]
    c = [torch.clamp((pos[a] / side[a]).floor().long(), 0, int(nc[a]) - 1) for a in range(3)]
    cell = (c[2] * int(nc[1]) + c[1]) * int(nc[0]) + c[0]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=int(nc.prod()))
    first = torch.cumsum(count, 0) - count
    me = torch.arange(n, device=dev)
    found = []
    for dz in range(-reach[2], reach[2] + 1):
        for dy in range(-reach[1], reach[1] + 1):
            for dx in range(-reach[0], reach[0] + 1):
                keep = torch.ones(n, dtype=torch.bool, device=dev)
                at, shift = [], []
                for a, d in enumerate((dx, dy, dz)):
                    x = c[a] + d
                    if not pbc[a]:
                        keep &= (x >= 0) & (x < int(nc[a]))
                    at.append(torch.remainder(x, int(nc[a])))
                    shift.append((x - at[a]).double() / int(nc[a]) * float(box[a]))
                other = (at[2] * int(nc[1]) + at[1]) * int(nc[0]) + at[0]
                many = torch.where(keep, count[other], torch.zeros_like(count[other]))
                i = torch.repeat_interleave(me, many)
                start = torch.cumsum(many, 0) - many
                j = order[first[other[i]] + (torch.arange(i.numel(), device=dev) - start[i])]
                d = torch.stack([pos[a][j] + shift[a][i] - pos[a][i] for a in range(3)])
                r2 = (d * d).sum(0)
                ok = (r2 < rc * rc) & ~((i == j) & (r2 == 0.0))
                found.append((i[ok], j[ok], d[:, ok]))
    i = torch.cat([f[0] for f in found])
    o = torch.argsort(i, stable=True)
    return i[o], torch.cat([f[1] for f in found])[o], torch.cat([f[2] for f in found], dim=1)[:, o]


def _radial_functions(r, rc, coef):
    """g_n(r) of every pair: coef [pairs][n][k] on the Chebyshev basis with its cosine cutoff."""
    x = 2.0 * (r / rc - 1.0) ** 2 - 1.0
    fc = 0.5 + 0.5 * torch.cos(math.pi * r / rc)
    t = [torch.ones_like(x), x]
    for _ in range(coef.shape[2] - 2):
        t.append(2.0 * x * t[-1] - t[-2])
    f = torch.stack([0.5 * (tk + 1.0) * fc for tk in t], dim=1)
    return torch.einsum("pnk,pk->pn", coef, f)


def _harmonics(u):
    """Real orthonormal spherical harmonics of unit vectors u [3][pairs], per l = 1..4."""
    x, y, z = u
    re, im = [torch.ones_like(x)], [torch.zeros_like(x)]  # (x + iy)^m
    for _ in range(4):
        re.append(x * re[-1] - y * im[-1])
        im.append(x * im[len(re) - 2] + y * re[-2])
    out = []
    leg = {}
    for m in range(5):
        leg[m, m] = torch.ones_like(z) * float(np.prod(np.arange(1, 2 * m, 2)))
        if m < 4:
            leg[m + 1, m] = (2 * m + 1) * z * leg[m, m]
        for l in range(m + 2, 5):
            leg[l, m] = ((2 * l - 1) * z * leg[l - 1, m] - (l + m - 1) * leg[l - 2, m]) / (l - m)
    for l in range(1, 5):
        rows = []
        for m in range(l + 1):
            c = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            if m == 0:
                rows.append(c * leg[l, 0])
            else:
                rows += [math.sqrt(2.0) * c * leg[l, m] * re[m], math.sqrt(2.0) * c * leg[l, m] * im[m]]
        out.append(torch.stack(rows, dim=1))
    return out


def _evaluate(p, form, types, pos, box, pbc):
    """Energy, total virial, site energies, forces and per-particle virials of one configuration."""
    dev = pos.device
    n, T = pos.shape[1], p.n_types
    t64 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    w0, b0, w1, b1 = t64(p.w0), t64(p.b0), t64(p.w1), t64(p.b1)
    if form == "bf16":  # the form evaluates the model with W0 rounded to BF16
        w0 = w0.float().bfloat16().double()
    cr, ca = t64(p.c_radial).reshape(T * T, p.n_desc_radial, -1), t64(p.c_angular).reshape(T * T, p.n_desc_angular, -1)
    rcr, rca = t64(p.rc_radial).reshape(-1), t64(p.rc_angular).reshape(-1)
    ii, jj, dd = _neighbours(pos, box, pbc, float(max(p.rc_radial.max(), p.rc_angular.max())))
    U = torch.zeros(n, dtype=torch.float64, device=dev)
    F = torch.zeros(3, n, dtype=torch.float64, device=dev)
    W = torch.zeros(9, n, dtype=torch.float64, device=dev)
    edge = torch.searchsorted(ii, torch.arange(0, n + 1, device=dev))
    step = 1 << 16
    for b in range(0, n, step):
        e = min(n, b + step)
        lo, hi = int(edge[b]), int(edge[e])
        i, j, d = ii[lo:hi], jj[lo:hi], dd[:, lo:hi].clone().requires_grad_(True)
        me = i - b
        pair = types[i] * T + types[j]
        r = (d * d).sum(0).sqrt()
        inR, inA = r < rcr[pair], r < rca[pair]
        zeros = lambda *s: torch.zeros(e - b, *s, dtype=torch.float64, device=dev)  # noqa: E731
        g = _radial_functions(r[inR], rcr[pair[inR]], cr[pair[inR]])
        q = [zeros(p.n_desc_radial).index_add(0, me[inR], g)]
        g = _radial_functions(r[inA], rca[pair[inA]], ca[pair[inA]])
        u = d[:, inA] / r[inA]
        for Y in _harmonics(u):
            A = zeros(p.n_desc_angular, Y.shape[1]).index_add(0, me[inA], g[:, :, None] * Y[:, None, :])
            q.append((A * A).sum(2))
        if p.l_max_4b:
            Q = (u[:, None, :] * u[None, :, :]).permute(2, 0, 1) - torch.eye(3, dtype=torch.float64, device=dev) / 3.0
            M = zeros(p.n_desc_angular, 3, 3).index_add(0, me[inA], g[:, :, None, None] * Q[:, None])
            kappa = -math.sqrt(2.0 / 35.0) * (5.0 / (4.0 * math.pi)) ** 1.5 * 4.5
            q.append(kappa * torch.einsum("bnij,bnjk,bnki->bn", M, M, M))
        if p.l_max_5b:
            q.append(q[1] ** 2)
        q = torch.cat(q, dim=1)
        t = types[b:e]
        x = torch.zeros(e - b, p.hidden, dtype=torch.float64, device=dev)
        for k in range(T):
            x = torch.where((t == k)[:, None], q @ w0[k].T - b0[k], x)
        u_site = (w1[t] * torch.tanh(x)).sum(1) - b1[t]
        f = torch.autograd.grad(u_site.sum(), d)[0]  # dU_i / dr_ij
        U[b:e] = u_site.detach()
        d = d.detach()
        F.index_add_(1, i, f)
        F.index_add_(1, j, -f)
        W.index_add_(1, j, -(d[:, None, :] * f[None, :, :]).reshape(9, -1))
    return U.sum().reshape(1), W.sum(1), U, F, W


def _wrap(x, box, pbc):
    x = x.clone()
    for a in range(3):
        if pbc[a]:
            y = x[a] - float(box[a]) * torch.floor(x[a] / float(box[a]))
            x[a] = torch.where((x[a] >= 0) & (x[a] < float(box[a])), x[a],
                               torch.where((y >= float(box[a])) | (y < 0), torch.zeros_like(y), y))
    return x


def _exact_md(case, seed, dev):
    p = _model(case["system"], seed)
    s, vel, noise = _md_inputs(case, seed)
    dt, steps = SYSTEMS[case["system"]]["dt"], case["steps"]
    types = torch.from_numpy(s.types).long().to(dev)
    mass = torch.from_numpy(np.asarray(s.masses, np.float64)).to(dev)[types]
    fe = torch.tensor(FIELD, dtype=torch.float64, device=dev)

    def forces(x):
        E, Wt, U, F, W = _evaluate(p, case["form"], types, x, s.box, s.pbc)
        if case["drive"]:
            F = F + torch.einsum("a,abn->bn", fe, W.reshape(3, 3, -1)) - (fe @ Wt.reshape(3, 3) / s.n)[:, None]
        return E, Wt, U, F, W

    x, v = torch.from_numpy(s.pos).to(dev), torch.from_numpy(vel).to(dev)
    E, Wt, U, F, W = forces(_wrap(x, s.box, s.pbc))
    heat = torch.zeros(6, dtype=torch.float64, device=dev)
    kinetic = lambda v: float((0.5 * mass * v * v).sum()) / ACC  # noqa: E731
    for k in range(steps):
        v = v + 0.5 * dt * ACC * F / mass
        x = _wrap(x + dt * v, s.box, s.pbc)
        E, Wt, U, F, W = forces(x)
        v = v + 0.5 * dt * ACC * F / mass
        if case["drive"]:  # stochastic velocity rescaling, then the heat current
            c, nf = math.exp(-dt / TAU), 3.0 * s.n - 3.0
            kbar, K, (r1, chi) = 0.5 * nf * KB * TEMPERATURE, kinetic(v), noise[k]
            new = c * K + (1 - c) * kbar / nf * (r1 * r1 + chi) + 2 * r1 * math.sqrt(c * (1 - c) * K * kbar / nf)
            v = v * math.sqrt(max(0.0, new) / K)
            heat[:3] += torch.einsum("abn,bn->a", W.reshape(3, 3, -1), v)
            heat[3:] += ((0.5 * mass * (v * v).sum(0) / ACC + U) * v).sum(1)
    row = torch.tensor([[float(steps), float(E), kinetic(v)] + Wt.tolist()], dtype=torch.float64)
    out = dict(pos=x, vel=v, force=F, thermo=row)
    if case["drive"]:
        out["heat"] = (heat / steps).reshape(1, 6)
    return out


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    names = ("energy", "virial_total", "site_energy", "force", "virial")
    on = lambda s: (torch.from_numpy(s.types).long().to(dev),  # noqa: E731
                    _wrap(torch.from_numpy(np.ascontiguousarray(s.pos)).to(dev), s.box, s.pbc), s.box, s.pbc)
    if case["kind"] == "md":
        return _exact_md(case, seed, dev)
    if case["kind"] == "batch":
        p = [_model("water", seed), _model("monolayer", seed)]
        rows = [_evaluate(p[m], case["form"], *on(s)) for m, s in _requests(case, seed)]
        return {name: torch.cat([r[k].reshape(-1) for r in rows]) for k, name in enumerate(names)}
    got = _evaluate(_model(case["system"], seed, case["many_body"]), case["form"],
                    *on(_system(case["system"], case["n"], seed)))
    if case["mem"] == "host":
        return dict(zip(names, got))
    return {name: g.reshape(-1) for name, g in zip(names, got)}
