"""The workloads that this library's speed is judged by.

A case is a dict of plain values:

* call: the entry point.  "forces" (Context.forces: one mixed force evaluation
  at the current positions), "steps" (Context.step: velocity-Verlet steps from
  a saved state), "host" (Context.step_host: one step with the arrays in host
  memory), "batch" (Batch.step: many cells advanced together), "lists"
  (neighbours_noalloc: neighbour lists and the reverse-slot map alone);
* cell: "si_vacancy" and "fe_vacancy" (periodic defect boxes with a core sphere
  holding the fraction core of the atoms), "si215" and "fe8001" (the small
  silicon vacancy and iron dumbbell cells with their own core radii), "screw"
  (iron cylinder about a screw dislocation, free in x and y), "si_replicas";
* pot: the potential pair, "si" (n 8, lmax 3, body order 3), "fe" (n 10, lmax 4,
  body order 4) or "fe12" (n 12, lmax 5, body order 4);
* precision: "f64", "f32", "bf16", "bf16x3" (arithmetic of the potentials);
* weights: "region" (geometric core) or "rule" (core seeded on the device by
  coordination number), blend: "linear" or "cubic";
* atoms, core, temp (K, initial velocities), steps.

Forces, positions and velocities come back in the type of the case's arithmetic:
float64 where the potentials run in float64, else float32 (what a program that
asked for float potentials hands on: analysis and trajectory files are in
single precision).

exact() evaluates the same mixed forces, and the same steps, in float64 with
plain torch: pair vectors, basis functions and splines written out, forces by
automatic differentiation, the weights blended over the full potentials.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2502_19081_gb300 import inputs as I
from paper_2502_19081_gb300 import mix

PREC = {"f64": mix.MIX_FP64, "f32": mix.MIX_FP32, "bf16": mix.MIX_BF16, "bf16x3": mix.MIX_BF16_SPLIT}
BLEND = {"linear": mix.MIX_BLEND_LINEAR, "cubic": mix.MIX_BLEND_CUBIC}
DT = 1.0            # fs
SKIN = 0.3          # A
KAPPA = 9.6485332e-3
# coordination rule of the silicon vacancy: between the first and second
# shells, atoms with at most three neighbours seed the core
RULE = dict(r_coord=3.0, z_lo=0.0, z_hi=3.0, period=1, r_core=4.0, r_blend=4.5)


def _case(name, call, cell, pot, precision, atoms, core=0.0, temp=0.0, steps=1, weights="region", blend="linear"):
    return {"name": name, "call": call, "cell": cell, "pot": pot, "precision": precision, "atoms": atoms, "core": core,
            "temp": temp, "steps": steps, "weights": weights, "blend": blend}


def listed():
    return [
        # the smallest cell in use, in the reference arithmetic: a force call of a relaxation or a NEB image
        _case("si215_forces_f64", "forces", "si215", "si", "f64", 215),
        # a small defect cell run for its trajectory: launches and latency count
        _case("si1000_steps_f32", "steps", "si_vacancy", "si", "f32", 1000, core=0.05, temp=900.0, steps=10),
        # silicon vacancy seeded by coordination number, cubic blending (the vacancy runs)
        _case("si5831_rule_f32", "steps", "si_vacancy", "si", "f32", 5831, temp=600.0, steps=5, weights="rule",
              blend="cubic"),
        # the iron dumbbell cell: one force call of a caller that integrates by itself
        _case("fe8001_forces_f32", "forces", "fe8001", "fe", "f32", 8001),
        # its checking path
        _case("fe8001_steps_f64", "steps", "fe8001", "fe", "f64", 8001, steps=2),
        # the same cell driven from host memory, a step a call (a host program owns the state)
        _case("fe8001_host_f32", "host", "fe8001", "fe", "f32", 8001, temp=300.0),
        # dislocation glide: the 256,000-atom cylinder with the readout on the tensor cores
        _case("screw256000_steps_bf16", "steps", "screw", "fe12", "bf16", 256000, steps=3),
        # a smaller cylinder in float, where the expensive set is a larger share
        _case("screw40000_forces_f32", "forces", "screw", "fe12", "f32", 40000),
        # the hi/lo split, for potentials that plain bf16 does not serve, in a periodic box
        _case("fe30000_forces_bf16x3", "forces", "fe_vacancy", "fe12", "bf16x3", 29791, core=0.03, temp=300.0),
        # a batch of independent silicon cells of uneven size, stepped together
        _case("si_batch24_f32", "batch", "si_replicas", "si", "f32", 24, steps=3),
        # a large iron request with a small core: the cheap potential carries it
        _case("fe200000_steps_f32", "steps", "fe_vacancy", "fe", "f32", 200000, core=0.01, temp=700.0, steps=2),
        # neighbour lists alone, for a caller that owns all device memory
        _case("lists_fe20000", "lists", "fe_vacancy", "fe", "f64", 20000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["forces", "forces", "steps", "steps", "steps", "host", "batch", "lists"])
    if call == "lists":
        cell = rng.choice(["si_vacancy", "fe_vacancy"])
        return _draw(call, cell, "si" if cell[0] == "s" else "fe", "f64", _log(rng, 700, 30000), 0.0, 300.0, 1)
    if call == "batch":
        precision = rng.choice(["f32", "f32", "f32", "f64"])
        return _draw(call, "si_replicas", "si", precision, _log(rng, 2, 24 if precision == "f32" else 6), 0.0, 0.0,
                     rng.randint(1, 4))
    precision = rng.choice(["f32", "f32", "f32", "f64", "bf16", "bf16x3"])
    cell = rng.choice(["si_vacancy", "si_vacancy", "fe_vacancy", "fe_vacancy", "screw"])
    if precision == "f64":
        cell = rng.choice(["si_vacancy", "fe_vacancy"])
    elif precision[0] == "b" and cell == "si_vacancy":
        cell = "fe_vacancy"
    pot = "si" if cell == "si_vacancy" else ("fe" if precision == "f64" else rng.choice(["fe", "fe12"]))
    atoms = _log(rng, 20000 if cell == "screw" else 700, 12000 if precision == "f64" else 250000)
    # fewer steps where a step is long, so that no case outgrows the largest listed one
    most = 10 if precision != "f64" and cell != "screw" and atoms < 20000 else (4 if atoms < 60000 else 2)
    steps = rng.randint(1, 2 if cell == "screw" or precision == "f64" else most) if call == "steps" else 1
    core = math.exp(rng.uniform(math.log(0.01), math.log(0.1 if atoms < 60000 else 0.04)))
    weights = "rule" if cell == "si_vacancy" and rng.random() < 0.25 else "region"
    return _draw(call, cell, pot, precision, atoms, round(core, 4), float(rng.randint(0, 1200)), steps, weights,
                 rng.choice(["linear", "linear", "cubic"]))


def _draw(call, cell, pot, precision, atoms, core, temp, steps, weights="region", blend="linear"):
    c = _case("", call, cell, pot, precision, atoms, core, temp, steps, weights, blend)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs


@functools.lru_cache(maxsize=None)
def _potentials(pot):
    """The pairs of the silicon vacancy and iron dumbbell cells, and the screw cylinder's recipe."""
    if pot == "fe12":
        return I.element_potentials("Fe", np.random.default_rng(3), 5.5, 12, 5, 4)
    wl = I.si_vacancy() if pot == "si" else I.fe_dumbbell()
    return wl.ace, wl.spline


@functools.lru_cache(maxsize=4)
def _screw_sites(n):
    """The undisplaced cylinder: its box, core cylinder and sites (slow to enumerate, the same for every seed)."""
    return I.fe_screw(n_atoms=n, nrep_z=26 if n >= 20000 else 13, sigma=0.0)


def _workload(case, seed):
    ace, spl = _potentials(case["pot"])
    cell = case["cell"]
    if cell == "si215":
        wl = I.si_vacancy(seed=seed)
    elif cell == "fe8001":
        wl = I.fe_dumbbell(seed=seed)
    elif cell == "screw":
        base = _screw_sites(case["atoms"])
        s = base.system
        rng = np.random.default_rng(seed)
        pos = I.wrap_into_box(s.x[:, :3] + rng.normal(0.0, 0.08, (s.n, 3)), s.box_len, s.periodic)
        x = np.zeros_like(s.x)
        x[:, :3] = pos
        wl = dataclasses.replace(base, system=dataclasses.replace(s, x=x))
    else:
        el = "Si" if cell == "si_vacancy" else "Fe"
        wl = I.serve_request(seed, el, case["atoms"], max(case["core"], 1e-3), case["temp"], {el: (ace, spl)})
    if case["temp"] > 0 and cell in ("fe8001", "screw"):
        v = I.maxwell_boltzmann(np.random.default_rng(seed + 1), wl.system.n, wl.system.mass, case["temp"])
        wl = dataclasses.replace(wl, system=dataclasses.replace(wl.system, v=v))
    return dataclasses.replace(wl, ace=ace, spline=spl, skin=SKIN)


@functools.lru_cache(maxsize=None)
def _replica_plan(count):
    """(target atoms, defect) of the replicas: sizes spread evenly in the logarithm over 1,000 .. 20,000."""
    out = []
    for k in range(count):
        f = (k + 0.5) / count
        out.append((int(round(1000.0 * 20.0 ** f)), "vacancy" if k % 2 == 0 else "interstitial", 300.0 + 1200.0 * ((7 * k) % count) / count))
    return out


def _replicas(case, seed):
    ace, spl = _potentials("si")
    return [I.si_replica(seed * 1009 + k, n, defect, temp, ace, spl)
            for k, (n, defect, temp) in enumerate(_replica_plan(case["atoms"]))]


# ---------------------------------------------------------------------------
# the measured calls


def _open(case, wl):
    ctx = mix.open_context(wl, precision=PREC[case["precision"]], blend=BLEND[case["blend"]])
    if case["weights"] == "rule":
        ctx.set_seed_rule(**RULE)
        ctx.forces()
        ctx.sync()
    return ctx


def _saved(ctxs):
    """Device copies of the trajectories' x, v, f (a checkpoint) and the buffers they go back to."""
    live = [t for c in ctxs for t in (c.x, c.v, c.f)]
    return live, [t.clone() for t in live]


def prepare(case, seed):
    dev = torch.device("cuda:0")
    st = {"case": case, "half": case["precision"] != "f64"}
    if case["call"] == "lists":
        s = _workload(case, seed).system
        rc = _potentials(case["pot"])[0].r_cut
        cap = 64 if case["pot"] == "si" else 128
        n = s.n
        st.update(x=torch.from_numpy(s.x).to(dev), lo=s.box_lo, len=s.box_len, per=s.periodic, rl=rc + SKIN, cap=cap,
                  nnb=torch.zeros(n, dtype=torch.int32, device=dev),
                  nbr=torch.zeros((n, cap), dtype=torch.int32, device=dev),
                  rev=torch.zeros((n, cap), dtype=torch.int32, device=dev))
        return st
    if case["call"] == "batch":
        ctxs = [_open(case, wl) for wl in _replicas(case, seed)]
        st["ctxs"], st["batch"] = ctxs, mix.Batch(ctxs)
        st["live"], st["start"] = _saved(ctxs)
        return st
    ctx = _open(case, _workload(case, seed))
    st["ctx"] = ctx
    if case["call"] == "steps":
        st["live"], st["start"] = _saved([ctx])
    if case["call"] == "host":
        x, v, f, _ = ctx.get_state()
        st["start"] = [x, v, f]
        st["host"] = [torch.from_numpy(a).pin_memory().numpy() for a in (x, v, f)]
    return st


def run(st):
    case = st["case"]
    call = case["call"]
    if call == "forces":
        f = st["ctx"].forces()
        return f.float() if st["half"] else f
    if call == "steps":
        ctx = st["ctx"]
        torch._foreach_copy_(st["live"], st["start"])
        ctx.step(DT, case["steps"])
        out = [ctx.x, ctx.v, ctx.f]
        return [t.float() for t in out] if st["half"] else out
    if call == "host":
        for a, b in zip(st["host"], st["start"]):
            np.copyto(a, b)
        x, v, f = st["host"]
        st["ctx"].step_host(x, v, f, DT, case["steps"])
        return [a.astype(np.float32) for a in (x, v, f)] if st["half"] else [x, v, f]
    if call == "batch":
        torch._foreach_copy_(st["live"], st["start"])
        st["batch"].step(DT, case["steps"])
        out = [torch.cat(st["live"][k::3]) for k in range(3)]
        return [t.float() for t in out] if st["half"] else out
    code = mix.neighbours_noalloc(st["x"], st["lo"], st["len"], st["per"], st["rl"], st["cap"], st["nnb"], st["nbr"],
                                  st["rev"])
    if code != mix.MIX_OK:
        raise mix.MixError(code, "neighbours_noalloc")
    return [st["nnb"], st["nbr"], st["rev"]]


# ---------------------------------------------------------------------------
# what a pass cannot do without

RHO = {"si": 8 / 5.431 ** 3, "fe": 2 / 2.855 ** 3}


def _ball(r):
    return 4.0 / 3.0 * math.pi * max(r, 0.0) ** 3


def _expensive_flops(ace, rho):
    """Multiply-adds (2 each) per evaluated atom: density, nu <= 2 with adjoint, nu = 3 with adjoint, pair gradients."""
    n, nlm, nb = ace.n_rad, (ace.l_max + 1) ** 2, rho * _ball(ace.r_cut)
    fl = 2 * n * nlm * nb + (4 * n * nlm + 8 * nlm) * nb + 4 * n * n * nlm
    if ace.nu_max >= 3:
        for (l1, l2, l3), g in _gaunts(ace.l_max).items():
            nnz, d = int(torch.count_nonzero(g)), 2 * l1 + 1   # l1 is the smallest
            ways = 1 if l1 == l3 else (2 if l1 == l2 or l2 == l3 else 3)
            fl += 4 * d * n ** 3 + 2 * nnz * n * n * ways + 2 * d * n * n
    return fl


def _cheap_flops(spl, rho):
    n3 = rho * _ball(spl.r_cut3)
    return 40 * rho * _ball(spl.r_cut) + 650 * n3 * max(n3 - 1, 0) / 2


def work(case):
    ace, spl = _potentials(case["pot"])
    rho = RHO[case["pot"][:2]]
    rc = max(ace.r_cut, spl.r_cut)
    if case["call"] == "lists":
        n = case["atoms"]
        nb = rho * _ball(rc + SKIN)
        return {"bytes": n * (24 + 4 + 8 * nb), "flops": 8.0 * n * nb / 2}
    sizes = [n for n, _, _ in _replica_plan(case["atoms"])] if case["call"] == "batch" else [case["atoms"]]
    flops = nbytes = 0.0
    for n in sizes:
        ramp = 2.0 if case["pot"] == "si" else 3.0
        if case["weights"] == "rule":
            exp, deep = rho * _ball(2.4 + RULE["r_core"] + RULE["r_blend"]), 0.0
        elif case["cell"] == "screw":
            area, lz = math.pi, (26 if n >= 20000 else 13) * 2.855 * math.sqrt(3.0)
            exp, deep = rho * lz * area * (15.0 + 4.0 + rc) ** 2, rho * lz * area * (15.0 - rc) ** 2
        else:
            r = {"si215": 6.0, "si_replicas": 6.0, "fe8001": 8.0}.get(case["cell"])
            if r is None:
                r = (3.0 * max(case["core"], 1e-3) * n / (4.0 * math.pi * rho)) ** (1.0 / 3.0)
            exp, deep = rho * _ball(r + ramp + rc), rho * _ball(r - rc)
        flops += case["steps"] * (min(exp, n) * _expensive_flops(ace, rho) + max(n - deep, 0) * _cheap_flops(spl, rho))
        # positions in and forces out, and with steps velocities in, positions and velocities out
        nbytes += n * 24 * (2 if case["call"] == "forces" else 6)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same in float64 with plain torch


def _real_y(u, lmax):
    """Real orthonormal spherical harmonics (no Condon-Shortley phase) of unit vectors, index l^2 + l + m."""
    x, y, z = u.unbind(-1)
    c, s = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(lmax):
        c, s = c + [x * c[-1] - y * s[-1]], s + [x * s[-1] + y * c[-1]]
    p = {}
    for m in range(lmax + 1):          # d^m P_l / dz^m
        p[m, m] = torch.full_like(x, float(np.prod(np.arange(1, 2 * m, 2))) if m else 1.0)
        if m < lmax:
            p[m + 1, m] = (2 * m + 1) * z * p[m, m]
        for l in range(m + 2, lmax + 1):
            p[l, m] = ((2 * l - 1) * z * p[l - 1, m] - (l + m - 1) * p[l - 2, m]) / (l - m)
    out = []
    for l in range(lmax + 1):
        for m in range(-l, l + 1):
            k = abs(m)
            nrm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - k) / math.factorial(l + k))
            out.append(nrm * p[l, 0] if m == 0 else math.sqrt(2.0) * nrm * p[l, k] * (c[k] if m > 0 else s[k]))
    return torch.stack(out, -1)


@functools.lru_cache(maxsize=None)
def _gaunts(lmax):
    """{(l1 <= l2 <= l3): integral of Y Y Y over the sphere [m1, m2, m3]} by exact quadrature."""
    deg = 3 * lmax + 2
    t, w = np.polynomial.legendre.leggauss(deg // 2 + 2)
    ph = 2 * math.pi * np.arange(deg + 1) / (deg + 1)
    st = np.sqrt(1 - t * t)[:, None]
    u = np.stack([st * np.cos(ph), st * np.sin(ph), t[:, None] + 0 * ph], -1).reshape(-1, 3)
    wt = torch.from_numpy(np.repeat(w * 2 * math.pi / (deg + 1), deg + 1))
    yv = _real_y(torch.from_numpy(u), lmax)
    out = {}
    for a in range(lmax + 1):
        for b in range(a, lmax + 1):
            for c in range(b, min(a + b, lmax) + 1):
                if (a + b + c) % 2 == 0:
                    ya, yb, yc = (yv[:, l * l:(l + 1) ** 2] for l in (a, b, c))
                    g = torch.einsum("p,pi,pj,pk->ijk", wt, ya, yb, yc)
                    out[a, b, c] = torch.where(g.abs() < 1e-12, torch.zeros_like(g), g)
    return out


def _spline_weights(x, qmax):
    """Interval of a uniform cubic B-spline and the four weights of its control points."""
    q = x.detach().floor().clamp(0, qmax)
    u = x - q
    w = torch.stack([(1 - u) ** 3, 3 * u ** 3 - 6 * u ** 2 + 4, -3 * u ** 3 + 3 * u ** 2 + 3 * u + 1, u ** 3], -1) / 6
    return q.long(), w


def _spline(c, h, r, qmax=12):
    q, w = _spline_weights(r / h, qmax)
    return (c[q.unsqueeze(-1) + torch.arange(4, device=r.device)] * w).sum(-1)


def _ace_energy(a, d, ok):
    """Total energy of sites with pair vectors d [sites, slots, 3] (ok: the slots inside the cutoff)."""
    dev = d.device
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to(dev)  # noqa: E731
    n, lmax = a.n_rad, a.l_max
    far = torch.zeros(3, dtype=d.dtype, device=dev)
    far[2] = 0.5 * a.r_cut
    d = torch.where(ok.unsqueeze(-1), d, far)
    r = d.square().sum(-1).sqrt()
    z = 2 * r / a.r_cut - 1
    cheb = [torch.ones_like(z), z]
    for _ in range(n - 2):
        cheb.append(2 * z * cheb[-1] - cheb[-2])
    rad = torch.stack(cheb[:n], -1) * ((1 - (r / a.r_cut) ** 2) ** 3 * ok).unsqueeze(-1)
    A = _real_y(d / r.unsqueeze(-1), lmax).transpose(1, 2) @ rad          # [sites, lm, n]
    e = 0.5 * (_spline(t(a.pair), a.r_cut / 13, r) * ok).sum() + (A[:, 0] @ t(a.c1)).sum()
    if a.nu_max >= 2:
        for l in range(lmax + 1):
            Al = A[:, l * l:(l + 1) ** 2]
            e = e + ((Al @ t(np.triu(a.c2[l]))) * Al).sum()
    if a.nu_max >= 3:
        for (l1, l2, l3), g in _gaunts(lmax).items():
            w = np.array(a.c3[l1, l2, l3])
            if l1 == l2:
                w = w * (np.arange(n)[:, None] <= np.arange(n)[None, :])[:, :, None]
            if l2 == l3:
                w = w * (np.arange(n)[:, None] <= np.arange(n)[None, :])[None]
            A1, A2, A3 = (A[:, l * l:(l + 1) ** 2] for l in (l1, l2, l3))
            d1, d2, s = 2 * l1 + 1, 2 * l2 + 1, A.shape[0]
            x = g.to(dev).reshape(d1 * d2, -1) @ A3                        # [s, m1 m2, n3]
            x = x.reshape(s, d1, d2, n).permute(0, 2, 1, 3).reshape(s, d2, d1 * n)
            x = A2.transpose(1, 2) @ x                                     # [s, n2, m1 n3]
            x = x.reshape(s, n, d1, n).permute(0, 2, 1, 3).reshape(s, d1, n * n)
            e = e + ((x @ t(w).reshape(n, n * n).T) * A1).sum()
    return e


def _spline_energy(p, d, ok):
    dev = d.device
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to(dev)  # noqa: E731
    far = torch.zeros(3, dtype=d.dtype, device=dev)
    far[2] = 0.5 * p.r_cut
    r = torch.where(ok.unsqueeze(-1), d, far).square().sum(-1).sqrt()
    e = 0.5 * (_spline(t(p.c2), p.r_cut / 13, r) * ok).sum()
    near = ok & (r < p.r_cut3)
    k3 = int(near.sum(1).max()) if near.numel() else 0
    if k3 < 2:
        return e
    order = near.to(torch.int8).argsort(dim=1, descending=True, stable=True)[:, :k3]
    near, r3 = near.gather(1, order), r.gather(1, order)
    d3 = d.gather(1, order.unsqueeze(-1).expand(-1, -1, 3))
    i, j = torch.triu_indices(k3, k3, 1, device=dev)
    pick = (near[:, i] & near[:, j]).nonzero()
    s, i, j = pick[:, 0], i[pick[:, 1]], j[pick[:, 1]]
    rj, rk = r3[s, i], r3[s, j]
    rjk = (d3[s, i] - d3[s, j]).square().sum(-1).sqrt()
    qa, wa = _spline_weights(rj * 5 / p.r_cut3, 4)
    qb, wb = _spline_weights(rk * 5 / p.r_cut3, 4)
    qc, wc = _spline_weights(rjk * 2.5 / p.r_cut3, 4)
    o = torch.arange(4, device=dev)
    at = ((qa[:, None] + o)[:, :, None, None] * 8 + (qb[:, None] + o)[:, None, :, None]) * 8 + (qc[:, None] + o)[:, None, None]
    c = t(p.c3).reshape(-1)[at]
    return e + torch.einsum("tabc,ta,tb,tc->", c, wa, wb, wc)


class _Cell:
    """One system in float64: pairs, weights, mixed forces."""

    def __init__(self, wl, case, dev):
        s = wl.system
        self.wl, self.case, self.dev, self.mass = wl, case, dev, s.mass
        self.lo, self.L = (torch.tensor(np.asarray(v, dtype=np.float64), device=dev) for v in (s.box_lo, s.box_len))
        self.per = torch.tensor([bool(p) for p in s.periodic], device=dev)

    def fold(self, x):
        return torch.where(self.per, x - self.L * (x / self.L).floor(), x)

    def image(self, d):
        return torch.where(self.per, d - self.L * (d / self.L).round(), d)

    def pairs(self, x, rc):
        """[n, slots] partner (-1: none) of every atom, those closer than rc first."""
        n = x.shape[0]
        nc = (self.L / rc).floor().clamp(min=1).long()
        c = ((self.fold(x) - self.lo) / self.L * nc).floor().long().clamp(min=0).minimum(nc - 1)
        cid = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
        order = cid.argsort(stable=True)
        count = torch.bincount(cid, minlength=int(nc.prod()))
        start = count.cumsum(0) - count
        most = torch.arange(int(count.max()), device=self.dev)
        found = []
        me = torch.arange(n, device=self.dev)
        for o in range(27):
            q = c + torch.tensor([o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1], device=self.dev)
            inside = ((q >= 0) & (q < nc) | self.per).all(1)
            q = q % nc
            qid = (q[:, 2] * nc[1] + q[:, 1]) * nc[0] + q[:, 0]
            j = order[(start[qid][:, None] + most).clamp(max=n - 1)]
            d2 = self.image(x[j] - x[:, None]).square().sum(-1)
            ok = (most < count[qid][:, None]) & inside[:, None] & (d2 < rc * rc) & (j != me[:, None])
            i, k = ok.nonzero(as_tuple=True)
            found.append((i, j[i, k]))
        i, j = (torch.cat(v) for v in zip(*found))
        by = i.argsort(stable=True)
        i, j = i[by], j[by]
        num = torch.bincount(i, minlength=n)
        at = torch.arange(i.numel(), device=self.dev) - (num.cumsum(0) - num)[i]
        out = torch.full((n, max(1, int(num.max()) if n else 1)), -1, dtype=torch.long, device=self.dev)
        out[i, at] = j
        return out

    def weights(self, x, nbr):
        if self.case["weights"] == "rule":
            ok = nbr >= 0
            r = self.image(x[nbr.clamp(min=0)] - x[:, None]).square().sum(-1).sqrt()
            z = (ok & (r < RULE["r_coord"])).sum(1)
            seed = (z >= RULE["z_lo"]) & (z <= RULE["z_hi"])
            core = seed | (ok & (r < RULE["r_core"]) & seed[nbr.clamp(min=0)]).any(1)
            by = torch.where(ok & core[nbr.clamp(min=0)] & (r < RULE["r_blend"]), 1 - r / RULE["r_blend"], 0.0)
            lam = torch.where(core, 1.0, by.max(1).values)
        else:
            lam = torch.zeros_like(x[:, 0])
            for g in self.wl.regions:
                d = self.image(x - torch.tensor(g.centre, dtype=x.dtype, device=self.dev))
                d2 = d.square().sum(-1)
                if g.kind == I.REGION_CYLINDER:
                    ax = torch.tensor(g.axis, dtype=x.dtype, device=self.dev)
                    d2 = (d2 - (d @ (ax / ax.norm())) ** 2).clamp(min=0)
                lam = torch.maximum(lam, (1 - (d2.sqrt() - g.r_core) / g.ramp).clamp(0, 1))
        return lam * lam * (3 - 2 * lam) if self.case["blend"] == "cubic" else lam

    def pure(self, energy, rc, x, nbr, need, chunk):
        """Forces of one potential on the atoms `need` (its sites: those and every atom within rc of one)."""
        f = torch.zeros_like(x)
        site = need.clone()
        ok = nbr >= 0
        for b in range(0, x.shape[0], 1 << 17):
            e = slice(b, b + (1 << 17))
            r2 = self.image(x[nbr[e].clamp(min=0)] - x[e, None]).square().sum(-1)
            site[e] |= (ok[e] & need[nbr[e].clamp(min=0)] & (r2 < rc * rc)).any(1)
        for c in site.nonzero().flatten().split(chunk):
            j = nbr[c]
            d = self.image(x[j.clamp(min=0)] - x[c, None])
            inside = (j >= 0) & (d.square().sum(-1) < rc * rc)
            d.requires_grad_(True)
            g, = torch.autograd.grad(energy(d, inside), d)
            g = torch.where(inside.unsqueeze(-1), g, 0.0)
            f.index_add_(0, c, g.sum(1))
            f.index_add_(0, j[inside], -g[inside])
        return f

    def forces(self, x):
        a, p = self.wl.ace, self.wl.spline
        nbr = self.pairs(x, max(a.r_cut, p.r_cut))
        w = self.weights(x, nbr)
        fe = self.pure(lambda d, ok: _ace_energy(a, d, ok), a.r_cut, x, nbr, w > 0, 2000)
        fc = self.pure(lambda d, ok: _spline_energy(p, d, ok), p.r_cut, x, nbr, w < 1, 8000)
        w = w.unsqueeze(-1)
        return torch.where(w > 0, w * fe, 0.0) + torch.where(w < 1, (1 - w) * fc, 0.0)

    def steps(self, x, v, count):
        h = 0.5 * DT * KAPPA / self.mass
        f = self.forces(x)
        built = x
        for _ in range(count):
            v = v + h * f
            x = x + DT * v
            if bool(((x - built).square().sum(1) > (0.5 * SKIN) ** 2).any()):   # lists are rebuilt on folded positions
                x = built = self.fold(x)
            f = self.forces(x)
            v = v + h * f
        return x, v, f


def _rows(a):
    return torch.nn.functional.pad(a, (0, 1))


def exact(case, seed):
    if case["call"] == "lists":
        return None
    dev = torch.device("cuda:0" if torch.cuda.is_available() else "cpu")
    wls = _replicas(case, seed) if case["call"] == "batch" else [_workload(case, seed)]
    count = 0 if case["call"] == "forces" else case["steps"]
    if sum(w.system.n for w in wls) * (count + 1) > 1_200_000:   # longer than some twenty seconds
        return None
    out = []
    for wl in wls:
        cell = _Cell(wl, case, dev)
        x, v = (torch.from_numpy(t[:, :3].copy()).to(dev) for t in (wl.system.x, wl.system.v))
        out.append((cell.forces(x),) if count == 0 else cell.steps(x, v, count))
    got = [_rows(torch.cat(t)) for t in zip(*out)]
    return got[0] if count == 0 else got
