"""Timed cases of the adaptive ray-tracing step, through the calls a user's program makes.

A pass of most cases is a run: ``Simulation.reset()``, the run's RT steps and
the snapshot the program keeps (``Simulation.fields``; the library holds these
fields in single precision and a snapshot stores them so).  ``request`` makes
the simulation from host arrays in the pass, as a server that takes requests
one by one does, and ``batch`` admits, steps, reads and retires the members of
a kept ``Batch``.

Kinds of problem (seeded synthetic stand-ins for the workloads of the
repository's configurations, tests and benchmark):

``sphere``  uniform gas and one source (the isothermal Stromgren test and its
            Generalized Opacity form)
``cosmo``   lognormal gas, the sources in the densest cells, temperature
            evolution (the benchmark's workload at several sizes)
``many``    lognormal gas, sources drawn by density, the sub-grid mean free
            path law (the large-box production run, and the members of a batch
            and of a request stream)

``exact`` runs the same problem in plain torch: integer geometry, everything
else in 64 bits.
"""
import math
from types import SimpleNamespace as NS

import numpy as np
import torch

import paper_2409_04521_gb300 as F

EV = 1.602176634e-12
KB = 1.380649e-16
MYR = 3.15576e13
MPC = 3.0856775814913673e24
HUBBLE = 0.68
N_H0 = 0.76 * 0.048 * 1.87847e-29 * HUBBLE ** 2 / 1.67262192e-24   # mean hydrogen density today, cm^-3

# every case has these; a case gives what differs
BASE = dict(kind="cosmo", nx=32, ny=32, nz=32, steps=30, nsrc=16, bins=4, passes=1, gen=False, warm=False,
            merge=False, n_ex=16.0, members=0, how="run")


def _case(**kw):
    return {**BASE, **kw}


def listed():
    return [
        # the smallest run anyone makes: a smoke test's sphere, all launch latency
        _case(name="sphere_16", kind="sphere", nx=16, ny=16, nz=16, steps=6, nsrc=1, bins=1),
        # the Stromgren test at its own size and length
        _case(name="sphere_32", kind="sphere", steps=30, nsrc=1, bins=1),
        # the same sphere with moving screens, five passes a step, evolving temperature
        _case(name="sphere_32_gen", kind="sphere", steps=40, nsrc=1, bins=1, passes=5, gen=True, warm=True),
        # a convergence-test size of the benchmark workload
        _case(name="cosmo_64", nx=64, ny=64, nz=64, steps=60),
        # the benchmark workload, whole
        _case(name="cosmo_128", nx=128, ny=128, nz=128, steps=100),
        # a ragged box with a six-bin spectrum and the Gamma - <n_HI> iteration
        _case(name="ragged_iter", nx=75, ny=50, nz=61, steps=40, nsrc=7, bins=6, passes=3),
        # the large-box run: many sources, sub-grid mean free path
        _case(name="many_200", kind="many", nx=200, ny=200, nz=200, steps=60, nsrc=20000, bins=3),
        # it with ray merging at nearly every step (in gas as opaque as this the rays' brightness ranks
        # hardly ever tie; where it is transparent, rounding decides them, and two runs part)
        _case(name="many_200_merge", kind="many", nx=200, ny=200, nz=200, steps=40, nsrc=20000, bins=3,
              merge=True, n_ex=0.25),
        # it in Generalized Opacity mode
        _case(name="many_200_gen", kind="many", nx=200, ny=200, nz=200, steps=25, nsrc=20000, bins=3, passes=4,
              gen=True),
        # one served request from host arrays to host fields
        _case(name="request_96", kind="many", nx=96, ny=96, nz=96, steps=60, nsrc=12, bins=3, how="request"),
        # uneven members advanced together, host arrays to host fields
        _case(name="batch_16", kind="many", nx=96, ny=96, nz=96, steps=50, nsrc=16, bins=3, members=16, how="batch"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["sphere", "sphere_gen", "cosmo", "cosmo", "merge", "iter", "many", "many_gen", "request",
                       "batch"])
    n = _log_int(rng, 16, 120)
    edge = [n] * 3 if rng.random() < 0.5 else [max(8, int(n * rng.uniform(0.6, 1.2))) for _ in range(3)]
    c = _case(nx=edge[0], ny=edge[1], nz=edge[2], nsrc=_log_int(rng, 1, 32), bins=rng.choice([1, 2, 3, 4, 4, 5, 8]),
              steps=rng.randint(6, 80))
    if what in ("sphere", "sphere_gen"):
        n = rng.randint(12, 72)
        c.update(kind="sphere", nx=n, ny=n, nz=n, nsrc=1, bins=rng.choice([1, 1, 3]))
        if what == "sphere_gen":
            c.update(gen=True, passes=rng.randint(5, 7), warm=rng.random() < 0.5, steps=rng.randint(6, 50))
    elif what == "iter":
        c.update(passes=rng.randint(2, 4), steps=rng.randint(6, 40))
    elif what in ("many", "many_gen", "merge"):
        n = _log_int(rng, 24, 200)
        edge = [n] * 3 if rng.random() < 0.5 else [max(8, int(n * rng.uniform(0.6, 1.0))) for _ in range(3)]
        c.update(kind="many", nx=edge[0], ny=edge[1], nz=edge[2], bins=rng.choice([1, 3, 3, 4]),
                 nsrc=_log_int(rng, 20, max(40, edge[0] * edge[1] * edge[2] // 400)), steps=rng.randint(6, 60))
        if what == "many_gen":
            c.update(gen=True, passes=rng.randint(4, 5), steps=rng.randint(6, 25))
        elif what == "merge":
            c.update(merge=True, n_ex=rng.choice([0.1, 0.25, 0.5]), nsrc=max(20, edge[0] * edge[1] * edge[2] // 400))
    elif what == "request":
        c.update(kind="many", bins=3, how="request")
    elif what == "batch":
        n = _log_int(rng, 32, 96)
        c.update(kind="many", nx=n, ny=n, nz=n, bins=3, members=rng.randint(2, 16), how="batch",
                 steps=rng.randint(6, 50))
    while work(c)["flops"] > 1e12:                    # the benchmark workload's
        c["steps"] = max(4, c["steps"] * 3 // 4)
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _lognormal(shape, sigma, seed):
    """exp of a Gaussian field of power spectrum k^-2, mean 1, x fastest."""
    g = torch.Generator("cuda").manual_seed(seed)
    w = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))
    k2 = (torch.fft.fftfreq(shape[0], device="cuda", dtype=torch.float64)[:, None, None] ** 2
          + torch.fft.fftfreq(shape[1], device="cuda", dtype=torch.float64)[None, :, None] ** 2
          + torch.fft.rfftfreq(shape[2], device="cuda", dtype=torch.float64)[None, None, :] ** 2)
    f = torch.fft.irfftn(torch.where(k2 > 0, w / k2.clamp_min(1e-30).sqrt(), torch.zeros_like(w)), s=shape)
    f = (f - f.mean()) / f.std() * sigma
    return torch.exp(f - 0.5 * sigma * sigma).reshape(-1).cpu().numpy()


def _blackbody(T, nb, slope=2.75):
    """nb equal logarithmic bins of a blackbody over 13.6 .. 54.4 eV."""
    edges = 13.6 * 4.0 ** (np.arange(nb + 1) / nb)
    frac, sig, heat = [], [], []
    for lo, hi in zip(edges[:-1], edges[1:]):
        E = np.linspace(lo, hi, 2001)
        n = E * E / np.expm1(E / (8.617333262e-5 * T))
        s = 6.3e-18 * (E / 13.6) ** -slope * n
        frac.append(np.trapezoid(n, E))
        sig.append(np.trapezoid(s, E) / frac[-1])
        heat.append(np.trapezoid(s * (E - 13.6), E) / np.trapezoid(s, E) * EV)
    frac = np.array(frac) / np.sum(frac)
    return NS(nbins=nb, frac=frac, sigma_cm2=np.array(sig), eheat_erg=np.array(heat))


def _problem(c, seed):
    kind, grid = c["kind"], (c["nx"], c["ny"], c["nz"])
    ncell = grid[0] * grid[1] * grid[2]
    rng = np.random.default_rng(seed)
    opt = NS(l_src=0, l_max=12, n_ray_min=3.0, eps_term=1e-10, seed=int(seed) % (1 << 31) + 1, rotate=True,
             isothermal=kind != "cosmo" and not c["warm"], rates=0 if kind == "sphere" else 1, chem_iters=5,
             alpha_B_const=2.59e-13, x_init=1.2e-3, T_init=100.0 if kind == "cosmo" or c["warm"] else 1e4,
             merge=c["merge"], l_merge=0, n_ex=c["n_ex"], gamma_iters=c["passes"], gen_mode=c["gen"], chi=0.0,
             t_reion=2e4, alpha_pl=1.5)
    mfp = NS(mode=0, lambda0_cm_comoving=0.0, delta_exp=1.0, gamma_ref=1e-12, gamma_exp=2.0 / 3.0,
             gamma_floor=1e-15, xion_threshold=0.5, nH_mean=0.0)
    if kind == "sphere":
        z, dt = 0.0, 1.0 * MYR
        box = 12e-3 * MPC * grid[0] / 32.0
        nH = np.full(ncell, 1e-3 * math.exp(0.2 * rng.standard_normal()))
        cells = np.array([[g // 2 for g in grid]], np.int32)
        ndot = np.array([3e48 * math.exp(0.2 * rng.standard_normal())])
        if c["bins"] == 1:
            spec = NS(nbins=1, frac=np.ones(1), sigma_cm2=np.array([6.3e-18]), eheat_erg=np.zeros(1))
        else:
            spec = _blackbody(1e5, c["bins"])
        if c["gen"]:
            mfp.mode = 3
    elif kind == "cosmo":
        z, dt = 9.0, 0.1 * MYR
        box = 0.5 * MPC / HUBBLE * grid[0] / 128.0
        delta = _lognormal(grid[::-1], 1.0, seed)
        nH = N_H0 * (1 + z) ** 3 * delta
        lin = np.argsort(-delta, kind="stable")[:c["nsrc"]]
        ndot = 10.0 ** rng.uniform(51.0, 52.0, c["nsrc"])
        spec = _blackbody(1e5, c["bins"])
    else:
        z, dt = 7.0, 1.0 * MYR
        box = MPC / HUBBLE * grid[0]
        delta = _lognormal(grid[::-1], 0.6 if c["how"] == "run" else rng.uniform(0.3, 1.2), seed)
        nbar = N_H0 * (1 + z) ** 3
        nH = nbar * delta
        cum = np.cumsum(delta)
        lin = np.searchsorted(cum, rng.random(c["nsrc"]) * cum[-1]).clip(0, ncell - 1)
        ndot = np.exp(rng.normal(math.log(1e53), 1.0, c["nsrc"]))
        spec = _blackbody(1e5, c["bins"])
        mfp.mode, mfp.nH_mean = 2, nbar
        mfp.lambda0_cm_comoving = 5.0 * MPC if c["how"] == "run" else rng.uniform(1.0, 20.0) * box / grid[0]
    if kind != "sphere":
        lin = np.asarray(lin, np.int64)
        cells = np.stack([lin % grid[0], lin // grid[0] % grid[1], lin // (grid[0] * grid[1])], 1).astype(np.int32)
    return NS(grid=grid, box_cm_comoving=box, redshift=z, nH=nH, spectrum=spec, mfp=mfp, options=opt,
              source_cells=cells, source_ndot=ndot, dt=dt, nsteps=c["steps"])


def _problems(c, seed):
    return [_problem(q, seed + 1000 * k) for k, q in enumerate(_members(c))]


def _capacity(c):
    """Ray capacity a program that knows its run asks for: the shells of every
    source inside the box and the ionised region, with room to spare."""
    shells = _shells(c)
    live = c["nsrc"] * sum(r for r, first in shells if first <= c["steps"])
    return int(min(max(4 * live, 24 * c["nx"] * c["ny"] * c["nz"], 1 << 22), 400_000_000))


# --------------------------------------------------------------------------
# passes
# --------------------------------------------------------------------------
def _which(p):
    return ("gamma_HI", "x_HII") + (() if p.options.isothermal else ("T",))


def _snapshot(f):
    return {k: v.astype(np.float32) for k, v in f.items()}


def prepare(case, seed):
    c = {**BASE, **case}
    probs = _problems(c, seed)
    st = NS(case=c, probs=probs, sim=None, batch=None)
    if c["how"] == "run":
        st.sim = F.Simulation(probs[0], ray_capacity=_capacity(c))
    elif c["how"] == "batch":
        st.batch = F.Batch(max_sims=len(probs), max_grid=max(max(p.grid) for p in probs), nbins=c["bins"],
                           ray_capacity=sum(_capacity(q) for q in _members(c)),
                           cell_capacity=sum(p.nH.size for p in probs),
                           emitter_capacity=sum(len(p.source_ndot) for p in probs) + 64)
    return st


def run(st):
    c, p = st.case, st.probs[0]
    if c["how"] == "run":
        st.sim.reset()
        for _ in range(p.nsteps):
            st.sim.step(p.dt)
        st.sim.sync()                                 # raises if a step failed
        return _snapshot(st.sim.fields(_which(p)))
    if c["how"] == "request":
        s = F.Simulation(p, ray_capacity=max(1 << 20, 64 * p.nH.size))
        for _ in range(p.nsteps):
            s.step(p.dt)
        s.sync()
        out = _snapshot(s.fields(_which(p)))
        s.close()
        return out
    B = st.batch
    slots = [B.add(q) for q in st.probs]
    for _ in range(p.nsteps):
        B.step()
    B.sync()
    out = [_snapshot(B.fields(s, _which(q))) for s, q in zip(slots, st.probs)]
    for s in slots:
        B.retire(s)
    B.step()                                          # lets the members' slots and emitters be used again
    B.sync()
    return out


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _shells(c):
    """For each age in cells, a source's rays of that age inside the box, and
    the step from which the ionised region (and the front's width) holds them."""
    n = np.array([c["nx"], c["ny"], c["nz"]], float)
    i = np.arange(128) + 0.5
    mu, ph = 1 - 2 * i / 128, math.pi * (1 + 5 ** 0.5) * i
    u = np.abs(np.stack([np.sqrt(1 - mu * mu) * np.cos(ph), np.sqrt(1 - mu * mu) * np.sin(ph), mu], 1))
    if c["kind"] == "sphere":
        per_step, width = 3e48 * MYR / (1e-3 * (12e-3 * MPC / 32) ** 3), 3      # cells a source ionises in a step
    elif c["kind"] == "cosmo":
        per_step, width = 10 ** 51.5 * 0.1 * MYR / (N_H0 * (0.5 * MPC / HUBBLE / 128) ** 3), 5
    else:
        per_step, width = 1.6e53 * MYR / (N_H0 * (MPC / HUBBLE) ** 3), 1
    if c["gen"]:
        width = 0                                                               # screens stop the rays
    out = []
    for a in range(c["steps"]):
        level = sum(1 for k in range(12) if a >= math.ceil(2.0 ** k * math.sqrt(1 / math.pi)))
        if c["kind"] == "sphere":
            inside = float(np.mean(np.all(a * u < n / 2, 1)))
        else:
            inside = float(np.mean(np.prod(np.clip(1 - a * u / n, 0, 1), 1)))
        out.append((12 * 4.0 ** level * inside, max(a, 4.2 * max(a - width, 0) ** 3 / per_step)))
    return out


def _ray_steps(c):
    """Rays marched in a run, from geometry."""
    return c["nsrc"] * c["passes"] * sum(r * max(0.0, c["steps"] - first) for r, first in _shells(c))


def _members(c):
    if c["how"] != "batch":
        return [c]
    out = []
    for k in range(c["members"]):                    # uneven members, a third to the whole edge
        n = max(8, c["nx"] * (k % 3 + 1) // 3)
        out.append({**c, "nx": n, "ny": n, "nz": n, "nsrc": 1 + (5 * k) % c["nsrc"]})
    return out


def work(case):
    c = {**BASE, **case}
    by = fl = 0.0
    for q in _members(c):
        rays, cells = _ray_steps(q), q["nx"] * q["ny"] * q["nz"] * q["steps"] * q["passes"]
        if q["merge"]:
            rays = min(rays, (q["n_ex"] + 1.0) * cells)                      # what merging leaves, about
        # a ray's record in, its photons out; a cell's state, opacity and deposits in and out
        by += rays * (24 + 8 * q["bins"]) + cells * 76.0
        # 2.5 crossed cells a ray, some 20 operations a bin; some 200 a cell
        fl += rays * (150 + 50 * q["bins"]) + cells * 200.0
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------
# the same run in 64 bits
# --------------------------------------------------------------------------
ONE = 1 << 21
GOLD = np.uint64(0x9E3779B97F4A7C15)


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _rotations(seed, ne, step):
    """One uniform rotation per emitter, rounded to 2^-24 (int64 [ne, 9])."""
    with np.errstate(over="ignore"):
        h = _mix(np.full(ne, seed, np.uint64) + GOLD)
        h = _mix(h + GOLD * (np.arange(ne, dtype=np.uint64) + np.uint64(1)))
        h = _mix(h + GOLD * np.uint64(step + 1))
        q = np.tile(np.array([[1, 0, 0, 0]], np.int64), (ne, 1))
        todo = np.arange(ne)
        for t in range(64):
            if not len(todo):
                break
            v = _mix(h[todo] + GOLD * np.uint64(t + 1))
            d = np.stack([((v >> np.uint64(16 * k)) & np.uint64(0xFFFF)).astype(np.int64) - 32768 for k in range(4)], 1)
            n2 = (d * d).sum(1)
            ok = (n2 > 0) & (n2 <= 1 << 30)
            q[todo[ok]] = d[ok]
            todo = todo[~ok]
    w, x, y, z = q.T
    n = w * w + x * x + y * y + z * z
    m = np.stack([w * w + x * x - y * y - z * z, 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), w * w - x * x + y * y - z * z, 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), w * w - x * x - y * y + z * z], 1) << 24
    f, r = np.divmod(m, n[:, None])
    return f + ((2 * r > n[:, None]) | ((2 * r == n[:, None]) & (f & 1 == 1)))


def _pixel_vectors(level, p):
    """Centres of NESTED HEALPix pixels in units of 2^-24 (int64 [n, 3])."""
    ns = (torch.ones_like(p) << level)
    face, ipf = p // (ns * ns), p % (ns * ns)
    ix, iy = torch.zeros_like(p), torch.zeros_like(p)
    for b in range(13):
        ix |= ((ipf >> (2 * b)) & 1) << b
        iy |= ((ipf >> (2 * b + 1)) & 1) << b
    jr0 = torch.tensor([2] * 4 + [3] * 4 + [4] * 4, device=p.device)
    jp0 = torch.tensor([1, 3, 5, 7, 0, 2, 4, 6, 1, 3, 5, 7], device=p.device)
    jr = jr0[face] * ns - ix - iy - 1
    north, south = jr < ns, jr > 3 * ns
    nr = torch.where(north, jr, torch.where(south, 4 * ns - jr, ns))
    cap = (nr * nr).double() / (3 * ns * ns).double()
    z = torch.where(north, 1 - cap, torch.where(south, cap - 1, (2 * (2 * ns - jr)).double() / (3 * ns).double()))
    sh = torch.where(north | south, torch.zeros_like(jr), (jr - ns) & 1)
    jp = torch.div(jp0[face] * nr + ix - iy + 1 + sh, 2, rounding_mode="trunc")
    jp = torch.where(jp > 4 * ns, jp - 4 * ns, jp)
    jp = torch.where(jp < 1, jp + 4 * ns, jp)
    phi = math.pi * (2 * jp - sh - 1).double() / (4 * nr).double()
    st = ((1 - z) * (1 + z)).sqrt()
    return torch.round(torch.stack([st * phi.cos(), st * phi.sin(), z], 1) * 16777216.0).long()


def _directions(level, pix, R):
    v = _pixel_vectors(level, pix)
    X = (R.view(-1, 3, 3) * v[:, None, :]).sum(2)
    q = X >> 27
    r = X - (q << 27)
    return q + ((r > 1 << 26) | ((r == 1 << 26) & (q & 1 == 1))).long()


def _alpha_b(T):
    lam = 315614.0 / T
    return 2.753e-14 * lam ** 1.5 / (1 + (lam / 2.740) ** 0.407) ** 2.242


def _alpha_a(T):
    lam = 315614.0 / T
    return 1.269e-13 * lam ** 1.503 / (1 + (lam / 0.522) ** 0.470) ** 1.923


def _collisions(T):
    lam = 315614.0 / T
    return 21.11 * T ** -1.5 * torch.exp(-lam / 2) * lam ** -1.089 / (1 + (lam / 0.354) ** 0.874) ** 1.101


def _cooling(T, ne, nHI, nHII, z):
    lam = 315614.0 / T
    rec = 3.435e-30 * T * lam ** 1.970 / (1 + (lam / 2.250) ** 0.376) ** 3.720
    line = 13.6 * EV * _collisions(T) + 7.5e-19 * torch.exp(-118348.0 / T) / (1 + (T / 1e5).sqrt())
    ff = 1.42e-27 * (1.1 + 0.34 * torch.exp(-(5.5 - T.log10()) ** 2 / 3)) * T.sqrt()
    Tc = 2.7255 * (1 + z)
    comp = 4 * KB * 6.6524587e-25 * 7.5657e-15 * Tc ** 4 / (9.1093837e-28 * 2.99792458e10)
    return (rec + ff) * ne * nHII + line * ne * nHI + comp * (T - Tc) * ne


def _substeps(T, dt, rate, linear):
    """Sub-steps of at most 5% of T over dt: explicit, or (linear) the
    two-stage Rosenbrock scheme; rate(T, index of the cells)."""
    T = T.clone()
    at = torch.arange(T.numel(), device=T.device)
    left = torch.full_like(T, dt)
    g = 1 + 1 / math.sqrt(2)
    for k in range(1000):
        if not at.numel():
            break
        t = T[at]
        f = rate(t, at)
        h = left[at]
        if k < 999:
            h = torch.where(f != 0, torch.minimum(h, 0.05 * t / f.abs()), h)
        if linear:
            J = ((rate(t * 1.001, at) - f) / (0.001 * t)).clamp_max(0)
            w = 1 / (1 - g * h * J)
            k1 = w * f
            step = h * (1.5 * k1 + 0.5 * w * (rate(t + h * k1, at) - 2 * k1))
        else:
            step = f * h
        T[at] = t + step
        left[at] -= h
        at = at[left[at] > 0]
    return T


class _Exact:
    """One problem's run with 64-bit arithmetic (integers for the geometry)."""

    def __init__(self, p):
        self.p, o, m = p, p.options, p.mfp
        dev = dict(device="cuda", dtype=torch.float64)
        self.nH = torch.tensor(p.nH, **dev)
        n = self.nH.numel()
        self.dx = p.box_cm_comoving / p.grid[0] / (1 + p.redshift)
        self.gen = bool(o.gen_mode)
        self.y = torch.full((n,), 1.0 if self.gen else 1 - o.x_init, **dev)
        self.T = torch.full((n,), o.T_init, **dev)
        self.G = torch.zeros(n, **dev)
        self.xion, self.yion, self.rho = torch.zeros(n, **dev), torch.zeros(n, **dev), torch.ones(n, **dev)
        self.delta = self.nH / (m.nH_mean if m.nH_mean > 0 else self.nH.mean())
        self.ks = self.sub(self.y, self.G)
        self.sig = torch.tensor(p.spectrum.sigma_cm2, **dev)
        self.eh = torch.tensor(p.spectrum.eheat_erg, **dev)
        self.K = [max(1, math.ceil(2.0 ** l * math.sqrt(3 / (math.pi * o.n_ray_min)))) for l in range(13)]
        cells, rates = {}, []
        for ijk, q in zip(map(tuple, p.source_cells.tolist()), p.source_ndot):      # one emitter per cell
            if ijk in cells:
                rates[cells[ijk]] += q
            else:
                cells[ijk] = len(rates)
                rates.append(q)
        self.ec = torch.tensor(list(cells), device="cuda", dtype=torch.int64).reshape(-1, 3)
        self.nd = torch.tensor(rates, **dev)
        self.rot = []
        nb = p.spectrum.nbins
        z = torch.zeros(0, device="cuda", dtype=torch.int64)
        self.rays = (z, z, z, z, z.reshape(0, 3), torch.zeros(0, nb, **dev))
        self.step_no = 0

    def sub(self, y, G):
        """The sub-grid opacity 1/lambda, per cm."""
        m, z1 = self.p.mfp, 1 + self.p.redshift
        if m.mode != 2:
            return torch.full_like(y, z1 / m.lambda0_cm_comoving if m.mode == 1 else 0.0)
        lam = m.lambda0_cm_comoving * self.delta ** -m.delta_exp * (G.clamp_min(m.gamma_floor) / m.gamma_ref) ** m.gamma_exp
        on = G > 0 if self.gen else 1 - y >= m.xion_threshold
        return torch.where(on, z1 / lam, torch.zeros_like(y))

    def ion_y(self, G):
        o, m = self.p.options, self.p.mfp
        if m.mode != 3:
            return torch.zeros_like(G)
        alpha = _alpha_b(self.T) if o.rates else o.alpha_B_const
        y = (alpha * (1 + o.chi) * self.nH / G.clamp_min(m.gamma_floor)).clamp_max(1)
        return torch.where(G > 0, y, torch.zeros_like(y))

    def march(self, y, ks, keep):
        n = self.nH.numel()
        dep = [torch.zeros(n, device="cuda", dtype=torch.float64) for _ in range(5)]
        out = []
        total = self.rays[0].numel()
        for i in range(0, total, 1 << 23):
            got = self.chunk([r[i:i + (1 << 23)] for r in self.rays], y, ks, dep, keep)
            if keep:
                out.append(got)
        if keep and out:
            self.rays = tuple(torch.cat([o[k] for o in out]) for k in range(6))
        return dep

    def chunk(self, rays, y, ks, dep, keep):
        lev, pix, em, birth, d, N = rays
        N = N.clone()
        p, o, s = self.p, self.p.options, self.step_no
        nx, ny, nz = p.grid
        ng = torch.tensor(p.grid, device="cuda")
        age = s - birth
        p0 = (2 * self.ec[em] + 1) * (ONE // 2) + age[:, None] * d
        a, sg = d.abs(), d.sign()
        cell = torch.where(d < 0, p0 - 1, p0) >> 21
        D = torch.where(d < 0, p0 - (cell << 21), ((cell + 1) << 21) - p0)
        cross = (sg != 0) & (D < a)
        rank = torch.zeros_like(D)
        for u in range(3):
            for v in range(3):
                if u != v:
                    rank[:, u] += cross[:, v] & (D[:, v] * a[:, u] < D[:, u] * a[:, v])
        inside = ((cell >= 0) & (cell < ng)).all(1)
        tn, td = torch.zeros_like(age), torch.ones_like(age)
        last = torch.zeros_like(age)
        stopped = torch.zeros_like(inside)
        ion, heat, absd, front, fall = dep
        lastk = torch.zeros_like(N)
        for r in range(4):
            hit = cross & (rank == r)
            if r < 3:
                use = inside & hit.any(1)
                first = hit.long().argmax(1, keepdim=True)
                un, ud = D.gather(1, first)[:, 0], a.gather(1, first)[:, 0]
            else:
                use, un, ud = inside, torch.ones_like(age), torch.ones_like(age)
            w = (use & ~stopped).nonzero()[:, 0]
            ds = (un[w] * td[w] - tn[w] * ud[w]).double() / (ud[w] * td[w]).double() * self.dx
            c = cell[w]
            k = (c[:, 2] * ny + c[:, 1]) * nx + c[:, 0]
            if self.gen:
                ds = ds * self.xion[k]
            kap = (self.nH[k] * y[k])[:, None] * self.sig + ks[k][:, None]
            tau = kap * ds[:, None]
            n0 = N[w]
            ab = -n0 * torch.expm1(-tau)
            io = self.sig * torch.where(kap > 0, ab / kap, n0 * ds[:, None])
            ion.index_add_(0, k, io.sum(1))
            heat.index_add_(0, k, (io * self.eh).sum(1))
            absd.index_add_(0, k, ab.sum(1))
            n0 = n0 * torch.exp(-tau)
            if self.gen:
                part = self.xion[k] < 1
                nf = torch.where(part, n0.sum(1), torch.zeros_like(ds))
                fall.index_add_(0, k, nf)
                front.index_add_(0, k, self.rho[k] * nf)
                n0 = torch.where(part[:, None], n0 * (1 - self.rho[k])[:, None], n0)
                stopped[w] |= part & (self.rho[k] >= 1)
            N[w] = n0
            last[w] = k
            lastk[w] = kap
            if r < 3:
                cell = torch.where(hit & use[:, None], cell + sg, cell)
                tn, td = torch.where(use, un, tn), torch.where(use, ud, td)
                inside &= ((cell >= 0) & (cell < ng)).all(1)
        live = inside & ~stopped
        thr = o.eps_term * self.nd[em] * p.dt / (12 * 4 ** o.l_src) * 0.25 ** (lev - o.l_src).double()
        end = (live & (N.sum(1) < thr)).nonzero()[:, 0]
        q = torch.where(lastk[end] > 0, self.sig * N[end] / lastk[end], torch.zeros_like(N[end]))
        ion.index_add_(0, last[end], q.sum(1))
        heat.index_add_(0, last[end], (q * self.eh).sum(1))
        absd.index_add_(0, last[end], N[end].sum(1))
        if not keep:
            return None
        live[end] = False
        lev, pix, em, birth, d, N, age = (t[live] for t in (lev, pix, em, birth, d, N, age))
        while True:
            K = torch.tensor(self.K, device="cuda")
            sp = (lev < o.l_max) & (age + 1 >= K[lev.clamp_max(12)])
            if not bool(sp.any()):
                return lev, pix, em, birth, d, N
            cl, ce, cb, ca = (t[sp].repeat_interleave(4) for t in (lev + 1, em, birth, age))
            cp = (4 * pix[sp][:, None] + torch.arange(4, device="cuda")).reshape(-1)
            cd = _directions(cl, cp, self.rots[cb, ce])
            cn = (N[sp] / 4).repeat_interleave(4, 0)
            lev, pix, em, birth, d, N, age = (torch.cat([t[~sp], u]) for t, u in zip(
                (lev, pix, em, birth, d, N, age), (cl, cp, ce, cb, cd, cn, ca)))

    def step(self):
        p, o, s = self.p, self.p.options, self.step_no
        ne = len(self.nd)
        R = torch.tensor(_rotations(o.seed, ne, s), device="cuda")
        self.rot.append(R)
        self.rots = torch.stack(self.rot)
        nc = 12 * 4 ** o.l_src
        pix = torch.arange(nc, device="cuda").repeat(ne)
        em = torch.arange(ne, device="cuda").repeat_interleave(nc)
        lev = torch.full_like(pix, o.l_src)
        new = (lev, pix, em, torch.full_like(pix, s), _directions(lev, pix, R[em]),
               (self.nd[em] * p.dt / nc)[:, None] * torch.tensor(p.spectrum.frac, device="cuda"))
        self.rays = tuple(torch.cat([u, v]) for u, v in zip(self.rays, new))
        y, ks = self.yion if self.gen else self.y, self.ks
        V = self.dx ** 3
        for it in range(o.gamma_iters):
            final = it + 1 == o.gamma_iters
            dep = self.march(y, ks, final)
            y, ks = (self.chem_gen if self.gen else self.chem)(dep, V, final)
        self.step_no += 1

    def chem(self, dep, V, final):
        p, o = self.p, self.p.options
        G, heat = dep[0] / (V * p.dt), dep[1] / (V * p.dt)
        alpha = _alpha_b(self.T) if o.rates else torch.full_like(G, o.alpha_B_const)
        C = _collisions(self.T) if o.rates else torch.zeros_like(G)
        y0 = yb = y1 = self.y
        for _ in range(o.chem_iters):
            ne = self.nH * (1 - yb)
            b = alpha * ne
            sm = G + C * ne + b
            r = p.dt * sm
            eq = b / sm
            y1 = eq + (y0 - eq) * torch.exp(-r)
            yb = eq + (y0 - eq) * -torch.expm1(-r) / r
        if not final:
            return yb, self.sub(yb, G)
        if not o.isothermal:
            H, xb = self.nH * yb * heat, 1 - yb
            n, z = self.nH, p.redshift

            def rate(T, i):
                ne = n[i] * xb[i]
                return 2 / (3 * KB * (n[i] + ne)) * (H[i] - _cooling(T, ne, n[i] * yb[i], ne, z))
            self.T = _substeps(self.T * (2 - y0) / (2 - y1), p.dt, rate, False)
        self.y, self.G = y1, G
        self.ks = self.sub(y1, G)
        return self.y, self.ks

    def chem_gen(self, dep, V, final):
        p, o, x = self.p, self.p.options, self.xion
        ion, _, absd, front, fall = dep
        G = torch.where(x > 0, ion / (x * V * p.dt).clamp_min(1e-300), torch.zeros_like(x))
        A = (1 + o.chi) * self.nH * V
        share = lambda v: torch.where(fall > (1 - v) * A, (1 - v) * A / fall.clamp_min(1e-300), torch.ones_like(v))
        if not final:
            self.rho = share(x)
            return self.ion_y(G), self.sub(self.y, G)
        alpha = _alpha_b(self.T) if o.rates else o.alpha_B_const
        x1 = (x + (front + absd - alpha * (1 + o.chi) * self.nH ** 2 * x * V * p.dt) / A).clamp(0, 1)
        self.rho = share(x1)
        if not o.isothermal:
            yi, n, z = self.ion_y(G), self.nH, p.redshift
            s = o.alpha_pl + 2.75
            e = 13.6 * EV * (s / (s - 1) * (1 - 4 ** (1 - s)) / (1 - 4 ** -s) - 1)

            def rate(T, i):
                nHI, nHII = n[i] * yi[i], n[i] * (1 - yi[i])
                ne = nHII + o.chi * n[i]
                return 2 / (3 * KB * (n[i] * (1 + o.chi) + ne)) * (e * _alpha_a(T) * ne * nHII
                                                                   - _cooling(T, ne, nHI, nHII, z))
            T0 = torch.where(x1 > x, (x * self.T + (x1 - x) * o.t_reion) / x1.clamp_min(1e-300), self.T)
            on = (x1 > 0).nonzero()[:, 0]
            self.T = self.T.clone()
            self.T[on] = _substeps(T0[on], p.dt, lambda T, i: rate(T, on[i]), True)
        self.xion, self.G = x1, G
        self.yion = self.ion_y(G)
        self.ks = self.sub(self.y, G)
        self.y = (1 - x1) + x1 * self.yion
        return self.yion, self.ks

    def fields(self):
        f = {"gamma_HI": self.G, "x_HII": 1 - self.y, "T": self.T}
        return {k: f[k] for k in _which(self.p)}


def exact(case, seed):
    c = {**BASE, **case}
    # which rays merge is decided by their rank in single precision, and the
    # runs part where two decide otherwise: no 64-bit value to hold them to
    if c["merge"] or work(c)["flops"] > 8e11:
        return None
    out = []
    for p in _problems(c, seed):
        e = _Exact(p)
        for _ in range(p.nsteps):
            e.step()
        out.append(e.fields())
    return out if c["how"] == "batch" else out[0]
