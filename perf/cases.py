"""The work that users of this library have it do, as measurable cases.

A case is one call (or the short chain of calls that always go together) through the public
Python API: the force at the particles, a chained kick-drift-kick run, a binned spectrum, and
the vector-Jacobian products that training and reconstruction use.  Sizes are those of the
repository's own workloads (paper_2007_13394_gb300/workloads.py, the training configuration of
learned.py, the reconstruction test) and odd ones between them.

Inputs are Zel'dovich particles of a seeded Gaussian field with the BBKS spectrum, displaced at
the case's scale factor, so late cases are clustered as evolved particles are.  They are made
with torch alone; only scalars (growth, kick and drift factors, Fermi-Dirac shells) come from
the package's FP64 host tables.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2007_13394_gb300 import inputs, pm, reconstruct, workloads

TWO32 = 2.0 ** 32
H0_C = 2997.92458  # c / (100 km/s), Mpc/h


# ------------------------------------------------------------------ the cases
def _case(kind, box, nmesh, nc, nsites=0, nshell=10, nfib=3, m_nu=0.0, a=1.0, **more):
    c = {"kind": kind, "box": float(box), "nmesh": nmesh, "nc": nc, "nsites": nsites, "nshell": nshell, "nfib": nfib,
         "m_nu": float(m_nu), "a": float(a)}
    c.update(more)
    return c


def listed():
    cases = {
        # the smallest call: one force evaluation of the 64^3-mesh parity run; launches and latency
        "force_64": _case("force", 256, 64, 32, 8, m_nu=0.2, a=0.5),
        # a whole small run (10 steps from z = 99), as quick experiments and tests step through it
        "run_64": _case("run", 256, 64, 32, 8, m_nu=0.2, a=0.01, total=10, first=0, steps=10, learned=False),
        # the force of a ragged selection in random order (a caller's own particle order, with
        # ids): nothing is near-sorted, the counts are odd
        "force_256_shuffled": _case("force", 250, 256, 127, 9, m_nu=0.3, a=0.8, n=1000003),
        # corrected steps at the size the learned factor is evaluated at: force mesh as fine as the
        # CDM grid, two particles a cell
        "run_256_learned": _case("run", 512, 256, 256, 64, m_nu=0.3, a=0.5, total=10, first=7, steps=2, learned=True),
        # the ordinary throughput run: late steps of 256^3 CDM + 32^3 x 70 neutrinos on a 512^3 mesh
        "run_512": _case("run", 512, 512, 256, 32, m_nu=0.1, total=25, first=15, steps=5, learned=False),
        # the scale run at one eighth of its volume: 512^3 CDM + 64^3 x 70 neutrinos, mesh 1024^3
        "run_1024": _case("run", 1024, 1024, 512, 64, m_nu=0.6, total=25, first=20, steps=2, learned=False),
        # the scale run's own mesh (2048^3), one force evaluation on the boost-4 mesh of target runs
        "force_2048": _case("force", 1024, 2048, 512, 64, m_nu=0.6, a=0.7),
        # analysis of a snapshot: cross spectrum of CDM and neutrinos, bins up to the Nyquist mode
        "power_512_cross": _case("power", 512, 512, 256, 32, m_nu=0.1, a=0.9, nbins=256, sa=1, sb=2),
        # the spectrum loss's gradient with respect to the particles
        "power_vjp_256": _case("power_vjp", 256, 256, 128, 16, m_nu=0.1, a=0.9, nbins=128, sa=3),
        # one step of the reconstruction's backward pass at full size
        "step_vjp_256": _case("step_vjp", 256, 256, 128, 16, m_nu=0.2, total=10, first=7, learned=False),
        # one step of the training's backward pass with the learned factor, with its gradient
        "learned_vjp_128": _case("step_vjp", 256, 128, 128, 32, m_nu=0.3, total=10, first=7, learned=True),
        # a whole reconstruction call: ICs, steps and density forward, the gradient of the white noise
        "gradient_64": _case("gradient", 128, 128, 64, 8, m_nu=0.2, a=0.1, steps=3, a1=0.5),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def draw(rng):
    kind = rng.choice(["force", "force", "run", "run", "run", "power", "power_vjp", "step_vjp", "step_vjp", "gradient"])
    top = {"force": 10, "run": 10, "power": 9, "power_vjp": 8, "step_vjp": 8, "gradient": 7}[kind]
    nmesh = 2 ** rng.randint(6, top)
    boost = 2.0 ** rng.uniform(1.0 if nmesh >= 512 else 0.0, 2.0)
    nc = max(16, int(nmesh / boost))
    m_nu = round(rng.uniform(0.06, 0.6), 3)
    nshell, nfib = rng.choice([(10, 3), (10, 3), (4, 1), (7, 2)])
    nsites = rng.choice([0, 1, 1, 1]) * max(1, int(nc / rng.uniform(4.0, 12.0)))
    if kind == "gradient":  # pm_ic's lattice: powers of two, the sites a divisor of the CDM grid
        nc = max(32, nmesh // rng.choice([1, 2]))
        nsites = rng.choice([0, nc // 8, nc // 4])
    if nsites == 0:
        m_nu = 0.0
    c = _case(kind, round(nc * rng.uniform(0.8, 4.0), 1), nmesh, nc, nsites, nshell, nfib, m_nu, round(rng.uniform(0.05, 1.0), 3))
    n = nc ** 3 + nsites ** 3 * nshell * (2 * nfib + 1)
    if kind == "force" and rng.random() < 0.5:
        c["n"] = int(math.exp(rng.uniform(math.log(1000.0), math.log(min(n, 20e6)))))
    if kind == "run":
        c.update(total=rng.choice([10, 25, 40]), steps=rng.randint(1, 2 if nmesh >= 512 else 6),
                 learned=nmesh <= 512 and rng.random() < 0.3)
        c["first"] = rng.randint(0, c["total"] - c["steps"])
    if kind in ("power", "power_vjp"):
        two = kind == "power" and nsites > 0
        c.update(nbins=rng.randint(8, nmesh // 2), sa=rng.choice([1, 3]))
        if kind == "power":
            c["sb"] = rng.choice([1, 2, 3]) if two else c["sa"]
    if kind == "step_vjp":
        c.update(total=rng.choice([10, 25]), learned=rng.random() < 0.4)
        c["first"] = rng.randint(0, c["total"] - 1)
    if kind == "gradient":
        c.update(a=0.1, steps=rng.randint(1, 3), a1=round(rng.uniform(0.3, 0.6), 2))
    return c


# ------------------------------------------------------------------ inputs
def _config(c):
    m = c["m_nu"] / 3.0
    return pm.RunConfig(box=c["box"], nmesh=c["nmesh"], nc=c["nc"], nsites=c["nsites"], nshell=c["nshell"],
                        nfib=c["nfib"], m_nu=(m, m, m))


def _steps(c):
    """The steps of a run or step_vjp case: a slice of the paper's schedule."""
    return workloads.schedule_paper(c["total"])[c["first"]:c["first"] + c.get("steps", 1)]


def _a(c):
    return _steps(c)[0][0] if "total" in c else c["a"]


@functools.lru_cache(maxsize=256)
def _growth(m_nu, a):
    """(D, g_p, g_f) of the default cosmology with neutrinos of total mass m_nu."""
    return pm.cosmo_growth(pm.RunConfig(box=1.0, nmesh=32, nc=0, m_nu=(m_nu / 3.0,) * 3), a)[:3]


@functools.lru_cache(maxsize=32)
def _streaming(m_nu, a):
    """Drift factor of unaccelerated particles from z = 99 to a (sum of Delta over log steps)."""
    edges = [0.01 * (a / 0.01) ** (i / 8.0) for i in range(9)] if a > 0.01 else []
    return sum((_growth(m_nu, y)[0] - _growth(m_nu, x)[0]) / _growth(m_nu, math.sqrt(x * y))[1]
               for x, y in zip(edges, edges[1:]))


def _linear_power(k, cfg):
    """BBKS spectrum normalised to sigma_8 (numpy or torch float64 k > 0, h/Mpc)."""
    def shape(k, log):
        q = k / (cfg.omega_m * cfg.h)
        t = log(1.0 + 2.34 * q) / (2.34 * q) * (1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
        return k ** cfg.ns * t * t
    lk = np.linspace(math.log(1e-5), math.log(1e2), 8192)
    kk = np.exp(lk)
    w = 3.0 * (np.sin(8 * kk) - 8 * kk * np.cos(8 * kk)) / (8 * kk) ** 3
    s2 = np.sum(kk ** 3 * shape(kk, np.log) * w * w) * (lk[1] - lk[0]) / (2.0 * math.pi ** 2)
    return cfg.sigma8 ** 2 / s2 * shape(k, np.log if isinstance(k, np.ndarray) else torch.log)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _noise(nc, seed):
    return torch.randn((nc, nc, nc), generator=_generator(seed), device="cuda")


def _wavenumbers(n):
    """Signed integer wavenumbers of the full axis and of the r2c half axis (float64)."""
    full = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    return full, torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda")


def _displacement(cfg, seed):
    """Zel'dovich displacement at D = 1 on the CDM lattice, a list of three (nc, nc, nc)."""
    nc = cfg.nc
    full, half = _wavenumbers(nc)
    kf = 2.0 * math.pi / cfg.box
    n2 = (full ** 2)[:, None, None] + (full ** 2)[None, :, None] + (half ** 2)[None, None, :]
    n2[0, 0, 0] = 1.0
    amp = (torch.sqrt(_linear_power(torch.sqrt(n2) * kf, cfg) / cfg.box ** 3) * nc ** 1.5 / (n2 * kf)).float()
    del n2
    amp[0, 0, 0] = 0.0
    wk = torch.fft.rfftn(_noise(nc, seed)) * amp
    del amp
    axes = (full[:, None, None], full[None, :, None], half[None, None, :])
    return [torch.fft.irfftn(wk * (1j * k.float()), s=(nc,) * 3) for k in axes]


def _fixed(x, box):
    """Positions (float64, Mpc/h) -> uint32 fixed point, in int32 storage."""
    v = torch.round(x * (TWO32 / box)).to(torch.int64)
    return (((v + 2 ** 31) & 0xffffffff) - 2 ** 31).to(torch.int32)


def _particles(cfg, m_nu, a, seed):
    """Zel'dovich particles at a in canonical order: u (int32 bits), p, f = F of linear theory."""
    D, gp, gf = _growth(m_nu, a)
    nc, ns, ndir = cfg.nc, cfg.nsites, 2 * cfg.nfib + 1
    n, ncdm = cfg.n_particles(), cfg.n_cdm()
    u = torch.empty((3, n), dtype=torch.int32, device="cuda")
    p = torch.empty((3, n), dtype=torch.float32, device="cuda")
    f = torch.empty((3, n), dtype=torch.float32, device="cuda")
    if ns:
        _, q, _ = pm.nu_shells(cfg)
        kT = pm.cosmo_params(cfg)["kT_nu0"]
        i = np.arange(ndir) - cfg.nfib
        lat, lon = np.arcsin(2.0 * i / ndir), 4.0 * math.pi * i / (1.0 + math.sqrt(5.0))
        dirs = np.stack([np.cos(lat) * np.cos(lon), np.cos(lat) * np.sin(lon), np.sin(lat)])
        p_th = q * kT / max(cfg.m_nu) * H0_C
        radius = 0.45 * cfg.box / ns * q / q.max() + p_th * _streaming(m_nu, a)
        node = ((torch.arange(ns, device="cuda") * 2 + 1) * nc // (2 * ns)) % nc
        site = (torch.arange(ns, dtype=torch.float64, device="cuda") + 0.5) * (cfg.box / ns) + 0.5 * cfg.box / nc
    lattice = torch.arange(nc, dtype=torch.float64, device="cuda") * (cfg.box / nc)
    for d, s in enumerate(_displacement(cfg, seed)):
        shape = [-1 if e == d else 1 for e in range(3)]
        u[d, :ncdm] = _fixed(lattice.reshape(shape) + D * s.double(), cfg.box).reshape(-1)
        p[d, :ncdm] = (gp * s).reshape(-1)
        f[d, :ncdm] = (gf * s).reshape(-1)
        if ns:
            sv = s[node][:, node][:, :, node]
            off = torch.from_numpy(radius[:, None] * dirs[d][None, :]).cuda().reshape(-1)
            th = torch.from_numpy(p_th[:, None] * dirs[d][None, :]).cuda().float().reshape(-1)
            x = (site.reshape(shape) + D * sv.double()).reshape(-1)
            u[d, ncdm:] = _fixed(x[:, None] + off[None, :], cfg.box).reshape(-1)
            p[d, ncdm:] = ((gp * sv).reshape(-1)[:, None] + th[None, :]).reshape(-1)
            f[d, ncdm:] = (gf * sv).reshape(-1)[:, None].expand(-1, off.numel()).reshape(-1)
    return u, p, f


def _inputs(c, seed):
    """The tensors a case starts from, made from the seed alone."""
    cfg = _config(c)
    u, p, f = _particles(cfg, c["m_nu"], _a(c), seed)
    t = {"u": u, "p": p, "f": f, "id": torch.arange(u.shape[1], dtype=torch.int32, device="cuda")}
    if c["kind"] == "force" and c.get("n"):
        sel = torch.randperm(u.shape[1], generator=_generator(seed + 1), device="cuda")[:c["n"]]
        t = {"u": u[:, sel].contiguous(), "id": sel.to(torch.int32)}
    if c["kind"] == "force":
        t = {"u": t["u"], "id": t["id"]}
    if c.get("learned"):
        t["theta"] = inputs.mlp_parameters(seed % 1000, last_scale=0.3)
    if c["kind"] == "step_vjp":  # the cotangents that the later steps handed back
        g = _generator(seed + 2)
        t["lx"] = torch.randn(u.shape, generator=g, device="cuda")
        t["lp"] = torch.randn(u.shape, generator=g, device="cuda")
    if c["kind"] == "power_vjp":
        k = (np.arange(c["nbins"]) + 1.0) * 2.0 * math.pi / c["box"]
        r = np.random.default_rng(seed).standard_normal(c["nbins"]) * 0.1
        t["dL_dP"] = 2.0 * r / (_linear_power(k, cfg) * c["nbins"])
    return t


def prepare(case, seed):
    c = dict(case)
    cfg = _config(c)
    s = {"case": c}
    if c["kind"] == "gradient":
        s["steps"] = workloads.schedule_linear(c["a"], c["a1"], c["steps"])
        s["noise"] = _noise(c["nc"], seed).requires_grad_()
        u, _, _ = _particles(cfg, c["m_nu"], c["a1"], seed + 1)  # the target: another seed's density
        s["target"] = _paint64(_cells(u, c["nmesh"]), _masses(c, None, u.shape[1]), c["nmesh"]).float()
        del u
    else:
        s.update(_inputs(c, seed))
    torch.cuda.empty_cache()
    s["pm"] = pm.ParticleMesh(cfg)
    if c.get("learned"):
        s["pm"].set_mlp(s.pop("theta"))
    if c["kind"] in ("run", "step_vjp"):
        s["steps"] = _steps(c)
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    c, ctx, kind = state["case"], state["pm"], state["case"]["kind"]
    if kind == "force":
        return ctx.force(state["u"], state["id"])
    if kind == "run":
        # the run works on a copy (the caller keeps its initial state), and the final state is
        # read back by particle id: displacement since the start, and momentum
        st = {k: state[k].clone() for k in ("u", "p", "id", "f")}
        ctx.run(st, state["steps"])
        order = st["id"].long()
        u, p = torch.empty_like(st["u"]), torch.empty_like(st["p"])
        for d in range(3):
            u[d][order] = st["u"][d]
            p[d][order] = st["p"][d]
        return (u - state["u"]).float() * (c["box"] / TWO32), p
    if kind == "power":
        k, P, modes = ctx.power(state["u"], state["id"], c["sa"], c["sb"], nbins=c["nbins"])
        return k.astype(np.float32), P.astype(np.float32), modes  # spectra of an FP32 mesh
    if kind == "power_vjp":
        return ctx.power_vjp(state["u"], state["id"], state["dL_dP"], c["sa"])
    if kind == "step_vjp":
        lx, lp = ctx.step_vjp(state, *state["steps"][0], state["lx"], state["lp"])
        return (lx, lp, ctx.mlp_grad()) if c["learned"] else (lx, lp)
    rho = reconstruct.final_density(state["noise"], ctx, state["steps"], c["a"])
    loss = ((rho - state["target"]) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, state["noise"])
    return loss.detach(), rho.detach(), grad


def work(case):
    """Bytes and operations of one pass.  A force evaluation writes the mesh once, transforms it
    forward and back (three axes each way, the middle one shared) and reads it once: 48 B a cell;
    particles: 28 B read and written for a bare force, 76 B for a step with both half kicks and
    the drift.  Meshes that stay in the 129 MB second-level cache count no bytes."""
    n3 = float(case["nmesh"]) ** 3
    n = case.get("n") or case["nc"] ** 3 + case["nsites"] ** 3 * case["nshell"] * (2 * case["nfib"] + 1)
    cell = 1.0 if n3 * 4 > 129e6 else 0.0
    fft = 2.5 * n3 * math.log2(n3)
    force = {"bytes": 48.0 * cell * n3 + 28.0 * n, "flops": 2 * fft + 300.0 * n}
    step = {"bytes": 48.0 * cell * n3 + 76.0 * n, "flops": 2 * fft + 300.0 * n}
    kind = case["kind"]
    if kind == "force":
        return force
    if kind == "run":  # the first force, the steps, and the state read back by id
        k = case["steps"]
        return {"bytes": force["bytes"] + k * step["bytes"] + 52.0 * n, "flops": force["flops"] + k * step["flops"]}
    if kind in ("power", "power_vjp"):
        m = 2 if kind == "power_vjp" or case["sb"] != case["sa"] else 1  # transforms
        return {"bytes": m * 28.0 * cell * n3 + (16.0 if kind == "power" else 28.0) * n, "flops": m * fft + 100.0 * n}
    vjp = {"bytes": 2 * (2 * 48.0 * cell * n3) + 88.0 * n, "flops": 2 * (4 * fft + 900.0 * n)}
    if kind == "step_vjp":
        return vjp
    k = case["steps"]
    return {"bytes": k * (step["bytes"] + vjp["bytes"]) + 8 * n3, "flops": k * (step["flops"] + vjp["flops"])}


# ------------------------------------------------------------------ the same in 64 bits
def _cells(u, N):
    """Fixed-point positions (int32 bits) in units of mesh cells, float64."""
    return (u.long() & 0xffffffff).double() * (N / TWO32)


def _masses(c, ids, n):
    """Particle masses in units of the mean mass per mesh cell, float64, by id (None: 0 .. n - 1)."""
    cfg = _config(c)
    om = pm.cosmo_params(cfg)
    oc, on = om["omega_c"] / cfg.omega_m, om["omega_nu"] / cfg.omega_m
    ndir = 2 * cfg.nfib + 1
    i = torch.arange(n, device="cuda") if ids is None else ids.long() & 0xffffffff
    m = torch.full((n,), oc * cfg.nmesh ** 3 / cfg.nc ** 3, dtype=torch.float64, device="cuda")
    if cfg.nsites:
        _, _, ms = pm.nu_shells(cfg)
        tab = torch.from_numpy(on * ms / ndir * cfg.nmesh ** 3 / cfg.nsites ** 3).cuda()
        nu = i >= cfg.n_cdm()
        m[nu] = tab[(i[nu] - cfg.n_cdm()) // ndir % cfg.nshell]
    return m


def _corners(x, N):
    """The eight (flat cell index, CIC weight) of positions x (cells); weights follow x's graph."""
    i = torch.floor(x.detach())
    f = x - i
    i = i.long()
    for corner in range(8):
        b = (corner >> 2 & 1, corner >> 1 & 1, corner & 1)
        w, at = 1.0, 0
        for d in range(3):
            w = w * (f[d] if b[d] else 1.0 - f[d])
            at = at * N + (i[d] + b[d]) % N
        yield at, w


def _paint64(x, mass, N):
    rho = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
    if x.requires_grad:
        for at, w in _corners(x, N):
            rho = rho.index_add(0, at, mass * w)
    else:
        for lo in range(0, x.shape[1], 1 << 23):
            for at, w in _corners(x[:, lo:lo + (1 << 23)], N):
                rho.index_add_(0, at, mass[lo:lo + (1 << 23)] * w)
    return rho.reshape(N, N, N)


def _readout64(x, mesh, N):
    flat = mesh.reshape(-1)
    if x.requires_grad or mesh.requires_grad:
        return sum(w * flat[at] for at, w in _corners(x, N))
    out = torch.empty(x.shape[1], dtype=torch.float64, device="cuda")
    for lo in range(0, x.shape[1], 1 << 23):
        out[lo:lo + (1 << 23)] = sum(w * flat[at] for at, w in _corners(x[:, lo:lo + (1 << 23)], N))
    return out


def _factor64(theta, N, a):
    """1 + MLP(|k| / k_Ny, a) on the half spectrum, through the distinct |n|^2."""
    w1, b1, w2, b2, w3, b3 = torch.split(theta, [128, 64, 4096, 64, 64, 1])
    kap = torch.sqrt(torch.arange(3 * (N // 2) ** 2 + 1, dtype=torch.float64, device="cuda")) / (N // 2)
    z = torch.stack([kap, torch.full_like(kap, a)], dim=1) @ w1.reshape(64, 2).T + b1
    z = torch.nn.functional.silu(z) @ w2.reshape(64, 64).T + b2
    m = 1.0 + torch.nn.functional.silu(z) @ w3 + b3
    full, half = _wavenumbers(N)
    n2 = (full ** 2)[:, None, None] + (full ** 2)[None, :, None] + (half ** 2)[None, None, :]
    return m[n2.long()]


def _force64(x, mass, c, a, theta=None):
    """F (3, n) at positions x (cells): CIC paint, Poisson, 4-point gradient, CIC readout."""
    N, L = c["nmesh"], c["box"]
    cfg = _config(c)
    full, half = _wavenumbers(N)
    kf, cell = 2.0 * math.pi / L, L / N
    phi = torch.fft.rfftn(_paint64(x, mass, N))
    k2 = kf ** 2 * ((full ** 2)[:, None, None] + (full ** 2)[None, :, None] + (half ** 2)[None, None, :])
    k2[0, 0, 0] = math.inf
    phi = phi * (-1.5 * cfg.omega_m / k2)
    del k2
    if theta is not None:
        phi = phi * _factor64(theta, N, a)
    out = []
    for k, shape in ((full, (-1, 1, 1)), (full, (1, -1, 1)), (half, (1, 1, -1))):
        D = (8.0 * torch.sin(k * kf * cell) - torch.sin(2.0 * k * kf * cell)) / (6.0 * cell)
        D = torch.where(k.abs() == N // 2, torch.zeros_like(D), D).reshape(shape)
        out.append(_readout64(x, torch.fft.irfftn(phi * (-1j * D), s=(N, N, N)), N))  # 1 / N^3 in the inverse
    return torch.stack(out)


def _bins64(N, nbins):
    """Bin of every half-spectrum mode (nbins where none), its multiplicity and |n|."""
    full, half = _wavenumbers(N)
    n2 = (full ** 2)[:, None, None] + (full ** 2)[None, :, None] + (half ** 2)[None, None, :]
    r = torch.sqrt(n2)
    b = torch.floor(r - 0.5).long()
    b = torch.where((n2 == 0) | (b >= nbins), torch.full_like(b, nbins), b)
    mult = (1.0 + ((half > 0) & (half < N // 2)).double())[None, None, :].expand_as(r)
    return b.reshape(-1), mult.reshape(-1), r.reshape(-1)


def _power64(ra, rb, c):
    N, V, nb = c["nmesh"], c["box"] ** 3, c["nbins"]
    da = torch.fft.rfftn(ra / ra.mean())
    db = da if rb is None else torch.fft.rfftn(rb / rb.mean())
    full, half = _wavenumbers(N)
    w = [torch.sinc(k / N) ** -4 for k in (full, full, half)]
    P = (da * db.conj()).real * (V / float(N) ** 6) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    b, mult, r = _bins64(N, nb)
    total = lambda v: torch.zeros(nb + 1, dtype=torch.float64, device="cuda").index_add(0, b, v)[:nb]  # noqa: E731
    cnt = total(mult)
    safe = torch.clamp(cnt, min=1.0)
    return total(mult * r) / safe * (2.0 * math.pi / c["box"]), total(mult * P.reshape(-1)) / safe, cnt


def _species(c, m, which):
    n_cdm = c["nc"] ** 3
    m = m.clone()
    if which == 1:
        m[n_cdm:] = 0.0
    if which == 2:
        m[:n_cdm] = 0.0
    return m


def exact(case, seed):
    c, N, L = dict(case), case["nmesh"], case["box"]
    if c["kind"] in ("run", "gradient") or N > 1024:  # chained steps, and meshes beyond the memory
        return None
    t = _inputs(c, seed)
    n = t["u"].shape[1]
    x, m = _cells(t["u"], N), _masses(c, t["id"], n)
    if c["kind"] == "force":
        return _force64(x, m, c, 1.0)
    if c["kind"] == "power":
        ra = _paint64(x, _species(c, m, c["sa"]), N)
        rb = None if c["sb"] == c["sa"] else _paint64(x, _species(c, m, c["sb"]), N)
        k, P, _ = _power64(ra, rb, c)
        return k, P, None
    if c["kind"] == "power_vjp":
        x.requires_grad_()
        _, P, _ = _power64(_paint64(x, _species(c, m, c["sa"]), N), None, c)
        (g,) = torch.autograd.grad((P * torch.from_numpy(t["dL_dP"]).cuda()).sum(), x)
        return g * (N / L)
    a0, ah, a1 = _steps(c)[0]
    K1, delta, K2 = pm.cosmo_coeffs(_config(c), a0, ah, a1)
    theta = torch.from_numpy(t["theta"]).cuda().double().requires_grad_() if c["learned"] else None

    def transposed(x, lam, a):  # (dF / dx)^T lam in Mpc/h, and d <lam, F> / d theta
        x = x.detach().requires_grad_()
        F = _force64(x, m, c, a, theta)
        g = torch.autograd.grad((lam * F).sum(), [x] + ([theta] if c["learned"] else []))
        return g[0] * (N / L), g[1] if c["learned"] else 0.0

    lx, lp = t["lx"].double(), t["lp"].double()
    x1 = x + delta * (t["p"].double() + K1 * t["f"].double()) * (N / L)
    g, gt = transposed(x1 - torch.floor(x1 / N) * N, K2 * lp, a1)
    lx, gtheta = lx + g, gt
    lp = lp + delta * lx
    g, gt = transposed(x, K1 * lp, a0)
    lx, gtheta = lx + g, gtheta + gt
    return (lx, lp, gtheta) if c["learned"] else (lx, lp)
