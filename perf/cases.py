"""Performance cases of the SIDM scattering pass: what a simulation code has this
library do, through the public entry points of ``paper_2506_06269_gb300.sidm``.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare`` makes the inputs on the GPU together with the context a
program keeps, ``run`` is one pass, ``work`` what a pass cannot do without and
``exact`` the same results in 64-bit torch/numpy, without the library.

Families
  step       one step of a run: drift, reflecting boundary, cell build, kernel
             sizes (warm-started from the step before, as in any run), pairs,
             draws and scatter, energy and momentum
  satellite  one big step of a satellite in the analytic host: 2^(bins-1)
             sub-steps of kick, build, kernel sizes, scatter on individual
             steps, drift, kick; the new time steps; the host potential
  snapshot   analysis of a stored snapshot: build, kernel sizes without any
             earlier ones, local diagnostics
  neighbours neighbour lists of a stored snapshot
  stream     drift, cell build and energy of a uniform box far larger than L2
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2506_06269_gb300 import ics, sidm

SEED = 7                       # key of the scatter draws
S0, SIGMA_CONST, TAU, DT_MAX = 100.0, 10.0, 0.04, 0.02


def listed():
    return [
        # a small halo: every launch of the step counts
        dict(name="step_halo_2k", family="step", profile="hernquist", n=2048, ngb=32, fp64=False, dt=0.005),
        # a few small halos of uneven size in one context, all four neighbour numbers
        dict(name="step_batch_small", family="step", profile="nfw", halos=8, n_lo=1500, n_hi=30000, layout=5, ngb=0,
             fp64=False, dt=2.0 ** -6),
        # the benchmark halo: velocity-dependent cross-section, 64 neighbours
        dict(name="step_nfw_1m", family="step", profile="nfw", n=1 << 20, ngb=64, fp64=False, dt=0.005, vdep=True),
        # late core collapse at the paper's top resolution
        dict(name="step_cored_50m", family="step", profile="cored", n=50_000_000, ngb=64, fp64=False, dt=1e-4, vdep=True),
        # the convergence sweep: 64 halos from 10^4 to 2 10^6 particles, 16 to 128 neighbours
        dict(name="step_batch_64", family="step", profile="nfw", halos=64, n_lo=10_000, n_hi=2_000_000, layout=3, ngb=0,
             fp64=False, dt=0.01),
        # the plain method in FP64, small and at the benchmark's size
        dict(name="step_fp64_16k", family="step", profile="hernquist", n=16384, ngb=32, fp64=True, dt=0.001),
        dict(name="step_fp64_1m", family="step", profile="nfw", n=1 << 20, ngb=64, fp64=True, dt=0.005, vdep=True),
        # forward-dominated (frictional) scattering: every pair interacts
        dict(name="step_drag_16k", family="step", profile="hernquist", n=16384, ngb=32, fp64=False, dt=0.002, drag=True),
        # a satellite on the paper's orbit, individual time steps in four bins
        dict(name="satellite_4m", family="satellite", n=1 << 22, ngb=64, bins=4),
        # density, dispersion, h/l and Knudsen number of a snapshot at the paper's default of 48 neighbours
        dict(name="snapshot_300k", family="snapshot", profile="nfw", n=300_007, ngb=48, vdep=True),
        # neighbour lists of a snapshot
        dict(name="neighbours_100k", family="neighbours", profile="hernquist", n=100_003, ngb=48),
        # the streaming part of a step, far larger than L2
        dict(name="stream_33m", family="stream", profile="box", n=1 << 25),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["step", "step", "step", "batch", "fp64", "drag", "satellite", "snapshot", "neighbours", "stream"])
    ngb = rng.choice([16, 32, 48, 64, 128])
    profile = rng.choice(["hernquist", "nfw", "cored"])
    vdep = rng.random() < 0.5
    if family == "step":
        n = log_int(2000, 50_000_000 * min(1.0, 48 / ngb))
        return dict(family="step", profile=profile, n=n, ngb=ngb, fp64=False, dt=1e-3, vdep=vdep)
    if family == "batch":
        halos, lo = rng.randint(2, 64), log_int(1000, 20_000)
        hi = min(log_int(lo, 100 * lo), 60_000_000 // halos)
        return dict(family="step", profile=profile, halos=halos, n_lo=lo, n_hi=max(lo, hi), layout=rng.randrange(1 << 20),
                    ngb=0, fp64=False, dt=1e-3, vdep=vdep)
    if family == "fp64":
        n = log_int(2000, 1_000_000 * min(1.0, 64 / ngb))
        return dict(family="step", profile=profile, n=n, ngb=ngb, fp64=True, dt=1e-3, vdep=vdep)
    if family == "drag":
        return dict(family="step", profile=profile, n=log_int(2000, 40_000), ngb=rng.choice([16, 32, 48]), fp64=False,
                    dt=1e-3, vdep=vdep, drag=True)
    if family == "satellite":
        return dict(family="satellite", n=log_int(20_000, 4_000_000), ngb=rng.choice([32, 48, 64]), bins=rng.randint(2, 4))
    if family == "stream":
        return dict(family="stream", profile="box", n=log_int(100_000, 33_000_000))
    if family == "snapshot":
        return dict(family="snapshot", profile=profile, n=log_int(5000, 1_000_000), ngb=ngb, vdep=vdep)
    return dict(family="neighbours", profile=profile, n=log_int(5000, 1_000_000), ngb=ngb)


# ------------------------------------------------------------------ inputs
def _halos(case):
    """(particle numbers, neighbour numbers) of the case's halos."""
    if "halos" not in case:
        return [case["n"]], [case.get("ngb", 1)]
    r = random.Random(case["layout"])
    sizes = [int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))) for _ in range(case["halos"])]
    return sizes, [case["ngb"] or (16, 32, 64, 128)[h % 4] for h in range(case["halos"])]


@functools.lru_cache(maxsize=None)
def _profile(name):
    """Radius grid, mass inside it (1 at the truncation) and the isotropic Jeans dispersion there (G = 1)."""
    r = np.geomspace(1e-6, 1e4, 40001)
    if name == "hernquist":
        cut, rho = 20.0, 1.0 / (2.0 * math.pi * r * (1.0 + r) ** 3)
    else:
        cut, rho = 10.0, ics.NFW_RHO_S / (r * (1.0 + r) ** 2)
        if name == "cored":                       # the outer crossing joins the core to the NFW profile
            core = 1e3 * ics.NFW_RHO_S * (1.0 + (r / 0.05) ** 2) ** -1.5
            rho = np.where(np.arange(r.size) <= np.nonzero(core > rho)[0].max(), core, rho)

    def integral(f):                              # from r[0] up, trapezoid in log r
        y = f * r
        return np.concatenate([[0.0], np.cumsum(0.5 * (y[1:] + y[:-1]) * np.diff(np.log(r)))])

    m = integral(4.0 * math.pi * r * r * rho)
    down = integral(rho * m / r ** 2)
    sigma = np.sqrt(np.maximum((down[-1] - down) / rho, 1e-300))
    k = int(np.searchsorted(r, cut)) + 1
    return tuple(torch.tensor(x, device="cuda") for x in (r[:k], m[:k] / m[k - 1], sigma[:k] / math.sqrt(m[k - 1])))


def _interp(x, xp, fp):
    i = torch.searchsorted(xp, x).clamp_(1, xp.numel() - 1)
    t = (x - xp[i - 1]) / (xp[i] - xp[i - 1])
    return fp[i - 1] + t * (fp[i] - fp[i - 1])


def _make(case, seed):
    """Positions f64 [3][N], velocities [3][N], ids i32 [N]: every halo seeded and in no spatial order."""
    vdt = torch.float64 if case.get("fp64") else torch.float32
    sizes, _ = _halos(case)
    total = sum(sizes)
    pos = torch.empty((3, total), dtype=torch.float64, device="cuda")
    vel = torch.empty((3, total), dtype=vdt, device="cuda")
    ids = torch.empty(total, dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (seed + 1))
    at = 0
    for n in sizes:
        part = slice(at, at + n)
        at += n
        ids[part] = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
        u = torch.rand((3, n), generator=g, dtype=torch.float64, device="cuda")
        v = torch.randn((3, n), generator=g, dtype=torch.float32, device="cuda")
        if case.get("profile") == "box":
            pos[:, part], vel[:, part] = u, v
            continue
        r, m, sigma = _profile(case.get("profile", "nfw"))
        rad = _interp(u[0], m, r)
        mu, phi = 2.0 * u[1] - 1.0, (2.0 * math.pi) * u[2]
        st = torch.sqrt((1.0 - mu * mu).clamp_(min=0.0))
        pos[0, part], pos[1, part], pos[2, part] = rad * st * phi.cos(), rad * st * phi.sin(), rad * mu
        vel[:, part] = v * _interp(rad, r, sigma)
    if case["family"] == "satellite":
        x0, v0 = (torch.tensor(x, device="cuda")[:, None] for x in ics.satellite_orbit())
        pos += x0
        vel += v0.to(vdt)
    return pos, vel, ids


def _radius(case):
    return 20.0 if case.get("profile") == "hernquist" else 10.0


def prepare(case, seed):
    fam, n_ngb = case["family"], np.array(_halos(case)[1], np.int32)
    sizes = _halos(case)[0]
    H, N = len(sizes), sum(sizes)
    pos, vel, ids = _make(case, seed)
    flags, cap = 0, max(1 << 16, N // 8)
    if case.get("drag"):
        flags, cap = sidm.SIDM_FLAG_DRAG, 8 * N * int(n_ngb.max())
    if fam == "satellite":
        flags = sidm.SIDM_FLAG_SUM_P
    if fam == "snapshot":
        flags = sidm.SIDM_FLAG_LOCAL_DIAG
    ctx = sidm.Context(n_max=N, halo_max=H, ngb_max=int(n_ngb.max()), event_cap=cap,
                       precision="fp64" if case.get("fp64") else "mixed", flags=flags)
    xs = (1, S0, ics.nfw_vmax()) if case.get("vdep") or fam == "satellite" else (0, SIGMA_CONST, 1.0)
    s = dict(case=case, ctx=ctx, n=N, halos=H, off=np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), ngb=n_ngb,
             pos=pos, vel=vel, ids=ids, h=torch.zeros(N, dtype=ctx.vdtype, device="cuda"),
             xs=ctx.xs_tensor([xs + ((1,) if case.get("drag") else ())] * H), mass=ctx.f64([1.0 / n for n in sizes]),
             energy=torch.zeros((H, 4), dtype=torch.float64, device="cuda"), step=0)
    b = ctx.stats_buf            # the step's counts; its work counter n_tested is no result
    s["stats"] = [b[:40].view(torch.int64), b[40:48].view(torch.int32), b[48:56].view(torch.float64)]
    if fam in ("snapshot", "neighbours"):
        ctx.warm_start(False)
        s["stored"] = (pos.clone(), vel.clone(), ids.clone())
        return s
    ctx.build_cells(s["off"], pos, vel, ids)       # a run in progress: the step before left order and kernel sizes
    if fam == "stream":
        s["dt"] = ctx.f64([1e-3])
        return s
    ctx.kernel_sizes(n_ngb, s["h"])
    if fam == "satellite":
        S = 1 << (case["bins"] - 1)
        s.update(host=ics.milky_way_host(), dt=ctx.f64([DT_MAX / S]), dt_max=ctx.f64([DT_MAX]),
                 phi=torch.zeros(N, dtype=torch.float64, device="cuda"))
        # time steps held from the big step before: shorter where it is denser
        s["bins"] = (3.0 * torch.log2(0.08 / s["h"])).floor().clamp_(0, case["bins"] - 1).to(torch.int32)
    else:
        s["dt"] = ctx.f64([case["dt"]] * H)
        s["bound"] = ctx.f64([[0.0, 0.0, 0.0, _radius(case)]] * H)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    return _RUN[s["case"]["family"]](s)


def _run_step(s):
    c = s["ctx"]
    c.drift(s["dt"], s["pos"], s["vel"])
    c.reflect_boundary(s["bound"], s["pos"], s["vel"])
    c.build_cells(s["off"], s["pos"], s["vel"], s["ids"])
    c.kernel_sizes(s["ngb"], s["h"])
    c.scatter_step(SEED, s["step"], s["xs"], s["dt"], s["mass"], s["vel"])
    c.energy_momentum(s["mass"], s["vel"], s["energy"])
    s["step"] += 1
    return dict(pos=s["pos"], vel=s["vel"], ids=s["ids"], h=s["h"], energy=s["energy"], stats=s["stats"])


def _run_satellite(s):
    c, n, nb = s["ctx"], s["n"], s["case"]["bins"]
    S = 1 << (nb - 1)
    bins = s["bins"]
    for sub in range(S):
        c.host_kick(s["host"], DT_MAX, nb, sub, 0, bins, s["pos"], s["vel"])
        c.build_cells(s["off"], s["pos"], s["vel"], s["ids"])
        perm = c.perm(n).to(torch.int64)
        bins = bins[perm]                          # bins and new steps travel with their particles
        if sub:
            steps = steps[perm]
        c.kernel_sizes(s["ngb"], s["h"])
        c.scatter_step_binned(SEED, s["step"], s["xs"], DT_MAX, nb, sub, bins, s["mass"], s["vel"])
        if sub == 0:                               # every step opens: the rates of all pairs
            steps, _, shortest = c.timestep_criterion(TAU, 0.0, DT_MAX, nb, s["dt_max"], n, 1)
        c.drift(s["dt"], s["pos"], s["vel"])
        c.host_kick(s["host"], DT_MAX, nb, sub, 1, bins, s["pos"], s["vel"])
        s["step"] += 1
    c.host_potential(s["host"], s["pos"], s["phi"])
    s["bins"] = bins                               # a pass keeps the bins, so that every pass does the same work
    return dict(pos=s["pos"], vel=s["vel"], ids=s["ids"], h=s["h"], bins=bins, steps=steps, shortest=shortest,
                phi=s["phi"], stats=s["stats"])


def _restore(s):
    for x, y in zip((s["pos"], s["vel"], s["ids"]), s["stored"]):
        x.copy_(y)                                 # the build reorders in place: it works on a copy of the snapshot


def _run_snapshot(s):
    c = s["ctx"]
    _restore(s)
    c.build_cells(s["off"], s["pos"], s["vel"], s["ids"])
    c.kernel_sizes(s["ngb"], s["h"])
    local = c.local_diagnostics(s["xs"], s["mass"], s["vel"], s["n"])
    return dict(pos=s["pos"], vel=s["vel"], ids=s["ids"], h=s["h"], **local)


def _run_neighbours(s):
    c = s["ctx"]
    _restore(s)
    c.build_cells(s["off"], s["pos"], s["vel"], s["ids"])
    c.kernel_sizes(s["ngb"], s["h"])
    return dict(pos=s["pos"], ids=s["ids"], h=s["h"], lists=c.neighbours(s["ngb"], s["n"], int(s["ngb"][0])))


def _run_stream(s):
    c = s["ctx"]
    c.drift(s["dt"], s["pos"], s["vel"])
    c.build_cells(s["off"], s["pos"], s["vel"], s["ids"])
    c.energy_momentum(s["mass"], s["vel"], s["energy"])
    return dict(pos=s["pos"], vel=s["vel"], ids=s["ids"], energy=s["energy"])


_RUN = dict(step=_run_step, satellite=_run_satellite, snapshot=_run_snapshot, neighbours=_run_neighbours,
            stream=_run_stream)


def work(case):
    sizes, ngbs = _halos(case)
    N, R = sum(sizes), 8 if case.get("fp64") else 4
    state = 2 * (24 + 3 * R + 4)                   # positions, velocities and ids read and written
    near = sum(n * k for n, k in zip(sizes, ngbs))
    pairs = 4 * near                               # d < h_i + h_j, each unordered pair once
    fam = case["family"]
    if fam == "step":                              # a distance per neighbour; distance, speed and draw per pair
        return dict(bytes=N * (state + 2 * R), flops=8.0 * near + pairs * (140.0 if case.get("drag") else 70.0))
    if fam == "satellite":
        S = 1 << (case["bins"] - 1)
        return dict(bytes=N * (state + 2 * R + 4 + 8 + 8), flops=S * 8.0 * near + pairs * 2 * 70.0)
    if fam == "snapshot":
        return dict(bytes=N * (state + 6 * R), flops=near * 30.0)
    if fam == "neighbours":
        return dict(bytes=N * (state - 6 * R + R) + 4 * near, flops=near * 8.0)
    return dict(bytes=N * state, flops=N * 12.0)


# ------------------------------------------------------------------ 64-bit results
def exact(case, seed):
    """run()'s outputs in FP64, where that is quick: orders and energies of every single-pass case, kernel sizes
    and what follows from them by brute force up to 400,000 particles, scattered velocities up to 40,000."""
    fam = case["family"]
    sizes, ngbs = _halos(case)
    if fam == "satellite":
        return None
    pos, vel, ids = _make(case, seed)
    vel = vel.double()
    starts = np.concatenate([[0], np.cumsum(sizes)])
    out = dict(pos=[], vel=[], h=[], energy=[], local={})
    for k, (n, ngb) in enumerate(zip(sizes, ngbs)):
        part = slice(int(starts[k]), int(starts[k + 1]))
        x, v, d = pos[:, part], vel[:, part], ids[part]
        o = _order(x)
        x, v, d = x[:, o], v[:, o], d[o]
        if fam in ("step", "stream"):              # the drift (and the boundary), then the order of the pass
            x = x + v * (case["dt"] if fam == "step" else 1e-3)
            if fam == "step":
                r2, vr = (x * x).sum(0), (x * v).sum(0)
                v = torch.where((r2 > _radius(case) ** 2) & (vr > 0.0), v - 2.0 * vr / r2 * x, v)
            o = _order(x)
            x, v, d = x[:, o], v[:, o], d[o]
        m = 1.0 / n
        out["energy"].append(torch.cat([0.5 * m * (v * v).sum()[None], m * v.sum(1)]))   # a scatter keeps both
        h = None
        if fam != "stream" and sum(sizes) <= 400_000:
            h, near = _nearest(x, ngb)
            if fam == "snapshot":
                out["local"] = _local(case, x, v, h, near, ngb, m)
        if fam == "step":
            v = _scatter(case, x, v, d, h, k, m) if h is not None and n <= 40_000 and not case.get("drag") else None
        for key, value in (("pos", x), ("vel", v), ("h", h)):
            out[key].append(value)

    def joined(key, dim=0):
        return None if any(t is None for t in out[key]) else torch.cat(out[key], dim)

    res = dict(pos=joined("pos", 1), ids=None, h=joined("h"))
    if fam == "stream":
        return dict(pos=res["pos"], vel=joined("vel", 1), ids=None, energy=torch.stack(out["energy"]))
    if fam == "neighbours":
        return dict(res, lists=None)
    if fam == "snapshot":
        return dict(res, vel=joined("vel", 1), **out["local"]) if out["local"] else dict(
            res, vel=joined("vel", 1), rho=None, nu=None, sigma_eff=None, h_over_l=None, kn=None)
    return dict(res, vel=joined("vel", 1), energy=torch.stack(out["energy"]), stats=[None, None, None])


def _order(x):
    """Stable Morton order (17 bits per axis) in the power-of-two cube around the halo."""
    lo = x.amin(1)
    E = math.frexp(float((x.amax(1) - lo).amax()))[1]
    O = torch.floor(lo * 2.0 ** -E) * 2.0 ** E
    q = torch.floor((x - O[:, None]) * 2.0 ** (16 - E)).clamp_(0, (1 << 17) - 1).to(torch.int64)
    key = torch.zeros(x.shape[1], dtype=torch.int64, device=x.device)
    for b in range(17):
        for a in range(3):
            key |= ((q[a] >> b) & 1) << (3 * b + a)
    return torch.sort(key, stable=True)[1]


def _rows(n):
    step = max(1, (1 << 28) // n)
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _d2(x, a, b):
    d2 = (x[0, a:b, None] - x[0]).square_()
    for c in (1, 2):
        d2 += (x[c, a:b, None] - x[c]).square_()
    return d2


def _nearest(x, k):
    """Distance to the k-th nearest other particle, and the k nearest."""
    n = x.shape[1]
    h = torch.empty(n, dtype=torch.float64, device=x.device)
    near = torch.empty((n, k), dtype=torch.int32, device=x.device)
    for a, b in _rows(n):
        d2 = _d2(x, a, b)
        d2[torch.arange(b - a), torch.arange(a, b)] = math.inf
        t = torch.topk(d2, k, dim=1, largest=False)
        h[a:b] = t.values.amax(1).sqrt()
        near[a:b] = t.indices.to(torch.int32)
    return h, near


def _spline(q):
    return (8.0 / math.pi) * torch.where(q < 0.5, 1.0 - 6.0 * q * q * (1.0 - q), 2.0 * (1.0 - q).clamp(min=0.0) ** 3)


def _local(case, x, v, h, near, ngb, m):
    """Kernel-weighted density and dispersion, effective cross-section, h/l and Knudsen number."""
    j = near.long()
    d = torch.sqrt(sum((x[a][j] - x[a][:, None]) ** 2 for a in range(3)))
    w = m * _spline(d / h[:, None]) / h[:, None] ** 3
    self_w = m * (8.0 / math.pi) / h ** 3
    rho = w.sum(1) + self_w
    mean = [((w * v[a][j]).sum(1) + self_w * v[a]) / rho for a in range(3)]
    var = sum(((w * (v[a][j] - mean[a][:, None]) ** 2).sum(1) + self_w * (v[a] - mean[a]) ** 2) / rho for a in range(3))
    nu = torch.sqrt(var / 3.0)
    if case.get("vdep"):                           # <v^5 sigma> / <v^5> over the pair Maxwellian, t = v^2 / (4 nu^2)
        beta, gx, gw = 4.0 * nu * nu / ics.nfw_vmax() ** 2, *np.polynomial.legendre.leggauss(8)
        ratio = torch.zeros_like(nu)
        edge = 64.0 * (np.arange(401) / 400.0) ** 3
        for lo, hi in zip(edge[:-1], edge[1:]):
            for a, b in zip(gx, gw):
                t = 0.5 * (lo + hi) + 0.5 * (hi - lo) * a
                ratio += 0.5 * (hi - lo) * b * t ** 3 * math.exp(-t) / (1.0 + beta * t) ** 2
        sig = S0 * ratio / 6.0
    else:
        sig = torch.full_like(nu, SIGMA_CONST)
    hl = sig * rho ** (2.0 / 3.0) * (3.0 * m * ngb / (math.pi * math.sqrt(2.0))) ** (1.0 / 3.0)
    return dict(rho=rho, nu=nu, sigma_eff=sig, h_over_l=hl, kn=torch.sqrt(4.0 * math.pi / (rho * nu * nu)) / sig)


def _philox(c, key):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    lo32 = 0xFFFFFFFF
    c = list(c)
    k0, k1 = key & lo32, key >> 32

    def mul(a, x):                                 # (high, low) words of a 32 x 32-bit product
        p, q = a * (x & 0xFFFF), a * (x >> 16)
        low = p + ((q & 0xFFFF) << 16)
        return ((q >> 16) + (low >> 32)) & lo32, low & lo32

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & lo32, (k1 + 0xBB67AE85) & lo32
    return c


def _overlap(d, a, b):
    """Overlap integral of the spline kernels of support a and b at distance d (numpy, one pair)."""
    if d >= a + b:
        return 0.0
    P = np.polynomial.polynomial
    c = 8.0 / math.pi
    inner, outer = np.array([1.0, 0.0, -6.0, 6.0]) * c, np.array([2.0, -6.0, 6.0, -2.0]) * c
    w1 = lambda t: np.where(t < 0.5, P.polyval(t, inner), np.where(t < 1.0, P.polyval(t, outer), 0.0))
    s_in, s_out = P.polyint(np.r_[0.0, inner]), P.polyint(np.r_[0.0, outer])
    half = P.polyval(0.5, s_in) - P.polyval(0.5, s_out)
    s1 = lambda t: np.where(t < 0.5, P.polyval(t, s_in), P.polyval(np.minimum(t, 1.0), s_out) + half)
    lo, hi = max(0.0, d - b), min(a, d + b)
    br = [lo, hi] + [t for t in (a / 2, d, d - b / 2, d + b / 2, b / 2 - d, b - d) if lo < t < hi]
    br = np.sort(br)
    gx, gw = np.polynomial.legendre.leggauss(12)
    r = (0.5 * (br[1:] + br[:-1]))[:, None] + (0.5 * np.diff(br))[:, None] * gx
    f = r * w1(r / a) / a ** 3 * (s1((r + d) / b) - s1(np.abs(r - d) / b)) / b
    return 2.0 * math.pi / d * float((f * gw * (0.5 * np.diff(br))[:, None]).sum())


def _scatter(case, x, v, ids, h, halo, m):
    """The first step's events, drawn pair by pair and applied in key order."""
    n, dt, found = x.shape[1], case["dt"], []
    w = ics.nfw_vmax()
    for a, b in _rows(n):
        d2 = _d2(x, a, b)
        inside = d2 < (h[a:b, None] + h) ** 2
        inside &= torch.arange(n, device=x.device) > torch.arange(a, b, device=x.device)[:, None]
        i, j = torch.nonzero(inside, as_tuple=True)
        d = d2[i, j].sqrt()
        i = i + a
        lo, hi = torch.minimum(ids[i], ids[j]).long(), torch.maximum(ids[i], ids[j]).long()
        draws = _philox([torch.zeros_like(lo), lo, hi, torch.full_like(lo, halo)], SEED)
        speed = (v[:, i] - v[:, j]).square().sum(0).sqrt()
        rate = m * dt * speed * (S0 / (1.0 + (speed / w) ** 2) ** 2 if case.get("vdep") else SIGMA_CONST)
        u = draws[0].double() * 2.0 ** -32
        keep = u < 4.0 * rate / torch.maximum(h[i], h[j]) ** 3          # the overlap is at most (8/pi) / h_max^3
        cols = [t[keep].cpu().numpy() for t in (lo, hi, i, j, d, h[i], h[j], rate, u, draws[1], draws[2])]
        found += list(zip(*cols))
    v = v.cpu().numpy().copy()
    by_id = ids.cpu().numpy()
    for lo, hi, i, j, d, hi_, hj, rate, u, x1, x2 in sorted(found, key=lambda t: (t[0], t[1])):
        if not u < rate * _overlap(float(d), float(hi_), float(hj)):
            continue
        if by_id[i] != lo:
            i, j = j, i
        c = 2.0 * x1 * 2.0 ** -32 - 1.0
        phi = 2.0 * math.pi * x2 * 2.0 ** -32
        s = math.sqrt(1.0 - c * c)
        mean, half = 0.5 * (v[:, i] + v[:, j]), 0.5 * np.linalg.norm(v[:, i] - v[:, j])
        turn = half * np.array([s * math.cos(phi), s * math.sin(phi), c])
        v[:, i], v[:, j] = mean + turn, mean - turn
    return torch.tensor(v, device=x.device)
