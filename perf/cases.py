"""What the library is measured on: a made-to-measure run as its users have it.

A user creates a context (or a batch of them) over device particle arrays and
then, for hours, calls m2m_step with tens of steps at a time and reads the
record; in between it observes, recomputes the potential of the particles and
measures the velocity ellipsoid.  The cases are those calls over the
workloads of paper_1207_6403_gb300/inputs.py, from 20,000 particles (every
step is latency) to 8,000,000 (every step streams the state from HBM), in
both precisions.

Inputs are drawn with torch on the GPU from the seed alone (the realisations
of inputs.py, at the speed a measurement needs).  The model weights start
with the spread of a model that has been adapting (log-normal, 0.3) rather
than at 1/N, so that the entropy, its gradient and the prior-cell means take
the values they have in the middle of a run.
"""
import math

import numpy as np
import torch

from paper_1207_6403_gb300 import inputs as I
from paper_1207_6403_gb300 import m2m

DEV = "cuda:0"
DT, MU, ALPHA, ENT = 0.01, 1e-3, 0.02, 1.0
PERIOD = 25                     # steps between prior recomputes of every workload with moving priors
NOMINAL = {"plain": 20_000, "moving-priors": 1_000_000}    # the particle count the adaptation rate belongs to


def listed():
    return [
        # the smallest model, in double: every step is launch and memory latency
        dict(name="plain fp64 20k", work="plain", call="step", n=20_000, steps=10, prec="fp64", bins=40),
        # a driver that steps once per call and reads each record (lazy weight updates)
        dict(name="step by step 100k", work="moving-priors", call="loop", n=100_000, steps=1, prec="fp32c", bins=100),
        # forward model only: the observables of a set of particles
        dict(name="observe 1M", work="moving-priors", call="observe", n=1_000_000, steps=0, prec="fp32c", bins=100),
        # the anisotropy analysis of the recovery experiment (8 shells)
        dict(name="velocity moments 1M", work="moving-priors", call="moments", n=1_000_000, steps=0, prec="fp32c",
             bins=100),
        # shells and kinematic annuli, (E, L/Lc) priors recomputed once in the call
        dict(name="moving priors 1M", work="moving-priors", call="step", n=1_000_000, steps=25, prec="fp32c",
             bins=100),
        # a reference run in double of the pixel + IFU workload
        dict(name="flat-log fp64 300k", work="flat-log", call="step", n=300_000, steps=25, prec="fp64", bins=64),
        # the headline workload: pixels and IFU apertures, (E, L_z) priors
        dict(name="flat-log 4M", work="flat-log", call="step", n=4_000_000, steps=25, prec="fp32c", bins=64),
        # Voronoi bins and a long slit behind a PSF, an odd particle count
        dict(name="ifu-lut seeing 2M", work="ifu-lut-seeing", call="step", n=1_999_999, steps=25, prec="fp32c",
             bins=64),
        # bins of equal mass (no uniform spacing), four sets, halo potential: real data's set-up
        dict(name="adaptive bins 1M", work="adaptive", call="step", n=1_000_003, steps=25, prec="fp32c", bins=60),
        # 48 trial potentials advanced together, their records compared
        dict(name="batch 48", work="batched", call="batch", n=60_000, steps=25, prec="fp32c", bins=100),
        # the self-consistent potentials: one period of the expansion
        dict(name="triaxial 2M", work="sh-tri", call="step", n=2_000_000, steps=50, prec="fp32c", bins=100),
        dict(name="disc and bulge 8M", work="sh-selfcons", call="step", n=8_000_000, steps=50, prec="fp32c",
             bins=100),
    ]


def draw(rng):
    """A case of the same ranges: any workload, sizes spread over their logarithm."""
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1
    work = rng.choice(["plain", "moving-priors", "moving-priors", "flat-log", "flat-log", "ifu-lut",
                       "ifu-lut-seeing", "adaptive", "batched", "sh-selfcons", "sh-tri", "sh-full"])
    call, prec, steps = "step", "fp32c", rng.choice([5, 10, 25, 50])
    bins = {"flat-log": rng.randrange(40, 73), "ifu-lut": rng.randrange(40, 73),
            "ifu-lut-seeing": rng.randrange(40, 73), "plain": rng.randrange(20, 61)}.get(work, rng.randrange(40, 121))
    if work == "batched":
        return dict(work=work, call="batch", n=size(10_000, 60_000), steps=rng.choice([5, 10, 25]), prec="fp32c",
                    bins=bins)
    if work.startswith("sh-"):
        return dict(work=work, call="step", n=size(100_000, 4_000_000 if work == "sh-selfcons" else 2_000_000),
                    steps=rng.choice([25, 50]), prec=prec, bins=bins)
    if work in ("plain", "moving-priors") and rng.random() < 0.4:
        call = rng.choice(["loop", "observe", "moments"])
        return dict(work=work, call=call, n=size(20_000, 1_500_000), steps=1 if call == "loop" else 0, prec=prec,
                    bins=bins)
    if work in ("plain", "moving-priors", "flat-log") and rng.random() < 0.4:
        return dict(work=work, call="step", n=size(20_000, 300_000), steps=rng.choice([5, 10, 25]), prec="fp64",
                    bins=bins)
    return dict(work=work, call=call, n=size(20_000, 4_000_000), steps=min(steps, 25), prec=prec, bins=bins)


# ------------------------------------------------------------------ particles
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _u(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _directions(g, n):
    c, p = 2.0 * _u(g, n) - 1.0, 2.0 * math.pi * _u(g, n)
    s = torch.sqrt(1.0 - c * c)
    return torch.stack([s * torch.cos(p), s * torch.sin(p), c])


def _interp(x, xp, fp):
    xp, fp = torch.as_tensor(xp, device=DEV), torch.as_tensor(fp, device=DEV)
    k = torch.clamp(torch.searchsorted(xp, x.contiguous(), right=True) - 1, 0, len(xp) - 2)
    t = torch.clamp((x - xp[k]) / (xp[k + 1] - xp[k]), 0.0, 1.0)
    return fp[k] + t * (fp[k + 1] - fp[k])


def _jeans(rho, mass, ra=None):
    """ln r and sigma_r of the spherical Jeans equation (isotropic, or beta = r^2/(r^2+ra^2))."""
    lr = np.linspace(math.log(1e-5), math.log(1e4), 4001)
    r = np.exp(lr)
    g = np.ones_like(r) if ra is None else r * r + ra * ra
    f = g * rho(r) * mass(r) / r
    seg = 0.5 * (lr[1] - lr[0]) * (f[1:] + f[:-1])
    tail = np.concatenate([np.cumsum(seg[::-1])[::-1], [0.0]]) + f[-1] / 3.0
    return lr, np.sqrt(tail / (g * rho(r)))


def _hernquist(g, n, M=1.0, a=1.0, rmax=100.0, more=lambda r: 0.0, ra=None):
    """A Hernquist sphere in its own mass and `more`, ordered by radius."""
    s = torch.sqrt(_u(g, n) * (rmax / (rmax + a)) ** 2)
    r = torch.sort(a * s / (1.0 - s))[0]
    er = _directions(g, n)
    lr, sg = _jeans(lambda q: M * a / (2 * math.pi * q * (q + a) ** 3), lambda q: M * q * q / (q + a) ** 2 + more(q), ra)
    sr = _interp(torch.log(r), lr, sg)
    vel = _normal(g, 3, n) * sr
    if ra is not None:              # tangential dispersions smaller by sqrt(1 - beta)
        k = torch.sqrt(ra * ra / (r * r + ra * ra))
        vr = (vel * er).sum(0)
        vel = vel * k + er * (vr * (1.0 - k))
    return r * er, vel


def _log_galaxy(g, n, stream):
    """The density of the flattened logarithmic potential (v0 = 1, Rc = 0.1, q = 0.8) inside m = 5, ordered by m."""
    q, Rc, got, have = 0.8, 0.1, [], 0
    while have < n:
        k = int(2.4 * (n - have)) + 1024
        m = 5.0 * _u(g, k)
        m = m[_u(g, k) < m * m / (Rc * Rc + m * m)]
        p = m * _directions(g, m.numel())
        p[2] *= q
        R2 = p[0] ** 2 + p[1] ** 2
        rho = ((2 * q * q + 1) * Rc * Rc + R2 + (2 - 1 / (q * q)) * p[2] ** 2) / (Rc * Rc + m * m)
        p = p[:, _u(g, m.numel()) * (2 * q * q + 1) < rho]
        got.append(p)
        have += p.shape[1]
    pos = torch.cat(got, 1)[:, :n]
    pos = pos[:, torch.argsort(pos[0] ** 2 + pos[1] ** 2 + (pos[2] / q) ** 2, stable=True)].contiguous()
    vel = _normal(g, 3, n) / math.sqrt(2.0)
    R = torch.sqrt(pos[0] ** 2 + pos[1] ** 2)
    vc = stream * R / torch.sqrt(Rc * Rc + R * R) / torch.clamp(R, min=1e-30)
    vel[0] -= vc * pos[1]
    vel[1] += vc * pos[0]
    return pos, vel


def _disc_bulge(g, n):
    """A Miyamoto-Nagai disc (1, 0.2) and a Hernquist bulge (0.3), 1 : 3 by mass, ordered by radius."""
    nd, Md, Mb, a, b, ab = n // 4, 0.25, 0.75, 1.0, 0.2, 0.3
    Re = np.concatenate([[0.0], np.geomspace(1e-3, 30.0, 600)])
    ze = b * np.sinh(np.linspace(0.0, math.asinh(30.0 / b), 401))
    Rm, zm = 0.5 * (Re[1:] + Re[:-1])[:, None], 0.5 * (ze[1:] + ze[:-1])[None, :]
    zeta = np.sqrt(zm * zm + b * b)
    rho = (a * Rm * Rm + (a + 3 * zeta) * (a + zeta) ** 2) / ((Rm * Rm + (a + zeta) ** 2) ** 2.5 * zeta ** 3)
    cdf = np.cumsum((rho * (Re[1:] ** 2 - Re[:-1] ** 2)[:, None] * np.diff(ze)[None, :]).ravel())
    cell = torch.searchsorted(torch.as_tensor(cdf / cdf[-1], device=DEV), _u(g, nd)).clamp(max=cdf.size - 1)
    iR, iz = cell // 400, cell % 400
    Re, ze = torch.as_tensor(Re, device=DEV), torch.as_tensor(ze, device=DEV)
    R = torch.sqrt(Re[iR] ** 2 + _u(g, nd) * (Re[iR + 1] ** 2 - Re[iR] ** 2))
    z = (ze[iz] + _u(g, nd) * (ze[iz + 1] - ze[iz])) * torch.sign(_u(g, nd) - 0.5)
    phi = 2 * math.pi * _u(g, nd)
    vc = torch.sqrt(Md * R * R / (R * R + (a + b) ** 2) ** 1.5 + Mb * R / (R + ab) ** 2)
    v = 0.1 * vc * _normal(g, 3, nd)
    v[1] += vc
    c, s = torch.cos(phi), torch.sin(phi)
    dp, dv = torch.stack([R * c, R * s, z]), torch.stack([v[0] * c - v[1] * s, v[0] * s + v[1] * c, v[2]])
    bp, bv = _hernquist(g, n - nd, Mb, ab, 30.0, lambda r: Md * r ** 3 / (r * r + (a + b) ** 2) ** 1.5)
    pos, vel = torch.cat([dp, bp], 1), torch.cat([dv, bv], 1)
    o = torch.argsort((pos * pos).sum(0), stable=True)
    return pos[:, o].contiguous(), vel[:, o].contiguous()


def _halo(ratio, rs):
    c = math.log1p(10.0) - 10.0 / 11.0
    rho_s = ratio / (4 * math.pi * rs ** 3 * c)
    return rho_s, lambda r: ratio / c * (np.log1p(r / rs) - r / (r + rs))


# ------------------------------------------------------------------ workloads
def _annuli_gh(nb, M=1.0, a=1.0):
    e = I.log_shell_edges(nb, 0.05, 20.0)
    lr, sg = _jeans(lambda q: M * a / (2 * math.pi * q * (q + a) ** 3), lambda q: M * q * q / (q + a) ** 2)
    S = np.maximum(np.interp(0.25 * np.log(e[:-1] * e[1:]), lr, sg), 0.05)
    return I.ObservableSet("annulus", "gh", e, gh_V=np.zeros(nb), gh_S=S, sigma_kernel=0.1)


def _workload(case, seed):
    """Everything but the particle arrays' precision: model and target particles, sets, potential, priors."""
    g, n, b, work = _gen(seed), case["n"], case["bins"], case["work"]
    nt = min(n, 400_000)            # particles of the target galaxy
    P, S, U = I.PotentialComponent, I.ObservableSet, I.uniform_edges
    inc = 0.0
    sh2 = [S("shell", "mass", I.log_shell_edges(b, 0.05, 20.0))]
    if work in ("plain", "moving-priors"):
        model, target = _hernquist(g, n), _hernquist(g, nt, ra=1.0)
        pot = [P("hernquist", (1.0, 1.0))]
        if work == "plain":
            ann = I.log_shell_edges(b // 2, 0.05, 20.0)
            obs, prior = sh2 + [S("annulus", "mass", ann), S("annulus", "vlos2", ann.copy())], I.PriorSpec("flat")
        else:
            obs = sh2 + [_annuli_gh(3 * b // 5)]
            prior = I.PriorSpec("e_lc", 64, 32, PERIOD, (1.0, 1.0))
    elif work == "adaptive":
        # radii of equal mass fractions: no uniform spacing in r or log r
        rho_s, more = _halo(4.0, 5.0)
        model, target = _hernquist(g, n, more=more), _hernquist(g, nt, more=more, ra=1.0)
        pot = [P("hernquist", (1.0, 1.0)), P("nfw", (rho_s, 5.0))]
        s = np.sqrt(np.linspace(0.002, 0.95, b + 1))
        e = (s / (1.0 - s)) ** 2
        ap = np.concatenate([-np.geomspace(4.0, 0.1, 8), np.geomspace(0.1, 4.0, 8)])
        V, W = np.zeros(225), np.full(225, 0.4)
        obs = [S("shell", "mass", e), S("annulus", "mass", 0.7 * e), S("annulus", "vlos2", 0.7 * e),
               S("grid", "gh", ap, ap.copy(), gh_V=V, gh_S=W, sigma_kernel=0.1)]
        prior, inc = I.PriorSpec("e_l2", 64, 32, PERIOD), 30.0
    elif work in ("flat-log", "ifu-lut", "ifu-lut-seeing"):
        model, target = _log_galaxy(g, n, 0.0), _log_galaxy(g, nt, 0.5)
        pot = [P("log", (1.0, 0.1, 0.8))]
        px = U(b, -3.2, 3.2)
        obs = [S("grid", "mass", px, px.copy())]
        if work == "flat-log":
            na = 5 * b // 16
            ap = U(na, -2.0, 2.0)
            obs.append(S("grid", "gh", ap, ap.copy(), gh_V=np.zeros(na * na), gh_S=np.full(na * na, 0.5 ** 0.5),
                         sigma_kernel=0.1))
        else:
            vx, sx = U(160, -2.0, 2.0), U(256, -3.2, 3.2)
            for k, (ed, lut, nc) in enumerate((
                    (vx, I.voronoi_lut(vx, vx, I.ifu_generators(300, 11, 2.0), rmax=2.0), 300),
                    (sx, I.slit_lut(sx, sx, 30.0, 0.2, U(40, -3.0, 3.0)), 40))):
                more = {}
                if work == "ifu-lut-seeing":
                    more = dict(psf_q=_psf(), psf_seed=12346 + k)
                obs.append(S("lut", "gh", ed, ed.copy(), gh_V=np.zeros(nc), gh_S=np.full(nc, 0.5 ** 0.5),
                             sigma_kernel=0.1, lut=lut, n_apertures=nc, **more))
        prior, inc = I.PriorSpec("e_lz", 128, 64, PERIOD), 60.0
    elif work == "sh-selfcons":
        model, target = _disc_bulge(g, n), _disc_bulge(g, nt)
        pot, prior = [P("sh", (256, 1e-3, 100.0, 50))], I.PriorSpec("flat")
        obs = sh2 + [_annuli_gh(3 * b // 5, 0.75, 0.3)]
    else:                            # sh-tri, sh-full
        sets = []
        for m in (n, nt):
            p, v = _hernquist(g, m)
            k = torch.tensor([[1.0], [0.8], [0.6]], device=DEV, dtype=torch.float64)
            p, v = p * k, v * k
            if work == "sh-full":
                p, v = _turned(p) + torch.tensor([[0.05], [-0.03], [0.02]], device=DEV, dtype=torch.float64), _turned(v)
            sets.append((p, v))
        model, target = sets
        pot = [P("sh_tri", (256, 1e-3, 100.0, 50)) if work == "sh-tri" else P("sh_full", (128, 1e-3, 100.0, 50))]
        prior = I.PriorSpec("e_l2", 64, 32, PERIOD)
        obs = sh2 + [_annuli_gh(3 * b // 5)]
    return _problem(g, n, model, target, pot, obs, prior, inc, 0.05 / max(n, NOMINAL.get(work, 4_000_000)))


_PSF = []


def _psf():
    """A Gaussian PSF of dispersion 0.1 as 4096 quantiles (a table of the instrument, not of the seed)."""
    if not _PSF:
        _PSF.append(I.gaussian_psf_table(0.1))
    return _PSF[0]


def _turned(v):
    a, b = 0.5, 0.7
    x, y, z = v
    x, y = math.cos(a) * x - math.sin(a) * y, math.sin(a) * x + math.cos(a) * y
    return torch.stack([math.cos(b) * x + math.sin(b) * z, y, math.cos(b) * z - math.sin(b) * x])


def _problem(g, n, model, target, pot, obs, prior, inc, eps):
    w = torch.exp(0.3 * _normal(g, n))
    w = w / w.sum()
    par = dict(eps=eps, mu=MU, dt=DT, alpha=ALPHA, entropy_const=ENT, incl_sin=math.sin(math.radians(inc)),
               incl_cos=math.cos(math.radians(inc)))
    nt = target[0].shape[1]
    Y = _observe64(obs, par, *target, torch.full((nt,), 1.0 / nt, device=DEV, dtype=torch.float64))[0].cpu().numpy()
    sigma = I.error_model(Y, obs)
    sigma = np.where(sigma > 0, np.maximum(sigma, 0.2 / nt), 0.0)    # bins of a few target particles: no 2 per cent
    return dict(pos=model[0], vel=model[1], w=w, what=torch.full_like(w, 1.0 / n), pot=pot, obs=obs, prior=prior,
                par=par, Y=Y, sigma=sigma)


def _batch_models(case, seed):
    """48 halos (mass ratio x scale radius), particle counts spread by a factor of twenty about the case's n."""
    g, out, b = _gen(seed), [], case["bins"]
    for k in range(48):
        rho_s, more = _halo(I.HALO_MASS_RATIOS[k // 8], I.HALO_RS[k % 8])
        n = int(case["n"] * math.exp(math.log(20.0) * ((7 * k) % 48 / 47.0 - 0.5)))
        pot = [I.PotentialComponent("hernquist", (1.0, 1.0)), I.PotentialComponent("nfw", (rho_s, I.HALO_RS[k % 8]))]
        obs = [I.ObservableSet("shell", "mass", I.log_shell_edges(b, 0.05, 20.0)), _annuli_gh(3 * b // 5)]
        out.append(_problem(g, n, _hernquist(g, n, more=more), _hernquist(g, 20_000, more=more, ra=1.0), pot, obs,
                            I.PriorSpec("flat"), 0.0, 0.05 / 1_000_000))
    return out


# ------------------------------------------------------------------ the calls
class State:
    pass


ARRAYS = ("x", "y", "z", "vx", "vy", "vz", "w", "what")


def prepare(case, seed):
    s = State()
    s.case = case
    if case["call"] == "batch":
        probs = []
        for d in _batch_models(case, seed):
            n = d["w"].numel()
            probs.append(I.Problem(
                name="trial", n=n, pos=d["pos"].cpu().numpy(), vel=d["vel"].cpu().numpy(), w0=d["w"].cpu().numpy(),
                what0=d["what"].cpu().numpy(), potential=d["pot"], obs=d["obs"], incl_sin=0.0, incl_cos=1.0,
                eps=d["par"]["eps"], mu=MU, dt=DT, alpha=ALPHA, prior=d["prior"], nsteps=case["steps"],
                precision=case["prec"], Y=d["Y"], sigma=d["sigma"]))
        s.batch = m2m.m2m_batch_init(case["prec"], probs, device=DEV)
        return s
    d = _workload(case, seed)
    s.ctx = m2m.m2m_init(case["prec"], d["pos"], d["vel"], d["w"], d["what"], d["pot"], d["obs"], d["par"],
                         d["prior"], d["Y"], d["sigma"], DEV)
    if case["call"] == "loop":
        s.ctx.m2m_set_lazy_update(True)
    if case["call"] == "moments":
        s.edges = np.geomspace(0.2, 5.0, 9) ** 2
    return s


def _record(r):
    # S and sum w are sums of float terms (FP32C): returned as what they are
    return dict(chi2=r["chi2"], chi2_raw=r["chi2_raw"], max_abs_dt=r["max_abs_dt"], S=np.float32(r["S"]),
                sum_w=np.float32(r["sum_w"]))


def run(s):
    case = s.case
    if case["call"] == "batch":
        s.batch.m2m_batch_step(case["steps"])
        recs = s.batch.m2m_batch_get_records()
        out = {k: torch.cat([t[k] for t in s.batch.t]) for k in ARRAYS}
        out["chi2"] = np.array([r["chi2"] for r in recs])
        out["S"] = np.array([r["S"] for r in recs], dtype=np.float32)
        return out
    if case["call"] == "moments":
        return s.ctx.m2m_velocity_moments(s.edges)
    if case["call"] == "observe":
        s.ctx.m2m_observe(2)
        return list(s.ctx.m2m_get_obs())
    s.ctx.m2m_step(case["steps"])
    out = dict(s.ctx.t, record=_record(s.ctx.m2m_get_record()))
    if case["call"] == "step":
        out["obs"] = list(s.ctx.m2m_get_obs())
    return out


def work(case):
    """Bytes of the step's unit, the particle-step: position and velocity read and written, the weight read and
    written, the prior read (72 bytes in FP32C, 120 in FP64); a prior recompute reads the state and the weight and
    writes the prior; an expansion reads positions and weights.  Operations: the push's, the kernels' and the
    update's, counted by hand."""
    n, steps, f32 = case["n"], case["steps"], case["prec"] == "fp32c"
    r = 4 if f32 else 8
    if case["call"] == "batch":
        n = sum(int(case["n"] * math.exp(math.log(20.0) * (k / 47.0 - 0.5))) for k in range(48))
    if case["call"] == "observe":
        return dict(bytes=n * (6 * r + 8), flops=60 * n)
    if case["call"] == "moments":
        return dict(bytes=n * (6 * r + 8), flops=40 * n)
    per = {"sh-selfcons": 220, "sh-tri": 520, "sh-full": 620, "adaptive": 180}.get(case["work"], 140)
    b = 72.0 if f32 else 120.0
    if case["work"] not in ("plain", "batched", "sh-selfcons"):
        b += (6 * r + 16) / PERIOD
    if case["work"].startswith("sh-"):
        b += (3 * r + 8) / 50
    return dict(bytes=b * n * steps, flops=float(per) * n * steps)


# ------------------------------------------------------------------ in 64 bits
def _sky(par, p, v):
    s, c = par["incl_sin"], par["incl_cos"]
    return p[0], p[2] * s - p[1] * c, v[1] * s + v[2] * c


def _bin(v, edges):
    e = torch.as_tensor(np.ascontiguousarray(edges), device=DEV)
    k = torch.searchsorted(e, v.contiguous(), right=True) - 1
    return torch.where((v >= e[0]) & (v < e[-1]), k, torch.full_like(k, -1))


def _kernels(obs, par, p, v):
    """Per set and moment: (first observable, cells, moments, kernel values or None for 1), cells -1 where none."""
    X, Ys, vl = _sky(par, p, v)
    off, out = 0, []
    for s in obs:
        if s.geom == "shell":
            c = _bin((p * p).sum(0), s.edges_x)
        elif s.geom == "annulus":
            c = _bin(X * X + Ys * Ys, s.edges_x)
        else:
            ix, iy = _bin(X, s.edges_x), _bin(Ys, s.edges_y)
            c = torch.where((ix >= 0) & (iy >= 0), iy * s.nx + ix, torch.full_like(ix, -1))
            if s.geom == "lut":
                t = torch.as_tensor(np.asarray(s.lut, np.int64).reshape(-1), device=DEV)
                c = torch.where(c >= 0, t[c.clamp(min=0)], c)
        ks = [None]
        if s.quant == "vlos2":
            ks = [vl * vl]
        elif s.quant == "gh":
            # van der Marel & Franx H_0..H_4, averaged over a Gaussian of the kernel's width
            q = c.clamp(min=0)
            S = torch.as_tensor(s.gh_S, device=DEV)[q]
            nu, t = (vl - torch.as_tensor(s.gh_V, device=DEV)[q]) / S, (s.sigma_kernel / S) ** 2
            d = 1.0 + t
            m, t2 = nu / d, t / d
            G = math.sqrt(2.0) / torch.sqrt(d) * torch.exp(-0.5 * nu * nu / d)
            E2, E3, E4 = m * m + t2, m ** 3 + 3 * m * t2, m ** 4 + 6 * m * m * t2 + 3 * t2 * t2
            ks = [G, G * (math.sqrt(2.0) * m), G * (2 * E2 - 1) / math.sqrt(2.0), G * (2 * E3 - 3 * m) / math.sqrt(3.0),
                  G * (4 * E4 - 12 * E2 + 3) / math.sqrt(24.0)]
        out.append((off, c, len(ks), ks))
        off += s.nobs
    return off, out


def _observe64(obs, par, p, v, w):
    """The observables (summed as integers of 2^-58, so that the same particles give the same sums) and kernels."""
    nobs, kern = _kernels(obs, par, p, v)
    y = torch.zeros(nobs, device=DEV, dtype=torch.int64)
    for off, c, nm, ks in kern:
        ok = c >= 0
        for j, K in enumerate(ks):
            t = w[ok] if K is None else (w * K)[ok]
            y.index_add_(0, off + c[ok] * nm + j, torch.round(t * 2.0 ** 58).to(torch.int64))
    return y.double() * 2.0 ** -58, kern


def _force(pot, p):
    a = torch.zeros_like(p)
    r = torch.sqrt((p * p).sum(0))
    for c in pot:
        if c.kind == "hernquist":
            a -= c.params[0] / (r * (r + c.params[1]) ** 2) * p
        elif c.kind == "nfw":
            u = r / c.params[1]
            a -= 4 * math.pi * c.params[0] * c.params[1] ** 3 * (torch.log1p(u) - u / (1 + u)) / r ** 3 * p
        else:
            v0, Rc, q = c.params
            f = v0 * v0 / (Rc * Rc + p[0] ** 2 + p[1] ** 2 + (p[2] / q) ** 2)
            a -= torch.stack([f * p[0], f * p[1], f * p[2] / (q * q)])
    return a


def _energy(pot, p, v):
    r = torch.sqrt((p * p).sum(0))
    E = 0.5 * (v * v).sum(0)
    for c in pot:
        if c.kind == "hernquist":
            E -= c.params[0] / (r + c.params[1])
        elif c.kind == "nfw":
            E -= 4 * math.pi * c.params[0] * c.params[1] ** 3 * torch.log1p(r / c.params[1]) / r
        else:
            v0, Rc, q = c.params
            E += 0.5 * v0 * v0 * torch.log(Rc * Rc + p[0] ** 2 + p[1] ** 2 + (p[2] / q) ** 2)
    return E


def _priors(d, p, v, w):
    pr, E = d["prior"], _energy(d["pot"], p, v)
    L = torch.stack([p[1] * v[2] - p[2] * v[1], p[2] * v[0] - p[0] * v[2], p[0] * v[1] - p[1] * v[0]])
    L2 = (L * L).sum(0)
    lo, hi = float(E.min()), float(E.max())
    if pr.kind == "e_lz":
        l, l1 = L[2], float(L[2].abs().max())
        l0 = -l1
    elif pr.kind == "e_l2":
        l, l0, l1 = L2, 0.0, float(L2.max())
    else:
        # L^2 of the circular orbit of the same energy in a Hernquist sphere of GM = a = 1
        hi = 0.0
        e = torch.clamp(E, max=-1e-300)
        s = (-1.0 - torch.sqrt(1.0 - 8.0 * e)) / (4.0 * e)
        l, l0, l1 = L2 / ((s - 1.0) ** 3 / (s * s)), 0.0, 1.0
    def cell(q, a, b, m):
        return torch.searchsorted(torch.as_tensor(a + np.arange(1, m) * ((b - a) / m), device=DEV), q, right=True)
    c = cell(E, lo, hi, pr.nE) * pr.nL + cell(l, l0, l1, pr.nL)
    if pr.kind == "e_lc":
        c = torch.where(E >= 0, torch.full_like(c, pr.nE * pr.nL), c)
    sums = torch.zeros(pr.nE * pr.nL + 1, device=DEV, dtype=torch.float64).index_add_(0, c, w)
    return (sums / torch.bincount(c, minlength=sums.numel()).clamp(min=1))[c]


def _steps64(d, f32, steps, lazy):
    cast = (lambda t: t.float().double()) if f32 else (lambda t: t.clone())
    p, v, w, what = cast(d["pos"]), cast(d["vel"]), d["w"].clone(), d["what"].clone()
    par, Y, sg = d["par"], torch.as_tensor(d["Y"], device=DEV), torch.as_tensor(d["sigma"], device=DEV)
    inv = torch.where(sg > 0, 1.0 / sg, torch.zeros_like(sg))
    y, _ = _observe64(d["obs"], par, p, v, w)
    Dt = (y - Y) * inv
    rec = None
    for t in range(1, steps + 1):
        v = v + 0.5 * DT * _force(d["pot"], p)
        p = p + DT * v
        v = v + 0.5 * DT * _force(d["pot"], p)
        y, kern = _observe64(d["obs"], par, p, v, w)
        D = (y - Y) * inv
        Dt = ALPHA * D + (1.0 - ALPHA) * Dt
        rec = dict(chi2=float((Dt * Dt).sum()), chi2_raw=float((D * D).sum()), max_abs_dt=float(Dt.abs().max()),
                   S=float(-(w * torch.log(w / what)).sum()), sum_w=float(w.sum()))
        if not (lazy and t == steps):
            G = MU * (-torch.log(w / what) - ENT)
            cf = Dt * inv
            for off, c, nm, ks in kern:
                ok = c >= 0
                for j, K in enumerate(ks):
                    k = cf[off + c.clamp(min=0) * nm + j]
                    G = G - torch.where(ok, k if K is None else k * K, torch.zeros_like(k))
            w = w * torch.exp(par["eps"] * DT * G)
            if d["prior"].kind != "flat" and t % PERIOD == 0:
                what = _priors(d, p, v, w)
    return dict(zip(ARRAYS, [*p, *v, w, what])), rec, (y, D, Dt)


def exact(case, seed):
    """The call in 64 bits with plain torch.  None where orbits run in the expansion of the particles: those through
    the centre amplify the state's own rounding by orders of magnitude within a period, so 64-bit orbits are other
    orbits; and with seeing, whose draws are the library's generator's."""
    f32 = case["prec"] == "fp32c"
    if case["work"].startswith("sh-") or case["work"] == "ifu-lut-seeing":
        return None
    if case["call"] == "batch":
        runs = [_steps64(d, f32, case["steps"], False) for d in _batch_models(case, seed)]
        out = {k: torch.cat([r[0][k] for r in runs]) for k in ARRAYS}
        out["chi2"], out["S"] = np.array([r[1]["chi2"] for r in runs]), np.array([r[1]["S"] for r in runs])
        return out
    d = _workload(case, seed)
    if case["call"] == "moments":
        p, v = (t.float().double() if f32 else t for t in (d["pos"], d["vel"]))
        r, R = torch.sqrt((p * p).sum(0)), torch.sqrt(p[0] ** 2 + p[1] ** 2)
        vr, vp = (p * v).sum(0) / r, (p[0] * v[1] - p[1] * v[0]) / R
        q = p.float() if f32 else p           # the shell is decided in the state's precision
        c = _bin(((q[0] * q[0] + q[1] * q[1]) + q[2] * q[2]).double(), np.geomspace(0.2, 5.0, 9) ** 2)
        ok = c >= 0
        out = torch.zeros(8, 4, device=DEV, dtype=torch.float64)
        for k, t in enumerate((torch.ones_like(r), vr * vr, ((v * v).sum(0) - vr * vr) - vp * vp, vp * vp)):
            out[:, k].index_add_(0, c[ok], (d["w"] * t)[ok])
        return out
    if case["call"] == "observe":
        p, v = (t.float().double() if f32 else t for t in (d["pos"], d["vel"]))
        y = _observe64(d["obs"], d["par"], p, v, d["w"])[0]
        sg = torch.as_tensor(d["sigma"], device=DEV)
        D = torch.where(sg > 0, (y - torch.as_tensor(d["Y"], device=DEV)) / sg, torch.zeros_like(sg))
        return [y, D, D.clone()]
    st, rec, o = _steps64(d, f32, case["steps"], case["call"] == "loop")
    out = dict(st, record=rec)
    if case["call"] == "step":
        out["obs"] = list(o)
    return out
