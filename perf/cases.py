"""The work that users of the charging library have it do, as measurable cases.

A case is one call, or one short run of calls, through the package's public
entry points (Channel, Particles, Batch, mean_charge, tribo_poisson_noalloc):
coupled particle steps, Poisson solves, the adjoint, batched ensembles.  Sizes
are those of the workloads of `synth` and of the tests, and their
neighbourhood: every transform length 2^a 3^b the library takes, wall-normal
cell counts of any parity, particle counts from a few thousand to millions.

Inputs are those of a developed channel flow: tanh-stretched grid, Reichardt
mean profile with random Fourier modes damped at the walls, particles in cell
order (the order a simulation that sorts holds them in) carrying Gaussian
charges and velocities that fluctuate with the friction velocity, so that some
of them meet a wall in every step.  They are made on the GPU with torch from
the seed alone.  `exact` restates the method in plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_10761_gb300 as T

DELTA = 0.02            # channel half height [m]
NU, RHO = 1.46e-5, 1.2  # air
Q_SAT = 1.26e-13        # saturation charge of the reference particle [C]
LX, LY, LZ = 2 * math.pi * DELTA, 2 * DELTA, math.pi * DELTA
EPS = 8.854e-12
N_MODES = 256
# material constants of particles and wall, reference impact of the stochastic scaling model
MATERIAL = dict(mu_p=0.4, E_p=1e8, phi_p=1e13, k_e=0.95, mu_w=0.28, E_w=1e11, eps_w=5.0, h=1e-9, eps=EPS, eps0=EPS)
SSM = dict(r0=2e-4, un0=0.925, mu0=-4.12e-15, sigma0=6.49e-15, gamma0=-0.191, dq0_min=-2.19e-14, c_sat=500e-6, seed=7)
F64 = torch.float64
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases

def _step(name, nx, ny, nz, n, re_tau=180.0, dlo=1.0, dhi=1.0, ratio=1000.0, fp64=False, steps=20, sort=20,
          moving=False, sn=False, ssm=False, two_way=False, pairs=False, host=False):
    return dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, n=n, re_tau=re_tau, dlo=dlo, dhi=dhi, ratio=ratio,
                fp64=fp64, steps=steps, sort=sort, moving=moving, sn=sn, ssm=ssm, two_way=two_way, pairs=pairs,
                host=host)


def listed():
    return [
        # one coupled step per call of the small FP64 channel, as a gas solver that steps
        # with the particles calls it: the shortest call, all launches and latency
        _step("step_fp64_64", 64, 64, 64, 2000, fp64=True, steps=1, sort=0),
        # a production run of the plain FP64 method at a million particles
        _step("step_fp64_128", 128, 128, 128, 1_000_000, fp64=True),
        # mixed precision, polydisperse particles in a time-varying gas field
        _step("step_re180_128", 128, 128, 128, 1_000_000, dlo=0.5, dhi=2.0, moving=True),
        # the headline workload: Re_tau 550, 8M particles, one sort period per pass
        _step("step_re550_384", 384, 256, 256, 8_000_000, re_tau=550.0, dlo=2.5, dhi=2.5, ratio=2000.0),
        # 2-way coupling with the nonlinear drag and the stochastic charging model on a grid of
        # odd height whose transform lengths have factors 9 (the DNS heights are not powers of two)
        _step("step_two_way", 144, 101, 72, 300_000, re_tau=300.0, dlo=0.5, dhi=3.0, sn=True, ssm=True, two_way=True),
        # 4-way coupling: in-cell Coulomb forces and collisions of heavier loading
        _step("step_pairs", 128, 128, 128, 1_000_000, steps=5, sort=0, pairs=True),
        # a program that keeps its particles in host memory, one step per call
        _step("step_host", 128, 128, 128, 1_000_000, steps=1, sort=0, host=True),
        # stand-alone field solves: mixed precision on a ragged grid, FP64 with the potential,
        # and the solve of a caller that must not allocate
        dict(name="poisson_ragged", kind="poisson", nx=288, ny=145, nz=162, fp64=False, phi=False, noalloc=False),
        dict(name="poisson_fp64", kind="poisson", nx=192, ny=128, nz=128, fp64=True, phi=True, noalloc=False),
        dict(name="poisson_noalloc", kind="poisson", nx=64, ny=64, nz=64, fp64=False, phi=False, noalloc=True),
        # one iteration of a calibration: the mean charge and its gradients, from the same
        # starting ensemble each time
        dict(name="adjoint_re180_128", kind="adjoint", nx=128, ny=128, nz=128, n=1_000_000, re_tau=180.0, fp64=False,
             sn=False, steps=12, ckpt=4),
        # a sweep over friction Reynolds numbers and diameters, two sort periods per pass
        dict(name="batch_ensemble", kind="batch", channels=10, scale=0.25, fp64=False, steps=40, sort=20),
    ]


_LENGTHS = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384]
_MOST_CELLS = 384 * 256 * 256


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, most):
    """Transform lengths 2^a 3^b (nx even) and any height, between lo and `most` cells."""
    while True:
        nx, nz = rng.choice(_LENGTHS), rng.choice(_LENGTHS)
        ny = _log(rng, 24, 256)
        if nx >= nz and lo <= nx * ny * nz <= most:
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(["step", "step", "step", "poisson", "poisson", "adjoint", "batch"])
    fp64 = rng.random() < 0.3
    most = 128 ** 3 if fp64 else _MOST_CELLS
    if kind == "poisson":
        noalloc = rng.random() < 0.25
        nx, ny, nz = _grid(rng, 16 * 1024, (64 ** 3 if fp64 else 80 ** 3) if noalloc else 2 * most if fp64 else most)
        if noalloc and max(nx, ny, nz) > 256:
            nx, ny, nz = 96, ny % 64 + 24, 36
        return dict(kind="poisson", nx=nx, ny=ny, nz=nz, fp64=fp64, phi=fp64 and rng.random() < 0.5, noalloc=noalloc)
    if kind == "batch":
        return dict(kind="batch", channels=rng.randint(3, 10), scale=round(math.exp(rng.uniform(-4.0, -1.5)), 4),
                    fp64=False, steps=40, sort=20)
    nx, ny, nz = _grid(rng, 16 * 1024, most if kind == "step" else 128 ** 3)
    cells = nx * ny * nz
    n = max(1000, min(1_000_000 if fp64 else 8_000_000, int(cells * math.exp(rng.uniform(math.log(0.02), math.log(0.7))))))
    re_tau = rng.choice([180.0, 300.0, 395.0, 550.0])
    if kind == "adjoint":
        return dict(kind="adjoint", nx=nx, ny=ny, nz=nz, n=min(n, 1_000_000), re_tau=re_tau, fp64=False,
                    sn=rng.random() < 0.5, steps=rng.randint(4, 12), ckpt=rng.choice([2, 4, 5]))
    c = _step("", nx, ny, nz, n, re_tau=re_tau, dlo=round(rng.uniform(0.5, 1.5), 3), dhi=round(rng.uniform(1.5, 3.0), 3),
              ratio=rng.choice([1000.0, 2000.0]), fp64=fp64, sn=rng.random() < 0.4)
    del c["name"]
    use = rng.choice(["plain", "plain", "moving", "ssm", "two_way", "pairs", "host", "single"])
    if use in ("moving", "ssm", "two_way"):
        c[use] = cells <= 192 * 128 * 128
    elif use == "pairs":
        c.update(pairs=True, steps=5, sort=0, n=min(n, 1_000_000))
    elif use == "host":
        c.update(host=True, steps=1, sort=0)
    elif use == "single":
        c.update(steps=1, sort=0)
    return c


# ---------------------------------------------------------------------------
# inputs (torch, FP64, from the seed)

def _faces(ny):
    j = np.arange(ny + 1, dtype=np.float64)
    f = DELTA * (1.0 - np.tanh(2.0 * (1.0 - 2.0 * j / ny)) / math.tanh(2.0))
    f[0], f[-1] = 0.0, LY
    return f


def _nodes(f):
    return np.concatenate(([f[0]], 0.5 * (f[1:] + f[:-1]), [f[-1]]))


def _u_tau(re_tau):
    return re_tau * NU / DELTA


def _wall_plus(y, re_tau, lib):
    yw = lib.minimum(y, LY - y)
    return yw * (_u_tau(re_tau) / NU)


def _mean_velocity(y, re_tau, lib=np):
    yp = _wall_plus(y, re_tau, lib)
    return _u_tau(re_tau) * (lib.log1p(0.41 * yp) / 0.41
                             + 7.8 * (1.0 - lib.exp(-yp / 11.0) - (yp / 11.0) * lib.exp(-yp / 3.0)))


class _Modes:
    """Random Fourier modes, perpendicular to their wave vector, von Karman weights."""

    def __init__(self, nx, nz, re_tau, rng):
        lk = rng.uniform(math.log(2 * math.pi / LX), math.log(math.pi * nx / LX), N_MODES)
        k = np.exp(lk)
        mu, ang = rng.uniform(-1.0, 1.0, N_MODES), rng.uniform(0.0, 2 * math.pi, N_MODES)
        s = np.sqrt(1.0 - mu * mu)
        self.nxi = np.clip(np.rint(k * s * np.cos(ang) * LX / (2 * math.pi)), 1 - nx // 2, nx // 2 - 1).astype(np.int32)
        self.nzi = np.clip(np.rint(k * s * np.sin(ang) * LZ / (2 * math.pi)), 1 - nz // 2, nz // 2 - 1).astype(np.int32)
        self.ky = k * mu
        kv = np.stack([2 * math.pi * self.nxi / LX, self.ky, 2 * math.pi * self.nzi / LZ], 1)
        kn = np.maximum(np.linalg.norm(kv, axis=1), 1e-30)
        g = rng.standard_normal((N_MODES, 3))
        kh = kv / kn[:, None]
        a = g - (g * kh).sum(1)[:, None] * kh
        a /= np.linalg.norm(a, axis=1)[:, None]
        kr = kn / (2 * math.pi / DELTA)
        amp = a * (rng.standard_normal(N_MODES) * np.sqrt(kr ** 4 / (1 + kr ** 2) ** (17 / 6) * kn))[:, None]
        self.amp = amp * math.sqrt(6.0 * _u_tau(re_tau) ** 2 / (amp ** 2).sum())
        self.phase = rng.uniform(0.0, 2 * math.pi, N_MODES)


def _profiles(Y, re_tau):
    """Mean velocity and damping factor at the lattice y nodes."""
    yp = _wall_plus(Y, re_tau, np)
    ub, damp = _mean_velocity(Y, re_tau), yp / (yp + 10.0)
    for v in (ub, damp):
        v[0] = v[-1] = 0.0
    return ub, damp


def _lattice(m, Y, nx, nz, re_tau, t=0.0):
    """Gas velocity on the lattice at time t: (nz, ny+2, nx, 3), FP64."""
    ub, damp = _profiles(Y, re_tau)
    dev = dict(device=DEV)
    kx = 2 * math.pi * m.nxi / LX
    ph = m.ky[None] * Y[:, None] + m.phase[None] - kx[None] * ub[:, None] * t
    ph = ph + math.pi * (m.nxi / nx + m.nzi / nz)[None]
    coef = torch.polar(torch.as_tensor(np.broadcast_to(damp[:, None], ph.shape).copy(), **dev),
                       torch.as_tensor(ph, **dev))
    at = torch.as_tensor(np.mod(m.nzi, nz).astype(np.int64) * nx + np.mod(m.nxi, nx), **dev)
    amp = torch.as_tensor(m.amp, **dev)
    out = torch.empty((nz, len(Y), nx, 3), dtype=F64, **dev)
    for c in range(3):
        # modes that share a wavenumber are added on the host side of the scatter, in order
        spec = torch.zeros((len(Y), nz * nx), dtype=torch.complex128, **dev)
        one = torch.zeros((N_MODES, N_MODES), dtype=F64, **dev)
        uniq, inv = torch.unique(at, return_inverse=True)
        one[torch.arange(N_MODES, **dev), inv] = 1.0
        spec[:, uniq] = ((coef * amp[:, c]) @ one.to(torch.complex128))[:, :len(uniq)]
        out[..., c] = torch.fft.ifft2(spec.view(len(Y), nz, nx)).real.permute(1, 0, 2) * (nx * nz)
    out[..., 0] += torch.as_tensor(ub, **dev)[None, :, None]
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _cells(x, y, z, nx, nz, yf):
    i = (x / (LX / nx)).floor().long().clamp_(0, nx - 1)
    k = (z / (LZ / nz)).floor().long().clamp_(0, nz - 1)
    j = (torch.searchsorted(yf, y.contiguous(), right=True) - 1).clamp_(0, len(yf) - 2)
    return (k * (len(yf) - 1) + j) * nx + i


def _inputs(c, seed):
    """Grid, gas field and particles of one channel, in the values the library is given."""
    real = F64 if c["fp64"] else torch.float32
    rng = np.random.Generator(np.random.Philox(seed))
    g = _gen(seed)
    nx, ny, nz, n, re_tau = c["nx"], c["ny"], c["nz"], c["n"], c["re_tau"]
    f = _faces(ny)
    ut = _u_tau(re_tau)
    s = dict(faces=f, Y=_nodes(f), dt=0.05 * NU / ut ** 2, rho_p=c.get("ratio", 1000.0) * RHO)
    s["modes"] = _Modes(nx, nz, re_tau, rng)
    s["u"] = _lattice(s["modes"], s["Y"], nx, nz, re_tau).to(real)
    r = lambda: torch.rand(n, dtype=F64, device=DEV, generator=g)  # noqa: E731
    w = lambda: torch.randn(n, dtype=F64, device=DEV, generator=g)  # noqa: E731
    lo, hi = math.log(c.get("dlo", 1.0)), math.log(c.get("dhi", 1.0))
    d = torch.exp(lo + (hi - lo) * r()) * (NU / ut)
    x, z = LX * r(), LZ * r()
    y = 0.5 * d + (LY - d) * r()
    p = dict(x=x, y=y, z=z, vx=_mean_velocity(y, re_tau, torch) + 0.5 * ut * w(), vy=0.5 * ut * w(), vz=0.5 * ut * w(),
             d=d, q=0.01 * Q_SAT * w())
    p = {k: v if k == "q" else v.to(real) for k, v in p.items()}
    top = torch.tensor(LX, dtype=real, device=DEV), torch.tensor(LZ, dtype=real, device=DEV)
    p["x"], p["z"] = (torch.where(p[k] >= t, torch.zeros_like(p[k]), p[k]) for k, t in zip(("x", "z"), top))
    order = torch.argsort(_cells(p["x"].to(F64), p["y"].to(F64), p["z"].to(F64), nx, nz, torch.as_tensor(f, device=DEV)),
                          stable=True)
    s["p"] = {k: v[order].contiguous() for k, v in p.items()}
    if c.get("ssm"):
        s["p"]["site"] = 0.5 + 0.5 * r()
    return s


def _density(c, seed):
    """A charge density of both signs, as cell sums of particle charges give it."""
    g = _gen(seed)
    shape = (c["nz"], c["ny"], c["nx"])
    rho = torch.randn(shape, dtype=F64, device=DEV, generator=g)
    rho *= torch.rand(shape, dtype=F64, device=DEV, generator=g) < 0.3
    dy = torch.as_tensor(np.diff(_faces(c["ny"])), device=DEV)
    return rho * (0.01 * Q_SAT) / ((LX / c["nx"]) * (LZ / c["nz"]) * dy[None, :, None])


# ---------------------------------------------------------------------------
# what a user's program keeps, and one pass

def _params(c, rho_p, **kw):
    return T.Params(precision=T.TRIBO_FP64 if c["fp64"] else T.TRIBO_MIXED, rho_p=rho_p, nu=NU, rho=RHO, **MATERIAL,
                    drag_law=T.TRIBO_DRAG_SCHILLER_NAUMANN if c.get("sn") else T.TRIBO_DRAG_STOKES, **kw)


def _particles(p):
    n = p["x"].shape[0]
    dev = dict(device=DEV)
    return T.Particles(q_wall=torch.zeros(n, dtype=F64, **dev), n_imp=torch.zeros(n, dtype=torch.int32, **dev),
                       id=torch.arange(n, dtype=torch.int32, **dev), **p)


def _pinned(v):
    h = torch.empty(v.shape, dtype=v.dtype, pin_memory=True)
    h.copy_(v)
    return h.numpy()


_STATE = ("x", "y", "z", "vx", "vy", "vz", "q", "q_wall", "n_imp")


def prepare(case, seed):
    c = case
    if c["kind"] == "poisson":
        s = dict(c=c, rho=_density(c, seed), faces=_faces(c["ny"]))
        if c["noalloc"]:
            real = F64 if c["fp64"] else torch.float32
            s["E"] = torch.zeros((3, c["nz"], c["ny"] + 2, c["nx"]), dtype=real, device=DEV)
            s["phi"] = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=F64, device=DEV) if c["phi"] else None
        else:
            s["ch"] = T.Channel(c["nx"], c["ny"], c["nz"], LX, LZ, s["faces"], _params(c, 1000.0 * RHO))
        return s
    if c["kind"] == "batch":
        parts = _batch_cases(c, seed)
        chans, P, dt = [], [], []
        for k, b in enumerate(parts):
            i = _inputs(b, seed + 1000 * (k + 1))
            chans.append(T.Channel(b["nx"], b["ny"], b["nz"], LX, LZ, i["faces"],
                                   _params(b, i["rho_p"], sort_every=c["sort"]), i["u"], max_particles=b["n"]))
            P.append(_particles(i["p"]))
            dt.append(i["dt"])
        first = np.cumsum([0] + [p.n for p in P[:-1]])
        batch = T.Batch(chans, sort_every=c["sort"])
        batch.autotune(P, dt)
        return dict(c=c, batch=batch, chans=chans, P=P, dt=dt, first=[int(v) for v in first])
    i = _inputs(c, seed)
    kw = dict(sort_every=c["sort"], coulomb=int(c["pairs"]), collisions=int(c["pairs"])) if c["kind"] == "step" else {}
    ch = T.Channel(c["nx"], c["ny"], c["nz"], LX, LZ, i["faces"], _params(c, i["rho_p"], **kw), i["u"],
                   max_particles=c["n"])
    P = _particles(i["p"])
    s = dict(c=c, ch=ch, P=P, dt=i["dt"])
    if c["kind"] == "adjoint":
        s["one"] = torch.tensor(1.0)
        return s
    if c["moving"]:
        ch.set_modes(i["modes"], *_profiles(i["Y"], c["re_tau"]))
    if c["ssm"]:
        ch.set_ssm(T.SSMParams(**SSM))
    if c["two_way"]:
        s["F_s"] = ch.momentum_source()
    if c["host"]:
        s["P"] = T.Particles(**{k: _pinned(getattr(P, k)) for k in P.ALL if getattr(P, k) is not None})
    return s


def run(state):
    s = state
    c = s["c"]
    if c["kind"] == "poisson":
        if c["noalloc"]:
            T.tribo_poisson_noalloc(c["nx"], c["ny"], c["nz"], LX, LZ, s["faces"], EPS,
                                    T.TRIBO_FP64 if c["fp64"] else T.TRIBO_MIXED, s["rho"], s["phi"], s["E"])
            return dict(E=s["E"], phi=s["phi"])
        phi, E = s["ch"].poisson(s["rho"], want_phi=c["phi"])
        return dict(E=E, phi=phi)
    if c["kind"] == "adjoint":
        p = T.Particles(**{k: getattr(s["P"], k).clone() for k in s["P"].ALL if getattr(s["P"], k) is not None})
        U, K = s["one"].clone().requires_grad_(), s["one"].clone().requires_grad_()
        d = s["P"].d.clone().requires_grad_()
        J = T.mean_charge(s["ch"], p, s["dt"], c["steps"], U, K, d, c["ckpt"])
        dU, dK, dd = torch.autograd.grad(J, (U, K, d))
        return dict(J=float(J), dU=dU, dK=dK, dd=dd, y=p.y, vx=p.vx, q=p.q)
    if c["kind"] == "batch":
        s["batch"].step(s["P"], s["dt"], c["steps"])
        ids = torch.cat([p.id + f for p, f in zip(s["P"], s["first"])]).long()
        return {k: _by_id(torch.cat([getattr(p, k) for p in s["P"]]), ids) for k in _STATE}
    P = s["P"]
    s["ch"].step(P, s["dt"], c["steps"])
    if c["sort"]:
        # a sorting run hands its results out by particle
        ids = P.id.long()
        out = {k: _by_id(getattr(P, k), ids) for k in _STATE}
        if c["ssm"]:
            out["site"] = _by_id(P.site, ids)
    else:
        out = {k: getattr(P, k) for k in _STATE + (("site",) if c["ssm"] else ())}
    if c["two_way"]:
        out["F_s"] = s["F_s"]
    return out


def _by_id(v, ids):
    return torch.empty_like(v).index_copy_(0, ids, v)


_SWEEP_GRIDS = [(64, 64, 64), (96, 64, 64), (128, 96, 96), (128, 128, 128), (192, 128, 128)]


def _batch_cases(c, seed):
    """The channels of a sweep: uneven grids, counts, Re_tau and diameters (the sizes follow the
    case, the values the seed)."""
    rng = np.random.Generator(np.random.Philox(1004))
    out = []
    for _ in range(c["channels"]):
        nx, ny, nz = _SWEEP_GRIDS[int(rng.integers(len(_SWEEP_GRIDS)))]
        d = float(rng.uniform(0.5, 3.0))
        out.append(dict(nx=nx, ny=ny, nz=nz, n=max(1, int(rng.uniform(50_000, 2_000_000) * c["scale"])), fp64=c["fp64"],
                        re_tau=float(rng.choice([180.0, 300.0, 395.0, 550.0])), dlo=d, dhi=d, ratio=1000.0))
    return out


def work(case):
    """Bytes and operations a pass cannot do without: per step, the particle state read and
    written, the lattice nodes the particles touch, the charge sums and the field once each;
    transforms at 5 N log2 N operations per complex length-N line."""
    c = case
    if c["kind"] == "batch":
        w = [work(dict(b, kind="step", steps=c["steps"], moving=False)) for b in _batch_cases(c, 0)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    R = 8 if c["fp64"] else 4
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    cells, nodes = nx * ny * nz, nx * (ny + 2) * nz
    # half spectrum: 1 forward and 3 inverse transforms of cells/2 complex values, 4 y recurrences
    solve_flops = 4 * 2.5 * cells * math.log2(nx * nz) + 30 * cells
    if c["kind"] == "poisson":
        return dict(bytes=8 * cells + 3 * R * nodes + (8 * cells if c["phi"] else 0), flops=solve_flops)
    n, steps = c["n"], c["steps"]
    touched = nodes * -math.expm1(-8.0 * n / nodes)
    particle = n * (7 * R + 8 + 6 * R) + touched * 6 * R
    field = 8 * cells + 3 * R * nodes
    if c["kind"] == "adjoint":
        # forward, and a reverse step (state, adjoints, field adjoint, one solve) per step
        back = n * (7 * R + 8 + 2 * (6 * R + 8) + 16) + touched * 9 * R + 8 * cells
        return dict(bytes=steps * (particle + field + back), flops=steps * (2 * solve_flops + 1200 * n))
    modes = N_MODES * 10.0 * nodes if c["moving"] else 0.0
    return dict(bytes=steps * (particle + field + (3 * R * nodes if c["moving"] else 0)),
                flops=steps * (solve_flops + 300 * n + modes))


# ---------------------------------------------------------------------------
# the method in plain FP64 torch

class _Values:
    def __init__(self, **kw):
        self.__dict__.update(kw)


class _Field:
    """Poisson solve with grounded walls and E = -grad(phi) on the wall-extended lattice."""

    def __init__(self, nx, ny, nz, f):
        t = lambda v: torch.as_tensor(v, device=DEV)  # noqa: E731
        self.n = nx, ny, nz
        yc, dy = 0.5 * (f[1:] + f[:-1]), np.diff(f)
        a, c = np.zeros(ny), np.zeros(ny)
        a[1:] = 1 / (dy[1:] * np.diff(yc))
        c[:-1] = 1 / (dy[:-1] * np.diff(yc))
        b = -(a + c)
        self.h0, self.h1 = yc[0] - f[0], f[-1] - yc[-1]
        b[0] -= 1 / (dy[0] * self.h0)
        b[-1] -= 1 / (dy[-1] * self.h1)
        lam = lambda n, h, m: 4 / h ** 2 * np.sin(math.pi * np.arange(m) / n) ** 2  # noqa: E731
        L = t(lam(nz, LZ / nz, nz)[:, None] + lam(nx, LX / nx, nx // 2 + 1)[None])
        self.a = a
        self.inv, self.cp = [], []
        cp = torch.zeros_like(L)
        for j in range(ny):
            inv = 1 / ((b[j] - L) - a[j] * cp)
            cp = c[j] * inv
            self.inv.append(inv)
            self.cp.append(cp)
        self.w = t((f[1:-1] - yc[:-1]) / np.diff(yc))[None, :, None]     # interior faces
        self.dy = t(dy)[None, :, None]

    def phi(self, rho):
        nx, ny, nz = self.n
        s = torch.fft.fft(torch.fft.rfft(-rho / EPS, dim=2), dim=0).unbind(1)
        d = []
        for j in range(ny):
            d.append((s[j] - self.a[j] * d[-1]) * self.inv[j] if j else s[j] * self.inv[j])
        x = [d[-1]]
        for j in range(ny - 2, -1, -1):
            x.append(d[j] - self.cp[j] * x[-1])
        return torch.fft.irfft(torch.fft.ifft(torch.stack(x[::-1], 1), dim=0), n=nx, dim=2)

    def E(self, phi):
        nx, ny, nz = self.n
        zero = torch.zeros_like(phi[:, :1])
        pad = lambda v: torch.cat([zero, v, zero], 1)  # noqa: E731
        ex = (phi.roll(1, 2) - phi.roll(-1, 2)) * (nx / (2 * LX))
        ez = (phi.roll(1, 0) - phi.roll(-1, 0)) * (nz / (2 * LZ))
        face = pad((1 - self.w) * phi[:, :-1] + self.w * phi[:, 1:])
        ey = torch.cat([-phi[:, :1] / self.h0, -(face[:, 1:] - face[:, :-1]) / self.dy, phi[:, -1:] / self.h1], 1)
        return torch.stack([pad(ex), ey, pad(ez)])


def _gather(planes, st, c, Y):
    """Trilinear interpolation of (3, nz, ny+2, nx) planes at the particles."""
    nx, nz, nyn = c["nx"], c["nz"], len(Y)
    x, y, z = (st[k] for k in ("x", "y", "z"))
    sx, sz = x * (nx / LX) - 0.5, z * (nz / LZ) - 0.5
    i, k = sx.detach().floor().long(), sz.detach().floor().long()
    j = (torch.searchsorted(Y, y.detach().contiguous(), right=True) - 1).clamp_(0, nyn - 2)
    wx, wz = sx - i, sz - k
    wy = (y - Y[j]) / (Y[j + 1] - Y[j])
    flat = planes.reshape(3, -1)
    out = [0.0, 0.0, 0.0]
    for b in range(8):
        bx, by, bz = b & 1, b >> 1 & 1, b >> 2
        at = (((k + bz) % nz) * nyn + j + by) * nx + (i + bx) % nx
        w = (wx if bx else 1 - wx) * (wy if by else 1 - wy) * (wz if bz else 1 - wz)
        for q in range(3):
            out[q] = out[q] + w * flat[q][at]
    return out


def _elastic(P):
    return (1 - P.mu_p ** 2) / P.E_p + (1 - P.mu_w ** 2) / P.E_w


def _impact(P, d, speed, q, U, K):
    r = 0.5 * d
    alpha = r * (0.625 * math.pi * P.rho_p * (1 + P.k_e) * _elastic(P) * speed ** 2) ** 0.4
    A = K * math.pi * r * alpha
    dq = P.eps / P.h * A * U * torch.expm1(-2.94 * alpha / speed / (P.eps_w * P.eps0 * P.phi_p))
    return dq - A / (math.pi * d * d) * q


def _philox(ids, count, key):
    M = 0xFFFFFFFF
    c0, c1, c2, c3 = ids & M, count & M, torch.zeros_like(ids), torch.zeros_like(ids)
    k0, k1 = key & M, key >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M) ^ c1 ^ k0, p1 & M, ((p0 >> 32) & M) ^ c3 ^ k1, p0 & M
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1


def _ssm(P, m, d, speed, q, ids, count, site):
    """Charge and new site density of stochastic-scaling-model impacts."""
    coef = 0.625 * math.pi * P.rho_p * (1 + P.k_e) * _elastic(P)
    A = math.pi * (0.5 * d) ** 2 * (coef * speed ** 2) ** 0.4
    area = A / (math.pi * m.r0 ** 2 * (coef * m.un0 ** 2) ** 0.4)
    x = 4 * q / (m.c_sat * d * d)
    sw, di = math.copysign(1, m.dq0_min), m.dq0_min - m.mu0
    chi_w, chi_i = (1 - sw * x).clamp(0, 1), (1 + math.copysign(1, di) * x).clamp(0, 1)
    ni = area * chi_i * site
    new = (site * (1 - A / (math.pi * d * d) * chi_i * sw * x)).clamp(0, 1)
    g = torch.where(ni > 0, -m.gamma0 / ni, torch.zeros_like(ni)).clamp(-0.99, 0.99)
    ag = g.abs() ** (2 / 3)
    delta = g.sign() * (math.pi / 2 * ag / ((0.5 * (4 - math.pi)) ** (2 / 3) + ag)).sqrt()
    omega = m.sigma0 * ni.sqrt() / (1 - 2 * delta ** 2 / math.pi).sqrt()
    xi = di * ni - omega * delta * math.sqrt(2 / math.pi)
    w0, w1 = _philox(ids, count, m.seed)
    rad = (-2 * ((w0 + 0.5) * 2.0 ** -32).log()).sqrt()
    ang = 2 * math.pi * (w1 + 0.5) * 2.0 ** -32
    y = xi + omega * (delta * (rad * ang.cos()).abs() + (1 - delta ** 2).clamp(min=0).sqrt() * rad * ang.sin())
    return m.dq0_min * area * chi_w - y, new


def _near_field(st, key, P):
    """In-cell Coulomb acceleration: pairs at every distance in the cell-ordered list."""
    order = torch.argsort(key, stable=True)
    ks, acc = key[order], torch.zeros((3, len(key)), dtype=F64, device=DEV)
    pos = torch.stack([st[k] for k in ("x", "y", "z")])[:, order]
    q = st["q"][order]
    for i, j in _pairs(ks):
        r = pos[:, i] - pos[:, j]
        r2 = (r * r).sum(0)
        f = torch.where(r2 > 0, r2 ** -1.5, torch.zeros_like(r2)) * r
        acc.index_add_(1, i, q[j] * f)
        acc.index_add_(1, j, -q[i] * f)
    out = torch.empty_like(acc)
    out[:, order] = acc
    return out * (st["q"] / (4 * math.pi * P.eps * (math.pi / 6 * P.rho_p) * st["d"] ** 3))


def _pairs(ks):
    o = 1
    while o < len(ks):
        i = (ks[o:] == ks[:-o]).nonzero()[:, 0]
        if not len(i):
            return
        yield i, i + o
        o += 1


def _collide(st, key, P):
    """Elastic collisions of mutually nearest overlapping, approaching pairs of a cell."""
    n = len(key)
    order = torch.argsort(key, stable=True)
    ks = key[order]
    s = {k: v[order] for k, v in st.items() if k in _STATE + ("d",)}
    pos, vel = (torch.stack([s[k] for k in t]) for t in (("x", "y", "z"), ("vx", "vy", "vz")))
    near = torch.full((n,), math.inf, dtype=F64, device=DEV)
    mate = torch.full((n,), -1, dtype=torch.long, device=DEV)
    found = []
    for i, j in _pairs(ks):
        r, v = pos[:, i] - pos[:, j], vel[:, i] - vel[:, j]
        d2 = (r * r).sum(0)
        ok = (d2 < (0.5 * (s["d"][i] + s["d"][j])) ** 2) & ((r * v).sum(0) < 0)
        found.append((i[ok], j[ok], d2[ok]))
    if not found:
        return
    i, j, d2 = (torch.cat(v) for v in zip(*found))
    for a in (i, j):
        near.scatter_reduce_(0, a, d2, "amin")
    for a, b in ((i, j), (j, i)):
        m = d2 == near[a]
        mate[a[m]] = b[m]
    i = ((mate >= 0) & (mate[mate.clamp(min=0)] == torch.arange(n, device=DEV))).nonzero()[:, 0]
    i = i[mate[i] > i]
    j = mate[i]
    r, v = pos[:, i] - pos[:, j], vel[:, i] - vel[:, j]
    e = r / (r * r).sum(0).sqrt()
    di, dj, qi, qj = s["d"][i], s["d"][j], s["q"][i], s["q"][j]
    vn = (v * e).sum(0)
    vel[:, i] -= 2 * dj ** 3 / (di ** 3 + dj ** 3) * vn * e
    vel[:, j] += 2 * di ** 3 / (di ** 3 + dj ** 3) * vn * e
    sp = (v * v).sum(0).sqrt()
    Ci, Cj = 2 * math.pi * P.eps * di, 2 * math.pi * P.eps * dj
    el = 2 * (1 - P.mu_p ** 2) / P.E_p
    alpha = 0.5 * di * dj * (0.625 * math.pi * P.rho_p * (1 + P.k_e) * sp ** 2 * (di + dj).sqrt()
                             / (di ** 3 + dj ** 3) * el) ** 0.4
    A = math.pi * di * dj / (2 * (di + dj)) * alpha
    Cs = Ci * Cj / (Ci + Cj)
    dq = -Cs * (qj / Cj - qi / Ci) * torch.expm1(-2.94 * alpha / sp / (Cs * (di + dj) / (2 * A) * P.phi_p))
    s["q"][i] += dq
    s["q"][j] -= dq
    for k, v in zip(("vx", "vy", "vz"), vel):
        st[k][order] = v
    st["q"][order] = s["q"]


def _advance(c, i, P, st, U=1.0, K=1.0, ssm=None, steps=None):
    """`steps` coupled steps of state st (FP64 tensors; new tensors are made, so that autograd can
    follow); returns the mean momentum source when the case asks for it."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    steps = c["steps"] if steps is None else steps
    yf, Y = torch.as_tensor(i["faces"], device=DEV), torch.as_tensor(i["Y"], device=DEV)
    vol = ((LX / nx) * (LZ / nz) * (yf[1:] - yf[:-1]))[None, :, None]
    field = _Field(nx, ny, nz, i["faces"])
    u = i["u"].to(F64).permute(3, 0, 1, 2)
    dt, pairs = i["dt"], c.get("pairs")
    F_s = torch.zeros((3, nz * ny * nx), dtype=F64, device=DEV) if c.get("two_way") else None
    for s in range(steps):
        x, y, z, d, q = (st[k] for k in ("x", "y", "z", "d", "q"))
        v = [st[k] for k in ("vx", "vy", "vz")]
        key = _cells(x.detach(), y.detach(), z.detach(), nx, nz, yf)
        rho = torch.zeros(nz * ny * nx, dtype=F64, device=DEV).index_add(0, key, q).view(nz, ny, nx) / vol
        E = field.E(field.phi(rho))
        if c.get("moving"):
            u = _lattice(i["modes"], i["Y"], nx, nz, c["re_tau"], s * dt).permute(3, 0, 1, 2)
        g, e = _gather(u.contiguous(), st, c, Y), _gather(E, st, c, Y)
        mass = math.pi * P.rho_p / 6 * d ** 3
        a = [q / mass * b for b in e]
        if pairs:
            a = [b + f for b, f in zip(a, _near_field(st, key, P))]
        tau = P.rho_p / (18 * RHO * NU) * d * d
        if c.get("sn"):
            rel = sum((b - f) ** 2 for b, f in zip(v, g)).sqrt()
            re = rel * d / NU
            slow = tau / (1 + re ** (2 / 3) / 6)
            tau = torch.where(re > 1000, 4 / 3 * (P.rho_p / RHO) / 0.424 * d / rel.clamp(min=1e-30), slow)
        h = dt / tau
        p1 = -torch.expm1(-h)
        p2, term = torch.zeros_like(h), -h
        for m in range(2, 20):                       # series of h - p1 for small h
            term = -term * h / m
            p2 = p2 - term
        p2 = torch.where(h < 0.5, -p2, h - p1)
        t = [b + f * tau for b, f in zip(g, a)]
        if F_s is not None:
            for m in range(3):
                F_s[m].index_add_(0, key, -mass / RHO * ((g[m] - v[m]) * p1 - a[m] * tau * p2))
        vn = [b + (f - b) * p1 for b, f in zip(v, t)]
        xn, yn, zn = (b + tau * (f * p1 + m * p2) for b, f, m in zip((x, y, z), v, t))
        xn, zn = xn - LX * (xn.detach() / LX).floor(), zn - LZ * (zn.detach() / LZ).floor()
        lo, hi = yn < 0.5 * d, yn > LY - 0.5 * d
        yn = torch.where(lo, d - yn, torch.where(hi, 2 * LY - d - yn, yn))
        hit = lo | hi
        vn[1] = torch.where(hit, -vn[1], vn[1])
        at = hit.nonzero()[:, 0]
        speed = sum(b[at] ** 2 for b in vn).sqrt()
        if ssm is not None:
            dq, new = _ssm(P, ssm, d[at], speed, q[at], at, st["n_imp"][at].long(), st["site"][at])
            st["site"] = st["site"].index_copy(0, at, new)
        else:
            dq = _impact(P, d[at], speed, q[at], U, K)
        st.update(x=xn, y=yn, z=zn, vx=vn[0], vy=vn[1], vz=vn[2], q=q.index_add(0, at, dq),
                  q_wall=st["q_wall"].index_add(0, at, dq), n_imp=st["n_imp"] + hit.int())
        if pairs:
            _collide(st, _cells(xn, yn, zn, nx, nz, yf), P)
    if F_s is not None:
        F_s = (F_s.view(3, nz, ny, nx) / vol) / (dt * steps)
    return F_s


def _start(i):
    st = {k: v.to(F64).clone() for k, v in i["p"].items()}
    n = len(st["x"])
    st["q_wall"] = torch.zeros(n, dtype=F64, device=DEV)
    st["n_imp"] = torch.zeros(n, dtype=torch.int32, device=DEV)
    return st


def exact(case, seed):
    c = case
    if c["kind"] == "poisson":
        f = _Field(c["nx"], c["ny"], c["nz"], _faces(c["ny"]))
        phi = f.phi(_density(c, seed))
        return dict(E=f.E(phi), phi=phi if c["phi"] else None)
    if c["kind"] == "batch":
        outs = []
        for k, b in enumerate(_batch_cases(c, seed)):
            i = _inputs(b, seed + 1000 * (k + 1))
            st = _start(i)
            with torch.no_grad():
                _advance(dict(b, steps=c["steps"]), i, _Values(rho_p=i["rho_p"], **MATERIAL), st)
            outs.append(st)
        out = {k: torch.cat([st[k] for st in outs]) for k in _STATE}
    else:
        i = _inputs(c, seed)
        P, st = _Values(rho_p=i["rho_p"], **MATERIAL), _start(i)
        if c["kind"] == "adjoint":
            U, K = (torch.ones((), dtype=F64, device=DEV, requires_grad=True) for _ in range(2))
            d = st["d"].requires_grad_()
            _advance(c, i, P, st, U, K)
            J = st["q"].mean()
            dU, dK, dd = torch.autograd.grad(J, (U, K, d))
            return dict(J=float(J), dU=dU.cpu(), dK=dK.cpu(), dd=dd, **{k: st[k].detach() for k in ("y", "vx", "q")})
        with torch.no_grad():
            F_s = _advance(c, i, P, st, ssm=_Values(**SSM) if c["ssm"] else None)
        out = {k: st[k] for k in _STATE + (("site",) if c["ssm"] else ())}
        if c["two_way"]:
            out["F_s"] = F_s
    # positions along the periodic directions have a value only up to a box length: one
    # rounding at the seam is a whole box
    out["x"] = out["z"] = out["n_imp"] = None
    return out
