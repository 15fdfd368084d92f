"""What a user of this library has it do, as measurable cases.

Each case runs through the public Python entry points (`binding.Simulation`,
`adjoint.DrivenRun`, `granulation.Granulation`).  Kinds:

* ``steps``        restore a checkpoint, advance n RK3 steps, read the state
* ``restart``      write a state, fill its ghosts, take the time step and the
                   global diagnostics, read it back
* ``adjoint``      one taped step and its reverse step, gradients read
* ``gradient``     a driven run and its gradient through torch.autograd
* ``granulation``  one update of the driver's granules and its velocity field

A pass of ``steps`` starts from the same checkpoint every time (an ensemble or
a fit does so), so the state does not drift from pass to pass.  `exact` holds
the same model written plainly in FP64 torch, full variables, one operator at
a time, without any code of this library.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1908_08557_gb300.adjoint import BzPlane, DrivenRun
from paper_1908_08557_gb300.binding import Simulation
from paper_1908_08557_gb300.granulation import Granulation, paper_params

DEV = "cuda:0"
NG = 3
DT_FIXED = 0.01


def listed():
    return [
        # the plain-method box (32^3, FP64): a quick physics check, where
        # launches and latency are all there is
        dict(name="steps64_32", kind="steps", precision=64, nx=32, ny=32, nz=32, steps=10),
        # the forward run inside a small fit (64^3, FP32)
        dict(name="steps32_64", kind="steps", precision=32, nx=64, ny=64, nz=64, steps=10),
        # a wave or convergence study in a triply periodic box of odd sizes (FP64)
        dict(name="steps64_periodic", kind="steps", precision=64, nx=150, ny=99, nz=70, steps=2, periodic_z=True),
        # the throughput workload (256^3, FP32), diagnostics every 10 steps
        dict(name="steps32_256", kind="steps", precision=32, nx=256, ny=256, nz=256, steps=10, stats_every=10),
        # the same box in FP64 (the reference run of a precision comparison)
        dict(name="steps64_256", kind="steps", precision=64, nx=256, ny=256, nz=256, steps=1),
        # the production box, horizontal spacing 4x vertical, A stored about
        # its initial field
        dict(name="steps32_1024", kind="steps", precision=32, nx=1024, ny=1024, nz=256, steps=2, hscale=4.0,
             background=True),
        # a stretched vertical grid with Newtonian cooling, ragged in z
        dict(name="steps32_stretched", kind="steps", precision=32, nx=512, ny=256, nz=97, steps=4, stretched=True,
             cooling=True),
        # loading a 256^3 snapshot and looking at it
        dict(name="restart32_256", kind="restart", precision=32, nx=256, ny=256, nz=256),
        # one forward and reverse step of the throughput workload, taped
        dict(name="adjoint32_256", kind="adjoint", precision=32, nx=256, ny=256, nz=256),
        # a gradient of the small fit, the whole history taped
        dict(name="gradient32_64", kind="gradient", precision=32, nx=64, ny=64, nz=64, steps=10, slots=30),
        # a checkpointed gradient in FP64 (few slots, so steps are recomputed)
        dict(name="gradient64_ckpt", kind="gradient", precision=64, nx=64, ny=32, nz=45, steps=5, slots=2),
        # one driver update of a 1024^2 photosphere of 0.23 Mm pixels
        dict(name="granulation_1024", kind="granulation", precision=32, nx=1024, ny=1024),
    ]


def draw(rng):
    """One more case of the listed kinds; sizes spread over the logarithm."""
    pow2 = lambda lo, hi: 2 ** rng.randint(lo, hi)  # noqa: E731
    span = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(["steps"] * 5 + ["restart", "adjoint", "gradient", "gradient", "granulation"])
    prec = rng.choice([32, 64])
    if kind == "granulation":
        return dict(kind=kind, precision=prec, nx=pow2(6, 10), ny=pow2(6, 10))
    if kind == "gradient":
        n = rng.randint(2, 8)
        return dict(kind=kind, precision=prec, nx=pow2(4, 6), ny=pow2(4, 6), nz=span(14, 90), steps=n,
                    slots=rng.choice([1, 3, 3 * n]))
    if kind == "adjoint":
        return dict(kind=kind, precision=prec, nx=pow2(5, 7), ny=pow2(5, 8), nz=span(16, 160))
    if kind == "restart":
        return dict(kind=kind, precision=prec, nx=pow2(5, 8), ny=pow2(5, 8), nz=span(16, 200))
    big = 8 if prec == 32 else 7
    c = dict(kind=kind, precision=prec, nx=pow2(5, big + 1), ny=pow2(5, big), nz=span(16, 200), steps=rng.randint(1, 4))
    opt = rng.choice(["plain", "plain", "stats", "stretched", "cooling", "background", "periodic"])
    if opt == "stats":
        c["stats_every"] = c["steps"]
    elif opt == "periodic":
        c.update(nx=span(32, 2 ** big), ny=span(32, 2 ** big), nz=span(16, 150), periodic_z=True)
    elif opt != "plain":
        c[opt] = True
    if opt == "background":
        c["hscale"] = 4.0
    return c


# ---------------------------------------------------------------------------
# inputs

def _params(c):
    h = float(c.get("hscale", 1.0))
    nz = c["nz"]
    p = dict(gamma=5.0 / 3.0, gz=-0.2, nu=0.05, eta=0.05, kappa0=2e-8, diff_rho=0.05, eta_swamp=0.5, chi_swamp=0.5,
             diffrho_swamp=0.5, tau_u=0.5, tau_A=0.5, t_ramp=0.5, f_pfe_bottom=0.2, c_adv=0.4, c_diff=0.25,
             dt_fixed=0.0, bc_z=0, nc_tau=0.0, nc_lnrho_magn=8.0, nc_lnrho_width=2.0, nc_z_max=10.0, nc_z_width=1.0,
             nx=c["nx"], ny=c["ny"], nz=nz, dx=h, dy=h, dz=1.0, z_swamp_start=nz - 5.0, z_swamp_end=nz - 1.0)
    k = np.arange(-NG, nz + NG, dtype=np.float64)
    z = k.copy()
    if c.get("stretched"):
        # spacing rising from 0.5 to 1.5 around a third of the height
        kc, w = nz / 3.0, nz / 8.0
        lc = lambda x: np.log(np.cosh(x))  # noqa: E731
        z = 0.5 * k + 0.5 * (k + w * (lc((k - kc) / w) - lc(-kc / w)))
        top = z[NG + nz - 1]
        p.update(z=z, z_swamp_start=top - 4.0 * (top - z[NG + nz - 2]), z_swamp_end=top)
    if c.get("cooling"):
        p["nc_tau"] = 0.5
    if c.get("periodic_z"):
        p.update(bc_z=1, gz=0.0, eta_swamp=0.0, chi_swamp=0.0, diffrho_swamp=0.0)
    if c["kind"] in ("adjoint", "gradient"):
        p["dt_fixed"] = DT_FIXED
    return p, z


def _profiles(p, z):
    """Hydrostatic atmosphere, T from 1 to 100 through a tanh (zeros in the periodic box)."""
    if p["bc_z"]:
        return np.zeros_like(z), np.zeros_like(z)
    T = 1.0 + 49.5 * (1.0 + np.tanh((z - 12.0) / 2.0))
    lnp = np.zeros_like(z)
    for q in range(NG + 1, len(z)):
        lnp[q] = lnp[q - 1] + (z[q] - z[q - 1]) * p["gz"] * 0.5 * (1.0 / T[q - 1] + 1.0 / T[q])
    for q in range(NG - 1, -1, -1):
        lnp[q] = lnp[q + 1] - (z[q + 1] - z[q]) * p["gz"] * 0.5 * (1.0 / T[q + 1] + 1.0 / T[q])
    return lnp - np.log(T), np.log(T)


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(dtype)


def _bipoles(p, rng):
    """Flux-balanced bipoles, one per 1600 cells or so, log-normal fluxes (FP64 [ny, nx])."""
    nx, ny = p["nx"], p["ny"]
    n = max(4, nx * ny // 1638)
    d, th = rng.uniform(4.0, 16.0, n), rng.uniform(0.0, 2.0 * np.pi, n)
    xc, yc = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
    a = 0.1 * np.minimum(rng.lognormal(0.0, 1.0, n), 6.0)
    x = np.concatenate([xc + 0.5 * d * np.cos(th), xc - 0.5 * d * np.cos(th)])
    y = np.concatenate([yc + 0.5 * d * np.sin(th), yc - 0.5 * d * np.sin(th)])
    amp = _t(np.concatenate([a, -a]))

    def bump(c, m):
        r = (torch.arange(m, device=DEV, dtype=torch.float64)[None, :] - _t(c)[:, None] + 0.5 * m) % m - 0.5 * m
        return torch.exp(-r * r / 18.0)

    bz = (bump(y, ny) * amp[:, None]).T @ bump(x, nx)
    return bz - bz.mean()


def _wave(n, d):
    return 2.0 * math.pi * torch.fft.fftfreq(n, d=d, device=DEV, dtype=torch.float64)


def _potential(bz, p, z, out):
    """A_x, A_y of the potential field with B_z = bz at z = 0 into out[0], out[1]."""
    kx, ky = _wave(p["nx"], p["dx"])[None, :], _wave(p["ny"], p["dy"])[:, None]
    kk = torch.sqrt(kx * kx + ky * ky)
    bh = torch.fft.fft2(bz)
    bh[0, 0] = 0.0
    if p["nx"] % 2 == 0:
        bh[:, p["nx"] // 2] = 0.0
    if p["ny"] % 2 == 0:
        bh[p["ny"] // 2, :] = 0.0
    k2 = torch.where(kk > 0, kk * kk, torch.ones_like(kk))
    for c, h in ((0, 1j * ky * bh / k2), (1, -1j * kx * bh / k2)):
        for k in range(p["nz"]):
            out[c, k] = torch.fft.ifft2(h * torch.exp(-kk * float(z[NG + k]))).real


def _drivers(p, rng):
    """A solenoidal plane flow with a k^-5/3 spectrum, rms 0.01 (FP64 [2, ny, nx])."""
    nx, ny = p["nx"], p["ny"]
    mx = torch.fft.fftfreq(nx, d=1.0 / nx, device=DEV, dtype=torch.float64)[None, :]
    my = torch.fft.fftfreq(ny, d=1.0 / ny, device=DEV, dtype=torch.float64)[:, None]
    kk = torch.sqrt(mx * mx + my * my)
    on = (kk >= 1) & (kk <= min(32, nx // 2, ny // 2))
    amp = torch.where(on, torch.where(on, kk, torch.ones_like(kk)) ** (-4.0 / 3.0 - 1.0), torch.zeros_like(kk))
    psi = torch.polar(amp, _t(rng.uniform(0.0, 2.0 * np.pi, (ny, nx))))
    v = torch.stack([torch.fft.ifft2(1j * my / ny * psi).real, torch.fft.ifft2(-1j * mx / nx * psi).real])
    return v * (0.01 / torch.sqrt((v * v).sum(0).mean()))


def _ripple(f, p, rng, amp, waves=3):
    """Adds a few long plane waves of the given amplitude to the field f [nz, ny, nx]."""
    nz, ny, nx = f.shape
    for _ in range(waves):
        m = rng.integers(1, 4, 3)
        ph = rng.uniform(0.0, 2.0 * np.pi, 3)
        w = [amp * rng.uniform(0.5, 1.0) / waves, 1.0, 1.0]
        s = [_t(w[q] * np.sin(2.0 * np.pi * m[q] * np.arange(n) / n + ph[q]))
             for q, n in enumerate((nz, ny, nx))]
        f += (s[0][:, None, None] * s[1][None, :, None] * s[2][None, None, :]).to(f.dtype)


def _inputs(c, seed):
    """What a box starts from: parameters, profiles, state, background, magnetogram, drivers."""
    rng = np.random.default_rng(seed)
    dtype = torch.float32 if c["precision"] == 32 else torch.float64
    p, z = _params(c)
    lnrho0, lnT0 = _profiles(p, z)
    bz = _bipoles(p, rng)
    v0, v1 = _drivers(p, rng), _drivers(p, rng)
    st = torch.zeros((8, p["nz"], p["ny"], p["nx"]), dtype=dtype, device=DEV)
    bg = None
    if c.get("background"):
        bg = torch.zeros((3, p["nz"], p["ny"], p["nx"]), dtype=torch.float64, device=DEV)
        _potential(bz, p, z, bg)
    elif p["bc_z"]:
        for q in range(3):
            _ripple(st[q], p, rng, 0.5)
    else:
        _potential(bz, p, z, st)
    for q in range(3, 6):
        _ripple(st[q], p, rng, 0.5)  # rms a few 0.01: a box some way into its run
    for q, prof in ((6, lnrho0), (7, lnT0)):
        st[q] = _t(prof[NG:NG + p["nz"]])[:, None, None].to(dtype)
        _ripple(st[q], p, rng, 0.02)
    if not p["bc_z"]:
        st[5, 0] = 0.0
        st[5, -1] = 0.0
        st[6, 0] = float(lnrho0[NG])
    return dict(c=c, p=p, z=z, lnrho0=lnrho0, lnT0=lnT0, st=st, bg=bg, bz=bz.to(dtype), v0=v0.to(dtype),
                v1=v1.to(dtype), rng=rng)


def _simulation(s, adjoint=False):
    c = s["c"]
    sim = Simulation(s["p"], s["st"], s["lnrho0"], s["lnT0"], precision=c["precision"],
                     stats_every=c.get("stats_every", 0), device=DEV, adjoint=adjoint, a_background=s["bg"])
    if not s["p"]["bc_z"]:
        sim.set_driver(s["bz"], s["v0"], s["v1"], 0.0, 1.0)
    return sim


def _adjoint_seed(s):
    """dL/d(state) of a smooth loss on every field."""
    lam = torch.zeros_like(s["st"])
    for q in range(8):
        _ripple(lam[q], s["p"], s["rng"], 1.0)
    return lam


def _targets(s):
    """What a fit aims at: B_z on a layer and u_hor on the first layer above the photosphere."""
    p = s["p"]
    t = torch.zeros((3, p["ny"], p["nx"]), dtype=s["st"].dtype, device=DEV)
    for q, amp in ((0, 0.2), (1, 0.05), (2, 0.05)):
        _ripple(t[q:q + 1].view(1, p["ny"], p["nx"]), p, s["rng"], amp)
    return t


def _granulation(c, seed):
    p = paper_params(mm_per_unit=0.23)
    rng = np.random.default_rng(seed)
    ny, nx = c["ny"], c["nx"]
    draws = [(_t(rng.integers(-2 ** 31, 2 ** 31, (ny, nx)), torch.int32), _t(rng.standard_normal((ny, nx))),
              _t(rng.standard_normal((ny, nx)))) for _ in range(3)]
    return p, draws


GRAN_START = 20  # updates before the measured ones: the plane is full and granules have begun to die
GRAN_DT = 20.0


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "granulation":
        p, draws = _granulation(c, seed)
        gen = Granulation(c["nx"], c["ny"], 1.0, 1.0, p, device=DEV)
        for n in range(GRAN_START):
            gen.update(n * GRAN_DT, *draws[n % 3])
        return dict(c=c, gen=gen, draws=draws, n=GRAN_START)
    s = _inputs(c, seed)
    if c["kind"] == "gradient":
        s["target"] = _targets(s)
        s["sim"] = _simulation(s, adjoint=True)
    elif c["kind"] == "adjoint":
        s["lam"] = _adjoint_seed(s)
        s["sim"] = _simulation(s, adjoint=True)
        s["tape"] = s["sim"].new_tape()
        s["ck"] = s["sim"].new_checkpoint()
        s["sim"].save(s["ck"])
        s["st"] = None
    else:
        s["sim"] = _simulation(s)
        if c["kind"] == "steps":
            s["ck"] = s["sim"].new_checkpoint()
            s["sim"].save(s["ck"])
            s["st"] = s["bg"] = None
    return s


# ---------------------------------------------------------------------------
# one pass

def _told(d):
    # max |div B| and the net flux are rounding residuals of terms that cancel
    return {k: d[k] for k in ("t", "dt", "e_kin", "e_mag", "e_th", "mass", "flux_abs")}


def _fields(a):
    return {"a": a[0:3], "u": a[3:6], "lnrho": a[6], "lnTT": a[7]}


def _fit_layer(nz):
    return min(8, nz - 4)


def run(s):
    kind = s["c"]["kind"]
    if kind == "granulation":
        t = s["n"] * GRAN_DT
        s["gen"].update(t, *s["draws"][s["n"] % 3])
        s["n"] += 1
        v = s["gen"].velocity(t, s["c"]["precision"])
        occ, par = s["gen"].granules()
        return {"v": v, "occ": occ, "par": par}
    sim = s["sim"]
    if kind == "steps":
        sim.restore(s["ck"], 0.0)
        sim.step(s["c"]["steps"])
        out = _fields(sim.read())
        if s["c"].get("stats_every"):
            out["stats"] = _told(sim.read_stats())
        return out
    if kind == "restart":
        sim.write(s["st"])
        sim.set_time(0.0)
        sim.fill_ghosts()
        dt = sim.compute_dt()
        stats = sim.compute_stats()
        stats = {k: stats[k] for k in ("e_kin", "e_mag", "e_th", "mass", "flux_abs")}
        return {"dt": dt, "stats": stats, **_fields(sim.read())}
    if kind == "adjoint":
        sim.restore(s["ck"], 0.0)
        sim.step_taped(s["tape"])
        sim.adjoint_init(s["lam"])
        sim.adjoint_step_taped(s["tape"])
        g = sim.adjoint_read()
        return {"lam": _fields(g["lam"]), "bz": g["bz"], "v0": g["v0"], "v1": g["v1"], "state": _fields(sim.read())}
    bz, v0, v1, st = (x.detach().requires_grad_() for x in (s["bz"], s["v0"], s["v1"], s["st"]))
    fin = DrivenRun.apply(bz, v0, v1, sim, st, s["c"]["steps"], s["c"]["slots"])
    b = BzPlane.apply(fin, sim, _fit_layer(s["c"]["nz"]))
    loss = 0.5 * ((b - s["target"][0]) ** 2).sum() + 0.5 * ((fin[3:5, 1] - s["target"][1:]) ** 2).sum()
    loss.backward()
    return {"state": _fields(fin.detach()), "bz": bz.grad, "v0": v0.grad, "v1": v1.grad, "st": _fields(st.grad)}


def work(case):
    c = dict(case)
    e = c["precision"] // 8
    if c["kind"] == "granulation":
        n = c["nx"] * c["ny"]
        # draws, granule maps and velocity once each; one complex 2D FFT and its inverse
        return {"bytes": n * (20 + 36 + 36 + 2 * e), "flops": n * 10.0 * math.log2(n)}
    n = c["nx"] * c["ny"] * c["nz"]
    # a 2N-storage RK3 step: f read and written three times, df twice; about
    # a thousand operations per cell and substep
    step = {"bytes": 80.0 * n * e, "flops": 3.0 * 1000 * n}
    if c["kind"] == "steps":
        m = c["steps"]
        return {"bytes": m * step["bytes"] + 16.0 * n * e, "flops": m * step["flops"]}
    if c["kind"] == "restart":
        return {"bytes": 32.0 * n * e, "flops": 200.0 * n}
    m = c.get("steps", 1)
    # the reverse of a substep reads the state and D, writes and reads the 40
    # coefficients, reads and writes F and D
    back = {"bytes": 3.0 * (16 + 80 + 32) * n * e, "flops": 3.0 * 2500 * n}
    return {k: m * (step[k] + back[k]) for k in step}


# ---------------------------------------------------------------------------
# the same model in plain FP64 torch

C1 = (0.75, -0.15, 1.0 / 60.0)
C2 = (-49.0 / 18.0, 1.5, -0.15, 1.0 / 90.0)
RK_A = (0.0, -5.0 / 9.0, -153.0 / 128.0)
RK_B = (1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0)
RK_C = (0.0, 1.0 / 3.0, 0.75)


def _sl(f, ax, o):
    return f.narrow(ax, NG + o, f.shape[ax] - 2 * NG)


def _d1(f, ax, inv):
    """First derivative along ax; that axis loses its three-cell rims."""
    s = sum(C1[m] * (_sl(f, ax, m + 1) - _sl(f, ax, -m - 1)) for m in range(3))
    return s * inv


def _d2(f, ax, inv):
    s = C2[0] * _sl(f, ax, 0) + sum(C2[m + 1] * (_sl(f, ax, m + 1) + _sl(f, ax, -m - 1)) for m in range(3))
    return s * inv


def _core(f, *axes):
    for a in axes:
        f = _sl(f, a, 0)
    return f


class _Model:
    """The box's equations; the state is (f [8, nz, ny, nx], ug [3, 2, ny, nx]) with ug[m - 1] = u_x, u_y on layer -m."""

    def __init__(self, s):
        self.p = p = s["p"]
        z = s["z"]
        nz = p["nz"]
        self.zpos = lambda k: float(z[k + NG])
        self.lnrho0 = s["lnrho0"]
        col = lambda a: _t(a)[:, None, None]  # noqa: E731
        zi = z[NG:NG + nz]
        if "z" in p:
            z1 = sum(C1[m] * (z[NG + m + 1:NG + m + 1 + nz] - z[NG - m - 1:NG - m - 1 + nz]) for m in range(3))
            z2 = C2[0] * zi + sum(C2[m + 1] * (z[NG + m + 1:NG + m + 1 + nz] + z[NG - m - 1:NG - m - 1 + nz])
                                  for m in range(3))
        else:
            z1, z2 = np.full(nz, p["dz"]), np.zeros(nz)
        self.m1, self.r21 = col(1.0 / z1), col(-z2 / z1 ** 2)
        self.cell = col(0.5 * (z[NG + 1:NG + 1 + nz] - z[NG - 1:NG - 1 + nz]) if "z" in p else np.full(nz, p["dz"]))
        q = np.clip((zi - p["z_swamp_start"]) / (p["z_swamp_end"] - p["z_swamp_start"]), 0.0, 1.0)
        self.w = col(q * q * (3.0 - 2.0 * q))
        self.wp = col(6.0 * q * (1.0 - q) / (p["z_swamp_end"] - p["z_swamp_start"]))
        self.lr, self.lt = _t(s["lnrho0"][NG:NG + nz]), _t(s["lnT0"][NG:NG + nz])
        a = np.clip((zi - p["nc_z_max"] + p["nc_z_width"]) / p["nc_z_width"], 0.0, 1.0)
        self.cz = col(0.5 * (1.0 + np.cos(np.pi * a)))
        if not p["bc_z"]:
            kx, ky = _wave(p["nx"], p["dx"])[None, :], _wave(p["ny"], p["dy"])[:, None]
            kk = torch.sqrt(kx * kx + ky * ky)
            self.up = [torch.exp(-kk * (self.zpos(nz - 1 + m) - self.zpos(nz - 1))) for m in (1, 2, 3)]
            self.dn = [torch.exp(p["f_pfe_bottom"] * kk * (self.zpos(0) - self.zpos(-m))) for m in (1, 2, 3)]

    def target(self, bz):
        """A_x, A_y of the magnetogram with the first difference's own wavenumbers."""
        p = self.p

        def mod(n, h):
            th = 2.0 * np.pi * np.fft.fftfreq(n)
            k = (45.0 * np.sin(th) - 9.0 * np.sin(2 * th) + np.sin(3 * th)) / (30.0 * h)
            k[0] = 0.0
            if n % 2 == 0:
                k[n // 2] = 0.0
            return _t(k)

        kx, ky = mod(p["nx"], p["dx"])[None, :], mod(p["ny"], p["dy"])[:, None]
        k2 = kx * kx + ky * ky
        b = torch.fft.fft2(bz) * torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
        return torch.stack([torch.fft.ifft2(1j * ky * b).real, torch.fft.ifft2(-1j * kx * b).real])

    def ghosts(self, f, ug):
        """The six ghost layers: below [8, 3, ny, nx] (layers -3, -2, -1), above (nz, nz + 1, nz + 2)."""
        p, nz = self.p, self.p["nz"]
        if p["bc_z"]:
            return f[:, -NG:], f[:, :NG]
        fa, fb = torch.fft.fft2(f[0:3, -1]), torch.fft.fft2(f[0:3, 0])
        lo, hi = [], []
        th, lr = f[7, 0], f[6, 0]
        top = torch.exp(f[7, -1])
        for m in (1, 2, 3):
            l0 = torch.full_like(th, float(self.lnrho0[NG - m]))
            t0 = th + lr - l0 - (self.zpos(1 - m) - self.zpos(-m)) * p["gz"] / torch.exp(th)
            a = torch.fft.ifft2(fb * self.dn[m - 1]).real
            lo.append(torch.cat([a, ug[m - 1], -f[5:6, m], l0[None], t0[None]]))
            th, lr = t0, l0
            a = torch.fft.ifft2(fa * self.up[m - 1]).real
            g = f[:, nz - 1 - m]
            l1 = g[6] + (self.zpos(nz - 1 + m) - self.zpos(nz - 1 - m)) * p["gz"] / top
            hi.append(torch.cat([a, g[3:5], -g[5:6], l1[None], g[7:8]]))
        return torch.stack(lo[::-1], 1), torch.stack(hi, 1)

    def slabs(self, f, lo, hi, deep):
        """(k0, k1, layers k0 - 3 .. k1 + 2 with periodic x, y rims)."""
        nz = self.p["nz"]
        for k0 in range(0, nz, deep):
            k1 = min(nz, k0 + deep)
            part = [f[:, max(0, k0 - NG):min(nz, k1 + NG)]]
            if k0 < NG:
                part.insert(0, lo[:, k0:])
            if k1 > nz - NG:
                part.append(hi[:, :k1 + NG - nz])
            g = torch.cat(part, 1)
            g = torch.cat([g[:, :, -NG:], g, g[:, :, :NG]], 2)
            yield k0, k1, torch.cat([g[..., -NG:], g, g[..., :NG]], 3)

    def rhs(self, g, k0, k1):
        """Right-hand side on layers k0 .. k1 - 1 of the slab g, boundary rows left out."""
        p = self.p
        ix, iy = 1.0 / p["dx"], 1.0 / p["dy"]
        m1, r21, w, wp = self.m1[k0:k1], self.r21[k0:k1], self.w[k0:k1], self.wp[k0:k1]
        # axes of a single field: z 0, y 1, x 2
        X = lambda f: _d1(f, 2, ix)  # noqa: E731
        Y = lambda f: _d1(f, 1, iy)  # noqa: E731
        Z = lambda f: _d1(f, 0, 1.0) * m1  # noqa: E731
        dx = lambda f: X(_core(f, 0, 1))  # noqa: E731
        dy = lambda f: Y(_core(f, 0, 2))  # noqa: E731
        dz = lambda f: Z(_core(f, 1, 2))  # noqa: E731
        xx = lambda f: _d2(_core(f, 0, 1), 2, ix * ix)  # noqa: E731
        yy = lambda f: _d2(_core(f, 0, 2), 1, iy * iy)  # noqa: E731
        zz = lambda f: _d2(_core(f, 1, 2), 0, 1.0) * m1 * m1 + r21 * dz(f)  # noqa: E731
        xy = lambda f: Y(X(_core(f, 0)))  # noqa: E731
        xz = lambda f: Z(X(_core(f, 1)))  # noqa: E731
        yz = lambda f: Z(Y(_core(f, 2)))  # noqa: E731

        def second(a):
            """Laplacian and grad div of a vector field."""
            d = [[xx(a[q]), yy(a[q]), zz(a[q])] for q in range(3)]
            lap = [sum(d[q]) for q in range(3)]
            gd = [d[0][0] + xy(a[1]) + xz(a[2]), xy(a[0]) + d[1][1] + yz(a[2]), xz(a[0]) + yz(a[1]) + d[2][2]]
            return lap, gd

        def dot(a, b):
            return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

        def cross(a, b):
            return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

        A, U, L, T = g[0:3], g[3:6], g[6], g[7]
        B = [dy(A[2]) - dz(A[1]), dz(A[0]) - dx(A[2]), dx(A[1]) - dy(A[0])]
        lapA, gdA = second(A)
        J = [gdA[q] - lapA[q] for q in range(3)]
        divA = dx(A[0]) + dy(A[1]) + dz(A[2])
        u = [_core(U[q], 0, 1, 2) for q in range(3)]
        dU = [[dx(U[q]), dy(U[q]), dz(U[q])] for q in range(3)]
        lapU, gdU = second(U)
        div = dU[0][0] + dU[1][1] + dU[2][2]
        S = [[0.5 * (dU[a][b] + dU[b][a]) - (div / 3.0 if a == b else 0.0) for b in range(3)] for a in range(3)]
        gL, gT = [dx(L), dy(L), dz(L)], [dx(T), dy(T), dz(T)]
        lapL, lapT = xx(L) + yy(L) + zz(L), xx(T) + yy(T) + zz(T)
        lr, th = _core(L, 0, 1, 2), _core(T, 0, 1, 2)
        rho1, temp = torch.exp(-lr), torch.exp(th)
        uB, JB = cross(u, B), cross(J, B)
        out = [uB[q] - p["eta"] * J[q] + p["eta_swamp"] * w * lapA[q] for q in range(3)]
        out[2] = out[2] + p["eta_swamp"] * wp * divA
        for q in range(3):
            visc = p["nu"] * (lapU[q] + gdU[q] / 3.0 + 2.0 * dot(S[q], gL))
            out.append(-dot(u, dU[q]) - temp * (gL[q] + gT[q]) + JB[q] * rho1 + visc + (p["gz"] if q == 2 else 0.0))
        out.append(-dot(u, gL) - div + p["diff_rho"] * (lapL + dot(gL, gL)) + p["diffrho_swamp"] * w * lapL)
        gm1 = p["gamma"] - 1.0
        S2 = sum(dot(S[q], S[q]) for q in range(3))
        heat = gm1 * (p["eta"] * dot(J, J) * rho1 + 2.0 * p["nu"] * S2) / temp
        cond = gm1 * p["kappa0"] * torch.exp(2.5 * th - lr) * (lapT + 3.5 * dot(gT, gT))
        e = -dot(u, gT) - gm1 * div + heat + cond + p["chi_swamp"] * w * lapT
        if p["nc_tau"] > 0.0:
            e = e + self.cooling(lr, th, k0, k1)
        out.append(e)
        return torch.stack(out)

    def cooling(self, lr, th, k0, k1):
        """-tau (1 - T*/T) c_rho c_z, T* between T0(z) and the temperature the initial profile has at this density."""
        p, n = self.p, self.p["nz"]
        up = torch.flip(self.lr, [0]).contiguous()
        i = torch.clamp(torch.searchsorted(up, lr.contiguous(), right=False), 1, n - 1)
        a, b = n - i, n - 1 - i  # layers with lr[b] >= ln rho > lr[a]
        s = torch.clamp((lr - self.lr[b]) / (self.lr[a] - self.lr[b]), 0.0, 1.0)
        tp = self.lt[b] + s * (self.lt[a] - self.lt[b])
        q = torch.clamp((self.lr[0] - lr - p["nc_lnrho_magn"] + p["nc_lnrho_width"]) / p["nc_lnrho_width"], 0.0, 1.0)
        cr = 0.5 * (1.0 + torch.cos(math.pi * q))
        r = torch.exp(0.5 * (self.lt[k0:k1, None, None] + tp) - th)
        return -p["nc_tau"] * (1.0 - r) * cr * self.cz[k0:k1]

    def curl(self, g, k0, k1):
        p = self.p
        dx = lambda f: _d1(_core(f, 0, 1), 2, 1.0 / p["dx"])  # noqa: E731
        dy = lambda f: _d1(_core(f, 0, 2), 1, 1.0 / p["dy"])  # noqa: E731
        dz = lambda f: _d1(_core(f, 1, 2), 0, 1.0) * self.m1[k0:k1]  # noqa: E731
        return [dy(g[2]) - dz(g[1]), dz(g[0]) - dx(g[2]), dx(g[1]) - dy(g[0])]

    def look(self, f, lo, hi, deep):
        """CFL time step and the diagnostics of a state with its ghosts."""
        p = self.p
        gm1 = p["gamma"] - 1.0
        adv = dif = 0.0
        tot = dict(e_kin=0.0, e_mag=0.0, e_th=0.0, mass=0.0, flux_abs=0.0)
        for k0, k1, g in self.slabs(f, lo, hi, deep):
            B = self.curl(g, k0, k1)
            B2 = B[0] ** 2 + B[1] ** 2 + B[2] ** 2
            u, lr, th = f[3:6, k0:k1], f[6, k0:k1], f[7, k0:k1]
            m1, w = self.m1[k0:k1], self.w[k0:k1]
            sq = 1.0 / p["dx"] ** 2 + 1.0 / p["dy"] ** 2 + m1 * m1
            rho, temp = torch.exp(lr), torch.exp(th)
            a = u[0].abs() / p["dx"] + u[1].abs() / p["dy"] + u[2].abs() * m1 + torch.sqrt((p["gamma"] * temp + B2 / rho) * sq)
            d = torch.clamp(p["eta"] + p["eta_swamp"] * w, min=p["nu"])
            d = torch.maximum(d, p["diff_rho"] + p["diffrho_swamp"] * w)
            d = torch.maximum(d, p["chi_swamp"] * w + gm1 * p["kappa0"] * torch.exp(2.5 * th - lr)) * sq
            adv, dif = max(adv, float(a.max())), max(dif, float(d.max()))
            dv = p["dx"] * p["dy"] * self.cell[k0:k1]
            tot["e_kin"] += float((0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) * dv).sum())
            tot["e_mag"] += float((0.5 * B2 * dv).sum())
            tot["e_th"] += float((rho * temp * dv).sum()) / gm1
            tot["mass"] += float((rho * dv).sum())
            if k0 == 0:
                tot["flux_abs"] = float(B[2][0].abs().sum()) * p["dx"] * p["dy"]
        dt = p["dt_fixed"] if p["dt_fixed"] > 0 else min(p["c_adv"] / adv, p["c_diff"] / dif)
        return dt, tot

    def substep(self, f, ug, df, dug, sub, t, dt, drv, deep):
        """One Williamson substep; drv = (A target, v0, v1) or None."""
        p = self.p
        lo, hi = self.ghosts(f, ug)
        rows = []
        for k0, k1, g in self.slabs(f, lo, hi, deep):
            rows.append(self.rhs(g, k0, k1))
        r = torch.cat(rows, 1)
        du = torch.zeros_like(ug)
        if not p["bc_z"]:
            at, v0, v1 = drv
            ts = t + RK_C[sub] * dt
            v = min(1.0, max(0.0, ts / p["t_ramp"])) * (v0 + min(1.0, max(0.0, ts)) * (v1 - v0))
            z = torch.zeros_like(r[5, 0])
            bot = torch.cat([r[0:2, 0] - p["tau_A"] * (f[0:2, 0] - at), r[2:3, 0],
                             r[3:5, 0] - p["tau_u"] * (f[3:5, 0] - v), z[None], z[None], r[7:8, 0]])
            top = torch.cat([r[0:5, -1], z[None], r[6:8, -1]])
            r = torch.cat([bot[:, None], r[:, 1:-1], top[:, None]], 1)
            du = -p["tau_u"] * (ug - v[None])
        df, dug = RK_A[sub] * df + dt * r, RK_A[sub] * dug + dt * du
        return f + RK_B[sub] * df, ug + RK_B[sub] * dug, df, dug


def _start(s):
    f = s["st"].double()
    if s["bg"] is not None:
        f[0:3] = s["bg"]
    return f


def _deep(p):
    return max(4, int(1.2e7) // (p["nx"] * p["ny"]))


def _ref_steps(s):
    with torch.no_grad():
        m, c, p = _Model(s), s["c"], s["p"]
        f, t, told = _start(s), 0.0, None
        s["st"] = s["bg"] = None
        ug = f[3:5, 0].clone()[None].repeat(3, 1, 1, 1)
        drv = None if p["bc_z"] else (m.target(s["bz"].double()), s["v0"].double(), s["v1"].double())
        for n in range(c["steps"]):
            dt, tot = m.look(f, *m.ghosts(f, ug), _deep(p))
            if c.get("stats_every") and n % c["stats_every"] == 0:
                told = tot
            df, dug = torch.zeros_like(f), torch.zeros_like(ug)
            for sub in range(3):
                f, ug, df, dug = m.substep(f, ug, df, dug, sub, t, dt, drv, _deep(p))
            t += dt
        out = _fields(f)
        if c.get("stats_every"):
            # the time of the diagnostics is that of the step they were taken in
            out["stats"] = {"t": None, "dt": dt, **told}
        return out


def _ref_gradient(s, lam=None):
    m, c, p = _Model(s), s["c"], s["p"]
    bz, v0, v1, st = (x.double().requires_grad_() for x in (s["bz"], s["v0"], s["v1"], s["st"]))
    f, t, dt = st, 0.0, p["dt_fixed"]
    ug = f[3:5, 0][None].repeat(3, 1, 1, 1)
    at = m.target(bz)
    for _ in range(c.get("steps", 1)):
        df, dug = torch.zeros_like(f), torch.zeros_like(ug)
        for sub in range(3):
            go = lambda a, b, d, e, x, y, w, sub=sub, t=t: m.substep(a, b, d, e, sub, t, dt, (x, y, w), p["nz"])  # noqa: E731
            f, ug, df, dug = checkpoint(go, f, ug, df, dug, at, v0, v1, use_reentrant=False)
        t += dt
    if lam is not None:
        loss = (f * lam.double()).sum()
    else:
        k, tg = _fit_layer(p["nz"]), s["target"].double()
        a = torch.cat([f[0:2, k, -NG:], f[0:2, k], f[0:2, k, :NG]], 1)
        a = torch.cat([a[..., -NG:], a, a[..., :NG]], 2)
        b = _d1(_core(a[1], 0), 1, 1.0 / p["dx"]) - _d1(_core(a[0], 1), 0, 1.0 / p["dy"])
        loss = 0.5 * ((b - tg[0]) ** 2).sum() + 0.5 * ((f[3:5, 1] - tg[1:]) ** 2).sum()
    loss.backward()
    return f.detach(), bz.grad, v0.grad, v1.grad, st.grad


def _ref_granulation(c, seed):
    """The sequential visit by (key, index) as rounds of local minima, then Eqs. 2-4 term by term."""
    p, draws = _granulation(c, seed)
    ny, nx = c["ny"], c["nx"]

    def disk(r):
        m = int(math.ceil(r))
        return [(y, x) for y in range(-m, m + 1) for x in range(-m, m + 1) if (y or x) and y * y + x * x < r * r]

    near = disk(p["r_inner"])
    occ = torch.zeros((ny, nx), dtype=torch.bool, device=DEV)
    t0, life, vm, tm = (torch.zeros((ny, nx), dtype=torch.float64, device=DEV) for _ in range(4))
    spread = lambda q: torch.stack([torch.roll(q, o, (0, 1)) for o in near])  # noqa: E731
    index = torch.arange(nx * ny, device=DEV).view(ny, nx)
    for n in range(GRAN_START + 1):
        t = n * GRAN_DT
        keys, cl, ca = draws[n % 3]
        dead = occ & (t - t0 - tm > tm)
        occ = occ & ~dead
        order = (keys.long() & 0xffffffff) * (nx * ny) + index
        far = torch.full_like(order, 2 ** 62)
        open_ = ~(occ | spread(occ).any(0))
        born = torch.zeros_like(occ)
        while bool(open_.any()):
            o = torch.where(open_, order, far)
            join = open_ & (o < spread(o).min(0).values)
            born |= join
            open_ = open_ & ~join & ~spread(join).any(0)
        T = p["lifetime"] * (1.0 + p["lifetime_spread"] * cl.clamp(-1, 1))
        v = p["v0"] * (1.0 + p["amp_spread"] * ca.clamp(-1, 1))
        pk = T * torch.sqrt(torch.log(p["vmin_frac"] * p["v0"] / v).abs())
        zero = torch.zeros_like(t0)
        t0, life, vm, tm = (torch.where(born, new, torch.where(dead, zero, old)) for new, old in
                            ((torch.full_like(t0, t), t0), (T, life), (v, vm), (pk, tm)))
        occ = occ | born
    amp = torch.where(occ, vm * torch.exp(-((t - t0 - tm) / torch.where(occ, life, torch.ones_like(life))) ** 2), zero)
    vg = torch.zeros((2, ny, nx), dtype=torch.float64, device=DEV)
    for y, x in disk(p["r_lane"]):
        r = math.sqrt(y * y + x * x)
        f = r / p["r_granule"] if r <= p["r_granule"] else math.cos(
            0.5 * math.pi * (r - p["r_granule"]) / (p["r_lane"] - p["r_granule"])) ** 2
        a = torch.roll(amp, (y, x), (0, 1))
        vg[0] += a * (f * x / r)
        vg[1] += a * (f * y / r)
    kx, ky = _wave(nx, 1.0)[None, :], _wave(ny, 1.0)[:, None]
    k2 = kx * kx + ky * ky
    on = (k2 > 0).expand(ny, nx).clone()
    on[:, nx // 2] = False
    on[ny // 2, :] = False
    h = torch.fft.fft2(vg)
    dv = (kx * h[0] + ky * h[1]) / torch.where(k2 > 0, k2, torch.ones_like(k2))
    filt = torch.where(on, torch.exp(-(4.0 * k2 / math.pi ** 2) ** 2), torch.zeros_like(k2))
    vr = torch.stack([torch.fft.ifft2((h[0] - kx * dv) * filt).real, torch.fft.ifft2((h[1] - ky * dv) * filt).real])
    vv = vg + p["f_rot"] * vr
    return {"v": vv * torch.sqrt((vg * vg).sum() / (vv * vv).sum()), "occ": None, "par": torch.stack([t0, life, vm, tm])}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "granulation":
        return _ref_granulation(c, seed)
    s = _inputs(c, seed)
    if c["kind"] == "steps":
        return _ref_steps(s)
    if c["kind"] == "restart":
        with torch.no_grad():
            m, f = _Model(s), _start(s)
            dt, tot = m.look(f, *m.ghosts(f, f[3:5, 0][None].repeat(3, 1, 1, 1)), _deep(s["p"]))
            return {"dt": dt, "stats": tot, **_fields(f)}
    if c["kind"] == "adjoint":
        f, bz, v0, v1, st = _ref_gradient(s, _adjoint_seed(s))
        return {"lam": _fields(st), "bz": bz, "v0": v0, "v1": v1, "state": _fields(f)}
    s["target"] = _targets(s)
    f, bz, v0, v1, st = _ref_gradient(s)
    return {"state": _fields(f), "bz": bz, "v0": v0, "v1": v1, "st": _fields(st)}
