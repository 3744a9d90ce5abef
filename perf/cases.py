"""The work this framework is used for, as cases to measure.

Each case is one call sequence a user's program makes through the public entry
points (`stp.Channel`, `stp.Batch`, `stp.UNet`, `stp.poisson_residual_noalloc`),
on device arrays and on the program's own CUDA stream:

  step      set the fields of a channel, advance it a few projection steps, read
            the fields back
  solve     one pressure solve L p = rhs to 1e-8
  batch     uneven channels advanced together by one graph launch
  forward   the learned-guess network on a batch of residuals
  gradient  its loss and parameter gradient on a batch of training pairs
  residual  ||b - L p|| and b - L p on the caller's own arrays

A channel in FP32 keeps its velocities and viscosity in 32 bits, and its
pressure solves stop at 1e-8 of the right-hand side, so a program that runs one
keeps what it reads back in float32; a channel in FP64 is read in float64.  A
step leaves the constant of the pressure free, so the program removes the
volume mean, as it does before it compares or stores a pressure.

`exact` is the same discrete problem in 64 bits in plain torch: the step with
its Crank-Nicolson system iterated to rounding and its pressure solved directly
(Fourier in x and y, elimination in z), and the network without rounding.
"""
import math

import numpy as np
import torch

from paper_1511_07800_gb300 import inputs, stp

CH = (16, 32, 64, 128)  # channels of the network's levels


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _step(name, flow, nx, ny, nz, precision, steps, zline=0):
    return dict(name=name, kind="step", flow=flow, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, zline=zline)


def listed():
    return [
        # the laminar start-up check: the smallest channel anyone steps, in FP64
        _step("laminar_start_fp64", "laminar_startup", 32, 16, 32, "fp64", 2),
        # the smallest instance of the uneven-channel workload, on its own
        _step("small_channel_fp32", "os_instability", 32, 32, 32, "fp32", 3),
        # the instability study at its own grid, in the default precision
        _step("instability_fp32", "os_instability", 128, 64, 128, "fp32", 3),
        # the wall-stretched LES channel, the headline workload: z-line sweeps
        _step("les_channel_fp32", "les_channel", 256, 128, 192, "fp32", 3, zline=1),
        # the LES of the paper at its grid with the paper's point sweeps
        _step("les_paper_fp32", "les_paper", 240, 140, 120, "fp32", 2),
        # a stretched LES channel in FP64, z-line sweeps: growth rates and
        # reference runs need FP64
        _step("les_zline_fp64", "les_channel", 96, 48, 64, "fp64", 2, zline=1),
        # the pressure solve alone in FP64, as a host code with its own momentum step calls it
        dict(name="solve_fp64", kind="solve", nx=128, ny=64, nz=128, precision="fp64", zline=0, stretch=0.0),
        # the same call on rows that are no multiple of a vector, an odd level count, FP32
        dict(name="solve_ragged_fp32", kind="solve", nx=90, ny=42, nz=65, precision="fp32", zline=0, stretch=0.0),
        # uneven instability channels side by side (a parameter study)
        dict(name="batch_uneven_fp32", kind="batch", count=16, sizes="32,48,64,96", steps=2, draw=2),
        # the network's forward at the grid it is trained on (one guess a solve)
        dict(name="unet_forward", kind="forward", n=1, nx=128, ny=64, nz=128),
        # one training gradient on a batch of four pairs
        dict(name="unet_gradient", kind="gradient", n=4, nx=64, ny=32, nz=64),
        # the residual of a large channel on the caller's arrays
        dict(name="residual_noalloc", kind="residual", nx=256, ny=128, nz=192, stretch=2.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return n + (n & 1)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "solve", "solve", "batch", "forward", "gradient", "residual"])
    if kind in ("forward", "gradient"):
        top = (128, 64, 128) if kind == "forward" else (64, 32, 64)
        nx, ny, nz = (8 * _log(rng, 2, t // 8) for t in top)
        return dict(kind=kind, n=rng.choice([1, 2, 3]), nx=nx, ny=ny, nz=nz)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 14), sizes="32,48,64,96", steps=rng.randint(1, 2),
                    draw=rng.randint(3, 10 ** 6))
    if kind == "residual":
        return dict(kind=kind, nx=_log(rng, 16, 256), ny=_log(rng, 8, 128), nz=_log(rng, 8, 192),
                    stretch=rng.choice([0.0, 2.0]))
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    zline = rng.choice([0, 1])
    big = (240, 120, 180) if precision == "fp32" else (112, 56, 112)
    nx, ny, nz = _log(rng, 24, big[0]), _log(rng, 12, big[1]), _log(rng, 16, big[2])
    # channels are mostly even; rows of whole vectors are what most programs pick
    shape = rng.choice(["vector", "vector", "even", "any"])
    if shape == "vector":
        nx, ny, nz = 16 * max(2, nx // 16), _even(ny), _even(nz)
    elif shape == "even":
        nx, ny = _even(nx), _even(ny)
    if kind == "solve":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, zline=zline, stretch=2.0 if zline else 0.0)
    flow = "les_channel" if zline else rng.choice(["os_instability", "les_paper"])
    return dict(kind=kind, flow=flow, nx=nx, ny=ny, nz=nz, precision=precision, steps=rng.randint(1, 2), zline=zline)


def _shapes(case):
    """Grids of a batch: sizes drawn per dimension, as the uneven-channel workload draws them."""
    sizes = [int(s) for s in case["sizes"].split(",")]
    rng = np.random.default_rng(case["draw"])
    return [tuple(int(rng.choice(sizes)) for _ in range(3)) for _ in range(case["count"])]


def _cfg(case):
    z = case.get("zline", 0)
    return inputs.preset(case["flow"], nx=case["nx"], ny=case["ny"], nz=case["nz"], zline=z, cn_zline=z)


def _solve_cfg(case):
    return inputs.preset("os_instability", nx=case["nx"], ny=case["ny"], nz=case["nz"], stretch=case["stretch"],
                         zline=case.get("zline", 0))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dz(cfg):
    return torch.from_numpy(np.diff(inputs.zfaces(cfg))).cuda()[:, None, None]


def _uniform(shape, amp, gen):
    return (torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * amp


def _flow_fields(cfg, flow, seed):
    """Initial velocities of a flow: the base profile, a smooth wave, and uniform noise of the level its workload has."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nx, ny, nz = cfg["nx"], cfg["ny"], cfg["nz"]
    zc = torch.from_numpy(inputs.zcentres(cfg)).cuda() / (0.5 * cfg["Lz"])
    top, wave, noise = {"laminar_startup": (0.0, 1e-2, 1e-3), "os_instability": (1.0, 1e-2, 1e-2),
                        "les_channel": (1.5, 0.05, 0.15), "les_paper": (15.0, 1.0, 1.0)}[flow]
    x = torch.arange(nx, device="cuda", dtype=torch.float64) * (2 * math.pi / nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64) * (2 * math.pi / ny)
    ph = torch.rand(4, generator=gen, device="cuda", dtype=torch.float64) * (2 * math.pi)
    env = (zc * (2 - zc))[:, None, None]
    u = top * env + wave * env * torch.sin(x + ph[0])[None, None, :] * torch.cos(y + ph[1])[None, :, None]
    v = wave * env * torch.cos(x + ph[2])[None, None, :] * torch.sin(y + ph[3])[None, :, None]
    w = _uniform((nz + 1, ny, nx), noise, gen)
    w[0] = 0.0
    w[-1] = 0.0
    return u + _uniform((nz, ny, nx), noise, gen), v + _uniform((nz, ny, nx), noise, gen), w


def _rhs(cfg, seed):
    """A right-hand side as a projection step makes it: waves and noise, without a volume mean."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nx, ny, nz = cfg["nx"], cfg["ny"], cfg["nz"]
    b = torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    ph = torch.rand(3, generator=gen, device="cuda", dtype=torch.float64) * (2 * math.pi)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) * (2 * math.pi / nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64) * (2 * math.pi / ny)
    z = torch.from_numpy(inputs.zcentres(cfg)).cuda() * (math.pi / cfg["Lz"])
    b += torch.sin(x + ph[0])[None, None, :] * torch.cos(z + ph[2])[:, None, None]
    b += torch.cos(y + ph[1])[None, :, None] * torch.cos(2 * z)[:, None, None]
    return _no_mean(b, _dz(cfg))


def _no_mean(p, dz):
    return p - (p * dz).sum() / (dz.sum() * p.shape[1] * p.shape[2])


def _net_specs():
    s, cin = [], 1
    for c in CH:
        s += [(cin, c, 27), (c, c, 27)]
        cin = c
    for l in (2, 1, 0):
        s += [(CH[l + 1] + CH[l], CH[l], 27), (CH[l], CH[l], 27)]
    return s + [(CH[0], 1, 1)]


def _net_params(seed):
    rng = np.random.default_rng(seed)
    out = []
    for cin, cout, taps in _net_specs():
        out.append(rng.standard_normal(cout * cin * taps) * math.sqrt((2.0 if taps == 27 else 1.0) / (cin * taps)))
        out.append(rng.standard_normal(cout) * 0.05)
    return np.concatenate(out).astype(np.float32)


def _net_fields(case, seed):
    """Residuals of RMS one and corrections of order one, waves and noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["n"], case["nz"], case["ny"], case["nx"])
    x, t = (torch.randn(shape, generator=gen, device="cuda") for _ in range(2))
    k = torch.arange(case["nx"], device="cuda") * (2 * math.pi / case["nx"])
    ph = torch.rand(2, generator=gen, device="cuda") * (2 * math.pi)
    return 0.6 * x + torch.sin(k + ph[0]), 0.3 * t + torch.cos(k + ph[1])


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.Stream()
    s = dict(case=case, stream=stream)
    with torch.cuda.stream(stream):
        handle = stream.cuda_stream
        if kind == "step":
            cfg = _cfg(case)
            s.update(ch=stp.Channel(cfg, precision=case["precision"], stream=handle), dz=_dz(cfg),
                     fields=_flow_fields(cfg, case["flow"], seed), out=_out_buffers(cfg, cfg["les"]))
        elif kind == "solve":
            cfg = _solve_cfg(case)
            s.update(ch=stp.Channel(cfg, precision=case["precision"], stream=handle), rhs=_rhs(cfg, seed))
        elif kind == "batch":
            cfgs = [inputs.preset("os_instability", nx=nx, ny=ny, nz=nz) for nx, ny, nz in _shapes(case)]
            s["ch"] = [stp.Channel(c, precision="fp32", stream=handle) for c in cfgs]
            s["batch"] = stp.Batch(s["ch"], stream=handle)
            s["fields"] = [_flow_fields(c, "os_instability", seed + 1000 * i) for i, c in enumerate(cfgs)]
            s["dz"] = [_dz(c) for c in cfgs]
            s["out"] = [_out_buffers(c, 0) for c in cfgs]
        elif kind in ("forward", "gradient"):
            net = stp.UNet(case["n"], case["nz"], case["ny"], case["nx"], stream=handle)
            net.set_params(_net_params(seed))
            x, t = _net_fields(case, seed)
            s.update(net=net, x=x, t=t, y=torch.empty_like(x),
                     grad=torch.empty(stp.UNet.param_count(), device="cuda"))
        else:
            cfg = _solve_cfg(case)
            gen = torch.Generator(device="cuda").manual_seed(seed + 1)
            p = torch.randn((case["nz"], case["ny"], case["nx"]), generator=gen, device="cuda", dtype=torch.float64)
            s.update(cfg=cfg, b=_rhs(cfg, seed), p=p, r=torch.empty_like(p))
    return s


def _out_buffers(cfg, les):
    nx, ny, nz = cfg["nx"], cfg["ny"], cfg["nz"]
    new = lambda n: torch.empty((n, ny, nx), device="cuda", dtype=torch.float64)  # noqa: E731
    out = dict(u=new(nz), v=new(nz), w=new(nz + 1), p=new(nz))
    if les:
        out["nu"] = new(nz)
    return out


def _read(ch, out, dz, precision):
    """The channel's fields as the program keeps them."""
    ch.get_fields(out)
    got = dict(out, p=_no_mean(out["p"], dz))
    return {k: v.float() if precision == "fp32" else v for k, v in got.items()}


def run(s):
    case = s["case"]
    kind = case["kind"]
    with torch.cuda.stream(s["stream"]):
        if kind == "step":
            s["ch"].set_fields(*s["fields"])
            s["ch"].step(case["steps"])
            return _read(s["ch"], s["out"], s["dz"], case["precision"])
        if kind == "solve":
            p = torch.zeros_like(s["rhs"])
            s["ch"].poisson_solve(s["rhs"], p)
            return p.float() if case["precision"] == "fp32" else p
        if kind == "batch":
            for ch, f in zip(s["ch"], s["fields"]):
                ch.set_fields(*f)
            s["batch"].step(case["steps"])
            return [_read(ch, out, dz, "fp32") for ch, out, dz in zip(s["ch"], s["out"], s["dz"])]
        if kind == "forward":
            s["net"].forward(s["x"], s["y"])
            return s["y"]
        if kind == "gradient":
            loss = s["net"].gradient(s["x"], s["t"], s["grad"])
            return dict(loss=torch.tensor(loss), grad=s["grad"])
        norm = stp.poisson_residual_noalloc(s["cfg"], s["p"], s["b"], s["r"], stream=s["stream"].cuda_stream)
        return dict(norm=norm, r=s["r"])


def work(case):
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        vox = case["n"] * case["nz"] * case["ny"] * case["nx"]
        level = [0] * 2 + [1] * 2 + [2] * 2 + [3] * 2 + [2] * 2 + [1] * 2 + [0] * 2 + [0]
        flops = sum(2.0 * ci * co * t * vox / 8 ** l for (ci, co, t), l in zip(_net_specs(), level))
        weights = sum(ci * co * t + co for ci, co, t in _net_specs())
        if kind == "forward":
            return dict(bytes=8.0 * vox + 2.0 * weights, flops=flops)
        return dict(bytes=8.0 * vox + 6.0 * weights, flops=3.0 * flops)
    if kind == "residual":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=24.0 * n, flops=14.0 * n)
    if kind == "solve":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=24.0 * n, flops=14.0 * n)
    # u, v, w in and u, v, w, p out, and about 400 operations a cell and step outside the solve
    cells = sum(a * b * c for a, b, c in _shapes(case)) if kind == "batch" else case["nx"] * case["ny"] * case["nz"]
    return dict(bytes=(3 * 8.0 + 4 * 8.0) * cells, flops=400.0 * cells * case["steps"])


# ---------------------------------------------------------------------------
# 64 bits, plain torch
# ---------------------------------------------------------------------------
def _xp(a):
    return torch.roll(a, -1, 2)


def _xm(a):
    return torch.roll(a, 1, 2)


def _yp(a):
    return torch.roll(a, -1, 1)


def _ym(a):
    return torch.roll(a, 1, 1)


class _Grid:
    def __init__(self, cfg):
        nz, Lz, g = cfg["nz"], cfg["Lz"], cfg.get("stretch", 0.0)
        q = np.arange(nz + 1) / nz
        zf = 0.5 * Lz * (1 + np.tanh(g * (2 * q - 1)) / np.tanh(g)) if g > 0 else Lz * q
        zf[0], zf[-1] = 0.0, Lz
        dz, zc = np.diff(zf), 0.5 * (zf[1:] + zf[:-1])
        hz = np.diff(zc)                                          # faces 1 .. nz-1
        dzf = np.concatenate([dz[:1], hz, dz[-1:]])               # faces 0 .. nz
        up = np.concatenate([hz, dz[-1:]]) + np.concatenate([dz[:1], hz])
        self.cfg, self.dx, self.dy = cfg, cfg["Lx"] / cfg["nx"], cfg["Ly"] / cfg["ny"]
        put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()[:, None, None]  # noqa: E731
        self.dz, self.hz, self.dzf, self.up, self.zc = put(dz), put(hz), put(dzf), put(up), put(zc)


def _ghost(a):
    return torch.cat([-a[:1], a, -a[-1:]])


def _edges(nu):
    """nu at the xy, xz and yz edges."""
    s = nu + _xm(nu)
    t = nu + _ym(nu)
    pad = lambda a: torch.cat([a[:1], a, a[-1:]])  # noqa: E731
    s2, t2 = pad(s), pad(t)
    return 0.25 * (s + _ym(s)), 0.25 * (s2[1:] + s2[:-1]), 0.25 * (t2[1:] + t2[:-1])


def _eddy(g, u, v, w):
    c, dx, dy = g.cfg, g.dx, g.dy
    e12 = 0.5 * ((u - _ym(u)) / dy + (v - _xm(v)) / dx)
    ug, vg = _ghost(u), _ghost(v)
    e13 = 0.5 * ((ug[1:] - ug[:-1]) / g.dzf + (w - _xm(w)) / dx)
    e23 = 0.5 * ((vg[1:] - vg[:-1]) / g.dzf + (w - _ym(w)) / dy)
    s12 = e12 + _xp(e12)
    s12 = 0.25 * (s12 + _yp(s12))
    s13 = e13 + _xp(e13)
    s13 = 0.25 * (s13[1:] + s13[:-1])
    s23 = e23 + _yp(e23)
    s23 = 0.25 * (s23[1:] + s23[:-1])
    s11, s22, s33 = (_xp(u) - u) / dx, (_yp(v) - v) / dy, (w[1:] - w[:-1]) / g.dz
    mag = torch.sqrt(2 * (s11 ** 2 + s22 ** 2 + s33 ** 2) + 4 * (s12 ** 2 + s13 ** 2 + s23 ** 2))
    d = torch.minimum(g.zc, c["Lz"] - g.zc) * c["re_tau"] / (0.5 * c["Lz"])
    lm = c["cs"] * 2 * (dx * dy * g.dz) ** (1 / 3) * (1 - torch.exp(-d / c["vd_a"]))
    return c["nu"] + lm ** 2 * mag


def _explicit(g, u, v, w, nu, f):
    """-u.grad u + d_j(nu d_i u_j) + f of the three components (w on the inner faces)."""
    dx, dy, dz, hz = g.dx, g.dy, g.dz, g.hz
    xy, xz, yz = _edges(nu)
    dxc = lambda a: (_xp(a) - _xm(a)) / (2 * dx)  # noqa: E731
    dyc = lambda a: (_yp(a) - _ym(a)) / (2 * dy)  # noqa: E731
    ug, vg = _ghost(u), _ghost(v)
    t = v + _xm(v)
    r = w + _xm(w)
    nu_u = -(u * dxc(u) + 0.25 * (t + _yp(t)) * dyc(u) + 0.25 * (r[1:] + r[:-1]) * (ug[2:] - ug[:-2]) / g.up)
    fx, fy, fz = nu * (_xp(u) - u) / dx, xy * (v - _xm(v)) / dx, xz * (w - _xm(w)) / dx
    nu_u += (fx - _xm(fx)) / dx + (_yp(fy) - fy) / dy + (fz[1:] - fz[:-1]) / dz + f
    t = u + _ym(u)
    r = w + _ym(w)
    nu_v = -(0.25 * (t + _xp(t)) * dxc(v) + v * dyc(v) + 0.25 * (r[1:] + r[:-1]) * (vg[2:] - vg[:-2]) / g.up)
    fx, fy, fz = xy * (u - _ym(u)) / dy, nu * (_yp(v) - v) / dy, yz * (w - _ym(w)) / dy
    nu_v += (_xp(fx) - fx) / dx + (fy - _ym(fy)) / dy + (fz[1:] - fz[:-1]) / dz
    wi = w[1:-1]
    t = u + _xp(u)
    r = v + _yp(v)
    nu_w = -(0.25 * (t[1:] + t[:-1]) * dxc(wi) + 0.25 * (r[1:] + r[:-1]) * dyc(wi) +
             wi * (w[2:] - w[:-2]) / (dz[1:] + dz[:-1]))
    fx, fy, fz = xz[1:-1] * (u[1:] - u[:-1]) / hz, yz[1:-1] * (v[1:] - v[:-1]) / hz, nu * (w[1:] - w[:-1]) / dz
    nu_w += (_xp(fx) - fx) / dx + (_yp(fy) - fy) / dy + (fz[1:] - fz[:-1]) / hz
    return nu_u, nu_v, nu_w


class _Diffusion:
    """d_j(nu d_j a) of each component, and its diagonal weight."""

    def __init__(self, g, nu):
        self.g, self.nu = g, nu
        self.xy, self.xz, self.yz = _edges(nu)
        one = torch.ones_like(g.dz)
        gu, gd = one.clone(), one.clone()
        gu[-1] = 2.0
        gd[0] = 2.0
        wall = lambda e: (gu * e[1:] / g.dzf[1:] + gd * e[:-1] / g.dzf[:-1]) / g.dz  # noqa: E731
        dx2, dy2 = g.dx ** 2, g.dy ** 2
        xy, xz, yz = self.xy, self.xz, self.yz
        k = nu / g.dz
        self.diag = ((nu + _xm(nu)) / dx2 + (xy + _yp(xy)) / dy2 + wall(xz),
                     (xy + _xp(xy)) / dx2 + (nu + _ym(nu)) / dy2 + wall(yz),
                     ((xz + _xp(xz)) / dx2 + (yz + _yp(yz)) / dy2)[1:-1] + (k[1:] + k[:-1]) / g.hz)

    def __call__(self, c, a):
        g = self.g
        if c == 2:
            z = torch.zeros_like(a[:1])
            w = torch.cat([z, a, z])
            fx, fy = self.xz[1:-1] * (a - _xm(a)) / g.dx, self.yz[1:-1] * (a - _ym(a)) / g.dy
            fz = self.nu * (w[1:] - w[:-1]) / g.dz
            return (_xp(fx) - fx) / g.dx + (_yp(fy) - fy) / g.dy + (fz[1:] - fz[:-1]) / g.hz
        ag = _ghost(a)
        fz = (self.xz if c == 0 else self.yz) * (ag[1:] - ag[:-1]) / g.dzf
        if c == 0:
            fx, fy = self.nu * (_xp(a) - a) / g.dx, self.xy * (a - _ym(a)) / g.dy
            h = (fx - _xm(fx)) / g.dx + (_yp(fy) - fy) / g.dy
        else:
            fx, fy = self.xy * (a - _xm(a)) / g.dx, self.nu * (_yp(a) - a) / g.dy
            h = (_xp(fx) - fx) / g.dx + (fy - _ym(fy)) / g.dy
        return h + (fz[1:] - fz[:-1]) / g.dz


def _implicit(D, c, rhs, h):
    """(I - h D) a = rhs, Jacobi iteration to rounding."""
    a = rhs.clone()
    scale = rhs.abs().max()
    for it in range(400):
        d = (rhs - a + h * D(c, a)) / (1 + h * D.diag[c])
        a += d
        if it % 8 == 7 and d.abs().max() <= 1e-15 * scale:
            break
    return a


def _poisson(g, b):
    """L p = b with no volume mean: Fourier in x and y, elimination in z."""
    c = g.cfg
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    F = torch.fft.rfft2(b)
    m = torch.arange(F.shape[2], device="cuda", dtype=torch.float64)
    n = torch.arange(ny, device="cuda", dtype=torch.float64)
    lam = (4 / g.dx ** 2 * torch.sin(math.pi * m / nx) ** 2)[None, :] + (4 / g.dy ** 2 * torch.sin(math.pi * n / ny) ** 2)[:, None]
    dz, hz = g.dz.flatten().tolist(), g.hz.flatten().tolist()
    up = [1 / (hz[k] * dz[k]) if k < nz - 1 else 0.0 for k in range(nz)]
    dn = [1 / (hz[k - 1] * dz[k]) if k > 0 else 0.0 for k in range(nz)]
    cp, dp = [None] * nz, [None] * nz
    for k in range(nz):
        di = -(lam + up[k] + dn[k])
        if k == 0:
            di[0, 0] -= up[0]                 # the constant: any value of the lowest level does
        den = di - dn[k] * cp[k - 1] if k else di
        cp[k] = up[k] / den
        dp[k] = (F[k] - dn[k] * dp[k - 1]) / den if k else F[k] / den
    P = torch.empty_like(F)
    P[nz - 1] = dp[nz - 1]
    for k in range(nz - 2, -1, -1):
        P[k] = dp[k] - cp[k] * P[k + 1]
    return _no_mean(torch.fft.irfft2(P, s=(ny, nx)), g.dz)


def _exact_steps(cfg, fields, steps):
    g = _Grid(cfg)
    u, v, w = (a.clone() for a in fields)
    dt, h = cfg["dt"], 0.5 * cfg["dt"]
    f = cfg["fx"] if cfg["forcing"] == 0 else 0.0
    past = []
    zero = torch.zeros_like(w[:1])
    for n in range(steps):
        nu = _eddy(g, u, v, w) if cfg["les"] else torch.full_like(u, cfg["nu"])
        D = _Diffusion(g, nu)
        past = [_explicit(g, u, v, w, nu, f)] + past[:2]
        coef = [(1.0,), (1.5, -0.5), (23 / 12, -16 / 12, 5 / 12)][min(n, 2)]
        comp = []
        for c, a in enumerate((u, v, w[1:-1])):
            rhs = a + h * D(c, a) + dt * sum(q * N[c] for q, N in zip(coef, past))
            comp.append(_implicit(D, c, rhs, h))
        u, v, w = comp[0], comp[1], torch.cat([zero, comp[2], zero])
        div = (_xp(u) - u) / g.dx + (_yp(v) - v) / g.dy + (w[1:] - w[:-1]) / g.dz
        p = _poisson(g, div / dt)
        u = u - dt * (p - _xm(p)) / g.dx
        v = v - dt * (p - _ym(p)) / g.dy
        w[1:-1] -= dt * (p[1:] - p[:-1]) / g.hz
        if cfg["forcing"] == 1:
            u = u + cfg["ubulk"] - (u * g.dz).sum() / (cfg["Lz"] * cfg["nx"] * cfg["ny"])
    out = dict(u=u, v=v, w=w, p=p)
    if cfg["les"]:
        out["nu"] = nu
    return out


def _conv(x, wt, bias):
    """3 x 3 x 3 convolution of [n][z][y][x][c], periodic in x and y, zero past the walls."""
    n, d, hh, ww, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 0, 0, 0, 0, 1, 1))
    y = bias.expand(n, d, hh, ww, -1)
    for t in range(27):
        kz, ky, kx = t // 9, (t // 3) % 3 - 1, t % 3 - 1
        y = y + torch.roll(xp[:, kz:kz + d], (-ky, -kx), (2, 3)) @ wt[:, :, t].T
    return y


def _network(theta, x):
    q, layers = 0, []
    for ci, co, t in _net_specs():
        wt = theta[q:q + co * ci * t].reshape(co, ci, t)
        q += co * ci * t
        layers.append((wt, theta[q:q + co]))
        q += co
    it = iter(layers)
    block = lambda a: torch.relu(_conv(torch.relu(_conv(a, *next(it))), *next(it)))  # noqa: E731

    def pool(a):
        n, d, hh, ww, c = a.shape
        return a.reshape(n, d // 2, 2, hh // 2, 2, ww // 2, 2, c).mean((2, 4, 6))

    def grow(a):
        return a.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    a, skips = x[..., None], []
    for l in range(4):
        a = block(a)
        if l < 3:
            skips.append(a)
            a = pool(a)
    for l in (2, 1, 0):
        a = block(torch.cat([grow(a), skips[l]], -1))
    wt, bias = next(it)
    return (a @ wt[:, :, 0].T + bias)[..., 0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        cfg = _cfg(case)
        return _exact_steps(cfg, _flow_fields(cfg, case["flow"], seed), case["steps"])
    if kind == "solve":
        cfg = _solve_cfg(case)
        return _poisson(_Grid(cfg), _rhs(cfg, seed))
    if kind == "batch":
        cfgs = [inputs.preset("os_instability", nx=nx, ny=ny, nz=nz) for nx, ny, nz in _shapes(case)]
        return [_exact_steps(c, _flow_fields(c, "os_instability", seed + 1000 * i), case["steps"])
                for i, c in enumerate(cfgs)]
    if kind == "residual":
        cfg = _solve_cfg(case)
        g = _Grid(cfg)
        gen = torch.Generator(device="cuda").manual_seed(seed + 1)
        p = torch.randn((case["nz"], case["ny"], case["nx"]), generator=gen, device="cuda", dtype=torch.float64)
        fz = torch.zeros((case["nz"] + 1,) + tuple(p.shape[1:]), device="cuda", dtype=torch.float64)
        fz[1:-1] = (p[1:] - p[:-1]) / g.hz
        r = _rhs(cfg, seed) - ((_xp(p) - 2 * p + _xm(p)) / g.dx ** 2 + (_yp(p) - 2 * p + _ym(p)) / g.dy ** 2 +
                               (fz[1:] - fz[:-1]) / g.dz)
        return dict(norm=float(r.norm()), r=r)
    x, t = (a.double() for a in _net_fields(case, seed))
    theta = torch.from_numpy(_net_params(seed)).cuda().double()
    if kind == "forward":
        with torch.no_grad():
            return _network(theta, x)
    theta.requires_grad_(True)
    loss = ((_network(theta, x) - t) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, theta)
    return dict(loss=loss.detach().float().cpu(), grad=grad)
