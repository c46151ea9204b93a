"""Performance cases of the free-surface lattice Boltzmann library: what a
user's program has it do, through the public Python entry points.

A case is a dict of plain values; `prepare` builds what the program holds
before the call, `run` makes the call, `work` states the bytes and operations
the path cannot do without, `exact` gives the outputs in 64-bit arithmetic of
plain torch (independent of the library) where they have such a value.

Kinds of case
  steps      `Sim.step(n)`: time steps of a simulation in motion, in the
             set-ups droplet (periodic), cap (sessile droplet on a wall,
             wetting), pool (dense liquid between walls), bubble (gas bubble in
             liquid, bubble model) and pair (two droplets, learned curvature)
  curvature  `Sim.curvature` by every model on one state
  train      one epoch of the learned curvature and its held-out evaluation
  stencils   generation of training stencils
  window     forward and reverse pass of an adjoint window
  setup      fill levels, initial state and total mass of a new simulation
"""
import functools
import math
import random

import numpy as np
import torch

from paper_1509_07691_gb300 import fsl as F

DEV = "cuda"
LIQ, IF, GAS, OBS = 1, 2, 4, 8
CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0)
CY = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1)
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
CURV = {"lsqr": F.CURV_LSQR, "fd": F.CURV_FD, "mlp": F.CURV_MLP, "tr": F.CURV_TR}
STORE = {"f32": F.F32, "f16": F.F16_OFS, "bf16": F.BF16_OFS}
SHIFT = 8
LR = 2e-4


# ---- the cases -----------------------------------------------------------------
def listed():
    return [
        # static droplet of the Laplace test: the smallest simulation, bound by latency and launches
        dict(name="droplet32", kind="steps", setup="droplet", nx=32, ny=32, nz=32, R=8.0, curv="lsqr", storage="f32",
             trt=False, tau=1.0, sigma=1e-4, theta=90.0, steps=10),
        # oscillating droplet of the benchmark line: an ordinary droplet run, sparse in its box
        dict(name="oscillating256", kind="steps", setup="droplet", nx=256, ny=256, nz=256, R=40.0, curv="lsqr",
             storage="f32", trt=False, tau=0.6, sigma=1e-3, theta=90.0, steps=10),
        # sessile droplet spreading on a wall: contact-line fits, bounce-back, the TRT collision
        dict(name="sessile128", kind="steps", setup="cap", nx=128, ny=128, nz=64, R=30.0, curv="lsqr", storage="f32",
             trt=True, tau=0.8, sigma=5e-4, theta=60.0, steps=10),
        # dense liquid between walls: the stream-collide at the memory bandwidth
        dict(name="pool256", kind="steps", setup="pool", nx=256, ny=256, nz=256, R=64.0, curv="lsqr", storage="f32",
             trt=False, tau=0.6, sigma=1e-3, theta=90.0, steps=4),
        # the same in 16-bit storage, on a grid whose rows end in partial segments
        dict(name="pool251_f16", kind="steps", setup="pool", nx=251, ny=251, nz=256, R=62.75, curv="lsqr",
             storage="f16", trt=False, tau=0.6, sigma=1e-3, theta=90.0, steps=4),
        # gas bubble carried by liquid (Renardy's moving frame): FD curvature, bubble model, mostly liquid
        dict(name="bubble96_fd", kind="steps", setup="bubble", nx=96, ny=96, nz=96, R=12.0, curv="fd", storage="f32",
             trt=False, tau=0.6728, sigma=4.935168e-5, theta=90.0, steps=10),
        # two droplets about to merge with the learned curvature in the step: the largest simulation
        dict(name="coalescence384_mlp", kind="steps", setup="pair", nx=384, ny=384, nz=384, R=48.0, curv="mlp",
             storage="f32", trt=False, tau=0.7, sigma=1e-3, theta=90.0, steps=4),
        # curvature of a state by every model of the comparison
        dict(name="curvature256", kind="curvature", nx=256, ny=256, nz=256, R=40.0),
        # training of the learned curvature: an epoch of batches of 4096, then the held-out set
        dict(name="train4096", kind="train", rows=65536, batch=4096, held=10007),
        # training data: stencils by sub-sampling of ellipsoids, with noise
        dict(name="stencils", kind="stencils", n=65536, sub=8),
        # one evaluation of the surface fit: 50 frozen steps and their reverse, checkpoints every 10
        dict(name="window64", kind="window", nx=64, ny=64, nz=64, R=16.0, window=50, every=10),
        # a new simulation: fill levels of the shape, initial state, total mass
        dict(name="setup256", kind="setup", shape="mode2", nx=256, ny=256, nz=256, R=40.0, storage="f32"),
    ]


def _log(rng, lo, hi):
    return lo * math.exp(rng.random() * math.log(hi / lo))


def draw(rng):
    kind = rng.choice(["droplet", "droplet", "cap", "pool", "bubble", "pair", "curvature", "train", "stencils",
                       "window", "setup"])
    if kind in ("droplet", "bubble"):
        top = 256 if kind == "droplet" else 128
        n = [int(_log(rng, 28, top)) for _ in range(3)]
        R = round(min(n) * rng.uniform(0.12, 0.3), 2)
        return dict(kind="steps", setup=kind, nx=n[0], ny=n[1], nz=n[2], R=max(4.0, R),
                    curv=rng.choice(["lsqr", "lsqr", "fd", "tr"]), storage=rng.choice(["f32", "f32", "f16", "bf16"]),
                    trt=rng.random() < 0.3, tau=round(rng.uniform(0.6, 1.0), 3),
                    sigma=round(_log(rng, 5e-5, 1e-3), 6), theta=90.0, steps=rng.randint(1, 10))
    if kind == "cap":
        nx, nz = int(_log(rng, 40, 160)), int(_log(rng, 24, 80))
        return dict(kind="steps", setup="cap", nx=nx, ny=nx + rng.randint(0, 9), nz=nz,
                    R=round(min(nz - 6, nx / 2 - 4) * rng.uniform(0.5, 0.9), 2), curv=rng.choice(["lsqr", "lsqr", "fd"]),
                    storage="f32", trt=rng.random() < 0.7, tau=round(rng.uniform(0.6, 1.0), 3),
                    sigma=round(_log(rng, 1e-4, 1e-3), 6), theta=float(rng.choice([30, 60, 90, 120])),
                    steps=rng.randint(1, 10))
    if kind == "pool":
        nx, nz = int(_log(rng, 48, 256)), int(_log(rng, 48, 256))
        return dict(kind="steps", setup="pool", nx=nx, ny=nx, nz=nz, R=nx / max(1, round(nx / 64)), curv="lsqr",
                    storage=rng.choice(["f32", "f16", "bf16"]), trt=rng.random() < 0.3,
                    tau=round(rng.uniform(0.6, 1.0), 3), sigma=round(_log(rng, 1e-4, 1e-3), 6), theta=90.0,
                    steps=rng.randint(1, 4))
    if kind == "pair":
        n = int(_log(rng, 96, 384))
        return dict(kind="steps", setup="pair", nx=n, ny=n - rng.randint(0, 9), nz=n - rng.randint(0, 9),
                    R=round(n / 8, 2), curv="mlp", storage="f32", trt=False, tau=0.7, sigma=1e-3, theta=90.0,
                    steps=rng.randint(1, 4))
    if kind == "curvature":
        n = [int(_log(rng, 32, 256)) for _ in range(3)]
        return dict(kind="curvature", nx=n[0], ny=n[1], nz=n[2], R=round(max(4.0, min(n) * rng.uniform(0.12, 0.3)), 2))
    if kind == "train":
        batch = int(_log(rng, 256, 16384))
        return dict(kind="train", rows=batch * rng.randint(1, 4) + rng.randint(0, 99), batch=batch,
                    held=int(_log(rng, 100, 20000)))
    if kind == "stencils":
        return dict(kind="stencils", n=int(_log(rng, 500, 65536)), sub=rng.choice([4, 8, 8, 10]))
    if kind == "window":
        n, w = int(_log(rng, 32, 64)), rng.randint(5, 50)
        return dict(kind="window", nx=n, ny=n + rng.randint(0, 5), nz=n, R=round(n * rng.uniform(0.2, 0.3), 2), window=w,
                    every=rng.randint(2, 10))
    n = [int(_log(rng, 40, 256)) for _ in range(3)]
    return dict(kind="setup", shape=rng.choice(["sphere", "mode2", "cap", "pool"]), nx=n[0], ny=n[1], nz=n[2],
                R=round(min(n) * rng.uniform(0.15, 0.4), 2), storage=rng.choice(["f32", "f32", "f16"]))


# ---- shapes and initial flow, in plain torch -------------------------------------
def _grid(c):
    return c["nz"], c["ny"], c["nx"]


def _geometry(c, seed):
    """Plain numbers of the shape of a case: kind, centre(s), radius, ..."""
    r = random.Random(seed)
    off = [math.floor((r.random() - 0.5) * 1024) / 1024 for _ in range(3)]
    mid = [c["nx"] / 2, c["ny"] / 2, c["nz"] / 2]
    kind, R = c.get("setup") or c.get("shape") or "droplet", c["R"]
    cen = tuple(m + o for m, o in zip(mid, off))
    if kind in ("droplet", "mode2"):
        return dict(kind="mode2", c=cen, R=R, eps2=0.1 if kind == "mode2" or c.get("nx", 0) > 40 else 0.0)
    if kind in ("bubble", "sphere"):
        return dict(kind="sphere", c=cen, R=R, invert=int(kind == "bubble"))
    if kind in ("cap", "window"):
        return dict(kind="cap", c=(cen[0], cen[1], 0.5), R=R, zw=0.5)
    if kind == "pair":
        R2 = R * 2 / 3
        gap = R + R2 + 4.0
        return dict(kind="two_spheres", c=(mid[0] - gap * 0.5 + off[0], cen[1], cen[2]), R=R,
                    c2=(mid[0] + gap * 0.5 + off[0], cen[1], cen[2]), R2=R2)
    return dict(kind="pool", h0=c["nz"] * 0.625 + off[2], amp=2.0, wavelength=R)  # R: the wave length


def _inside(g, x, y, z):
    """Whether points (broadcast float64 tensors) lie in the shape."""
    if g["kind"] == "pool":
        k = 2 * math.pi / g["wavelength"]
        s = z < g["h0"] + g["amp"] * torch.sin(k * x) * torch.sin(k * y)
    else:
        dx, dy, dz = x - g["c"][0], y - g["c"][1], z - g["c"][2]
        r2 = dx * dx + dy * dy + dz * dz
        if g["kind"] == "mode2":
            mu2 = dz * dz / r2.clamp(min=1e-300)
            s = r2.sqrt() <= g["R"] * (1 + g["eps2"] * (1.5 * mu2 - 0.5))
        else:
            s = r2 <= g["R"] ** 2
        if g["kind"] == "cap":
            s = s & (z >= g["zw"])
        if g["kind"] == "two_spheres":
            ex, ey, ez = x - g["c2"][0], y - g["c2"][1], z - g["c2"][2]
            s = s | (ex * ex + ey * ey + ez * ez <= g["R2"] ** 2)
    return ~s if g.get("invert") else s


def _fill(c, g, sub=16):
    """Fill levels (float64) by sub-sampling: the fraction of sub^3 sample points inside."""
    nz, ny, nx = _grid(c)
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) for n in (nx, ny, nz)]
    x, y, z = ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)
    phi = _inside(g, x, y, z).expand(nz, ny, nx).double().contiguous()
    # cells whose 5x5x5 half-cell lattice of points is not all in or all out are sampled
    h = (-1.0, -0.5, 0.0, 0.5, 1.0)
    n_in = torch.zeros_like(phi, dtype=torch.int16)
    for a in h:
        for b in h:
            for d in h:
                n_in += _inside(g, x + a, y + b, z + d)
    cells = ((n_in > 0) & (n_in < 125)).reshape(-1).nonzero().reshape(-1)
    s = (torch.arange(sub, device=DEV, dtype=torch.float64) + 0.5) / sub - 0.5
    flat = phi.view(-1)
    for part in cells.split(16384):
        px = (part % nx).double().view(-1, 1, 1, 1) + s.view(1, 1, 1, -1)
        py = (part // nx % ny).double().view(-1, 1, 1, 1) + s.view(1, 1, -1, 1)
        pz = (part // (nx * ny)).double().view(-1, 1, 1, 1) + s.view(1, -1, 1, 1)
        flat[part] = _inside(g, px, py, pz).expand(-1, sub, sub, sub).double().mean(dim=(1, 2, 3))
    return phi


def _walls(c):
    """Obstacle layers at both ends of z for the walled set-ups, else None."""
    if (c.get("setup") or c.get("kind")) not in ("cap", "pool", "window"):
        return None
    m = torch.zeros(_grid(c), dtype=torch.uint8, device=DEV)
    m[0] = m[-1] = 1
    return m


def _velocity(c, g, seed):
    """Initial velocity (ux, uy, uz) of the liquid: each set-up caught in motion,
    so that cells convert from the first step on as they do in a running simulation."""
    nz, ny, nx = _grid(c)
    x = torch.arange(nx, device=DEV, dtype=torch.float32).view(1, 1, -1)
    y = torch.arange(ny, device=DEV, dtype=torch.float32).view(1, -1, 1)
    z = torch.arange(nz, device=DEV, dtype=torch.float32).view(-1, 1, 1)
    amp = random.Random(seed + 77).uniform(0.9, 1.1)
    if c["setup"] == "bubble":
        return 0.0024 * amp, 0.0, 0.0
    if c["setup"] == "pair":  # towards each other
        m = c["nx"] / 2
        return torch.where(x < m, 1.0, -1.0) * (1e-3 * amp), 0.0, 0.0
    if c["setup"] == "pool":
        k = 2 * math.pi / g["wavelength"]
        e = 1e-3 * amp * torch.exp(math.sqrt(2) * k * (z - g["h0"]).clamp(max=4.0))
        return (e * torch.cos(k * x) * torch.sin(k * y) / math.sqrt(2), e * torch.sin(k * x) * torch.cos(k * y) / math.sqrt(2),
                e * torch.sin(k * x) * torch.sin(k * y))
    s = 1.4e-3 * amp / g["R"]  # straining flow: the swing of a mode-2 oscillation, or a cap that spreads
    return s * (x - g["c"][0]), s * (y - g["c"][1]), -2 * s * (z - g["c"][2])


def _feq(q, rho, u):
    cu = CX[q] * u[0] + CY[q] * u[1] + CZ[q] * u[2]
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    return W[q] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)


def _initial_types(phi, obs):
    t = torch.where(phi <= 0, GAS, torch.where(phi >= 1, LIQ, IF)).to(torch.uint8)
    if obs is not None:
        t[obs > 0] = OBS
    gas = t == GAS
    near = torch.zeros_like(gas)
    for q in range(1, 19):
        near |= torch.roll(gas, (CZ[q], CY[q], CX[q]), (0, 1, 2))
    t[(t == LIQ) & near] = IF
    return t


def _initial_pdfs(c, g, seed, t):
    """PDFs of the initial flow as stored (FP32, or scaled 16-bit offsets); w_q away from the fluid."""
    dt = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[c["storage"]]
    u = _velocity(c, g, seed)
    fluid = (t & (LIQ | IF)) > 0
    f = torch.empty((19,) + _grid(c), dtype=dt, device=DEV)
    for q in range(19):
        v = torch.where(fluid, _feq(q, 1.0, u), W[q])
        f[q] = (v if c["storage"] == "f32" else (v - W[q]) * 2.0 ** SHIFT).to(dt)
    return f


@functools.lru_cache(maxsize=1)
def _network():
    """A learned curvature as training leaves it: two fixed random layers and a
    readout fitted to sphere stencils.  FP32 numpy arrays, the same for every seed."""
    gen = torch.Generator().manual_seed(20)
    W1 = torch.randn(128, 128, generator=gen) / math.sqrt(125)
    W1[:, 125:] = 0
    W2 = torch.randn(128, 128, generator=gen) / math.sqrt(128)
    b1, b2 = 0.1 * torch.randn(128, generator=gen), 0.1 * torch.randn(128, generator=gen)
    X, t = _sphere_stencils(21, 16384)
    r = lambda v: v.bfloat16().double().to(DEV)  # noqa: E731
    gelu = torch.nn.functional.gelu
    h = gelu(gelu(X.double() @ r(W1).T + b1.double().to(DEV)) @ r(W2).T + b2.double().to(DEV))
    A = torch.cat([h, torch.ones_like(h[:, :1])], 1)
    wgt = 1 / (t.double() ** 2 + 7e-5).sqrt().unsqueeze(1)
    Aw, tw = (A * wgt).cpu(), (t.double().unsqueeze(1) * wgt).cpu()
    eye = torch.eye(129, dtype=torch.float64)
    sol = torch.linalg.solve(Aw.T @ Aw + eye, Aw.T @ tw).squeeze(1)
    a = lambda v: v.float().numpy()  # noqa: E731
    return dict(W1=a(W1), b1=a(b1), W2=a(W2), b2=a(b2), w3=a(sol[:128]), b3=a(sol[128:]))


def _midway():
    """The network part-way through training: its readout not yet at the optimum."""
    net = dict(_network())
    net["w3"] = net["w3"] * np.float32(0.95)
    return net


def _moments(r):
    """Adam's moments as many steps have left them, at the scale of the gradients (readout larger)."""
    scale = torch.full((33153,), 3e-3, device=DEV)
    scale[32768:32896] = scale[33152:] = 5e-2
    v = (scale * (0.5 + torch.rand(scale.numel(), generator=r, device=DEV))) ** 2
    return 0.1 * v.sqrt() * torch.randn(scale.numel(), generator=r, device=DEV), v


def _sphere_stencils(seed, n, sub=4):
    """Canonical BF16 rows (2 phi - 1 on 5x5x5, zero padded) of spheres, radii
    log-uniform in [2, 60], and their curvature: stencils made without the library."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    u = torch.rand(n, 5, generator=gen, device=DEV, dtype=torch.float64)
    R = 2 * torch.exp(u[:, 0] * math.log(30.0))
    sign = torch.where(u[:, 1] < 0.3, -1.0, 1.0)
    d = torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64).abs()
    d = (d / d.norm(dim=1, keepdim=True)).sort(dim=1, descending=True).values
    cen = (R * sign).unsqueeze(1) * d + (u[:, 2:5] - 0.5) * 0.9
    e = torch.arange(125, device=DEV)
    s = (torch.arange(sub, device=DEV, dtype=torch.float64) + 0.5) / sub - 0.5
    X = torch.zeros(n, 128, dtype=torch.bfloat16, device=DEV)
    for k in range(0, n, 8192):
        cc = cen[k: k + 8192].float()
        p = [(e // w % 5 - 2).float().view(1, 125, 1, 1, 1) - cc[:, a].view(-1, 1, 1, 1, 1) for a, w in ((0, 25), (1, 5), (2, 1))]
        sf = s.float()
        ins = ((p[0] + sf.view(1, 1, -1, 1, 1)) ** 2 + (p[1] + sf.view(1, 1, 1, -1, 1)) ** 2 +
               (p[2] + sf.view(1, 1, 1, 1, -1)) ** 2) <= (R[k: k + 8192].float() ** 2).view(-1, 1, 1, 1, 1)
        phi = ins.float().mean(dim=(2, 3, 4))
        phi = torch.where(sign[k: k + 8192].view(-1, 1) < 0, 1 - phi, phi)
        X[k: k + 8192, :125] = (2 * phi - 1).bfloat16()
    return X, (sign / R).float()


def _ellipsoids(c, seed):
    """Shape parameters of training stencils: spheres and ellipsoids, radii log-uniform in [2, 60]."""
    r, n = np.random.RandomState(seed % (1 << 31)), c["n"]
    R = np.exp(np.log(2.0) + r.rand(n) * np.log(30.0))
    ell = r.rand(n) >= 0.5
    axes = np.stack([R, R * np.where(ell, 0.6 + 0.4 * r.rand(n), 1.0), R * np.where(ell, 0.6 + 0.4 * r.rand(n), 1.0)], 1)
    quat, d = r.randn(n, 4), r.randn(n, 3)
    f = lambda v: np.asarray(v, np.float32)  # noqa: E731
    return dict(axes=f(np.maximum(axes, 2.0)), quat=f(quat / np.linalg.norm(quat, axis=1, keepdims=True)),
                dir=f(d / np.linalg.norm(d, axis=1, keepdims=True)), delta=f(r.rand(n, 3) - 0.5),
                invert=(r.rand(n) < 0.3).astype(np.int32))


# ---- what the program holds, and the call -----------------------------------------
def _params(c, curv, **kw):
    return F.make_params(_grid(c), collision=F.TRT if c.get("trt") else F.BGK, curv_model=curv,
                         storage=STORE[c.get("storage", "f32")], storage_shift=SHIFT, tau=c.get("tau", 0.6),
                         sigma=c.get("sigma", 1e-3), theta=math.radians(c.get("theta", 90.0)), **kw)


def prepare(case, seed):
    c = case
    if c["kind"] in ("steps", "curvature", "window"):
        g = _geometry(c if c["kind"] != "window" else dict(c, setup="cap"), seed)
        phi, obs = _fill(c, g).float(), _walls(c)
        if obs is not None:
            phi[obs > 0] = 0
    if c["kind"] == "steps":
        sim = F.Sim(_params(c, CURV[c["curv"]]), phi0=phi, obstacle=obs)
        sim.f_current().copy_(_initial_pdfs(c, g, seed, sim.flags_current() & 15))
        if c["setup"] == "bubble":
            sim.set_bubble(1.0 / 3.0)
        if c["curv"] == "mlp":
            sim.attach_mlp(F.Mlp(_network()), 0.05)
        return dict(c=c, sim=sim)
    if c["kind"] == "curvature":
        sim = F.Sim(_params(c, F.CURV_LSQR), phi0=phi)
        return dict(c=c, sim=sim, out=[torch.zeros_like(sim.kappa) for _ in range(3)])
    if c["kind"] == "train":
        net = F.Mlp(_midway())
        r = torch.Generator(device=DEV).manual_seed(seed)
        m, v = _moments(r)
        net.m.copy_(m)
        net.v.copy_(v)
        net.step = 1000
        X, t = _sphere_stencils(seed, c["rows"])
        Xh, th = _sphere_stencils(seed + 1, c["held"])
        perm = torch.randperm(c["rows"], generator=r, device=DEV)
        return dict(c=c, net=net, X=X, t=t, Xh=Xh, perm=perm, losses=torch.zeros(c["rows"] // c["batch"], device=DEV))
    if c["kind"] == "stencils":
        return dict(c=c, p=_ellipsoids(c, seed), seed=seed)
    if c["kind"] == "window":
        sim = F.Sim(_params(dict(c, trt=True, tau=0.8, sigma=2e-4), F.CURV_LSQR), phi0=phi, obstacle=obs)
        start = sim.snapshot()
        ifc = (sim.flags_current() & 15) == IF
        r = torch.Generator(device=DEV).manual_seed(seed)
        target = phi + 1e-2 * torch.randn(phi.shape, generator=r, device=DEV)
        return dict(c=c, sim=sim, start=start, target=target, ifc=ifc)
    g = dict(_geometry(c, seed))
    g["R"] = g.get("R", 0.0)
    obs = torch.zeros(_grid(c), dtype=torch.uint8, device=DEV)
    if c["shape"] in ("cap", "pool"):
        obs[0] = obs[-1] = 1
    return dict(c=c, params=_params(c, F.CURV_LSQR), geom=F.make_geometry(g.pop("kind"), sub=16, **g),
                obs=obs if c["shape"] in ("cap", "pool") else None)


def _state_of(sim):
    return dict(f=sim.f_current(), flags=sim.flags_current(), mass=sim.mass, phi=sim.phi, kappa=sim.kappa)


def run(state):
    c = state["c"]
    if c["kind"] == "steps":
        state["sim"].step(c["steps"])
        return _state_of(state["sim"])
    if c["kind"] == "curvature":
        return [state["sim"].curvature(m, o) for m, o in zip((F.CURV_LSQR, F.CURV_FD, F.CURV_TR), state["out"])]
    if c["kind"] == "train":
        net = state["net"]
        net.train_epoch(state["X"], state["t"], state["perm"], c["batch"], LR, state["losses"])
        return dict(master=net.master, m=net.m, v=net.v, losses=state["losses"], held=net.forward(state["Xh"]))
    if c["kind"] == "stencils":
        X, t = F.mlp_stencils(state["p"], sub=c["sub"], noise=1e-3, noise_seed=state["seed"])
        return dict(X=X, target=t)
    if c["kind"] == "window":
        sim = state["sim"]
        sim.restore(state["start"])
        sim.set_surface(2e-4, math.radians(80.0))
        sim.window_forward(c["window"], c["every"])
        end = sim.phi.clone()
        g = 2.0 * torch.where(state["ifc"], end - state["target"], torch.zeros_like(end))
        ds, dt, dphi, dmass, df = sim.window_adjoint(g, inputs=True)
        return dict(phi=end, surface=torch.tensor([ds, dt], dtype=torch.float32), dphi=dphi, dmass=dmass, df=df)
    phi = torch.zeros(_grid(c), dtype=torch.float32, device=DEV)
    F.fill_geometry(state["params"], state["geom"], phi)
    if state["obs"] is not None:
        phi[state["obs"] > 0] = 0
    sim = F.Sim(state["params"], phi0=phi, obstacle=state["obs"])
    return dict(_state_of(sim), total=sim.mass_total()[0])


# ---- what a pass cannot do without --------------------------------------------------
def work(case):
    c = case
    pdf = 4 if c.get("storage", "f32") == "f32" else 2
    if c["kind"] == "train":
        n = c["rows"] // c["batch"] * c["batch"]
        return dict(bytes=n * 264.0 + c["held"] * 260.0 + 33153 * 26.0, flops=n * 197e3 + c["held"] * 66e3)
    if c["kind"] == "stencils":  # the cells a surface can cut, about 45 of 125, are sampled
        return dict(bytes=c["n"] * (56 + 260.0), flops=c["n"] * 45.0 * c["sub"] ** 3 * 6)
    cells = c["nx"] * c["ny"] * c["nz"]
    setup = c.get("setup") or c.get("shape") or c["kind"]
    R = c["R"]
    if setup == "pool":
        liquid, surface = 0.625 * cells, 1.6 * c["nx"] * c["ny"]
    else:
        liquid, surface = 4.19 * R ** 3, 18.0 * R ** 2
        if setup in ("cap", "window"):
            liquid, surface = liquid / 2, surface / 2
        if setup == "pair":
            liquid, surface = liquid * 1.3, surface * 1.44
        if setup == "bubble":
            liquid = cells - liquid
    if c["kind"] == "curvature":
        return dict(bytes=surface * 3 * (4 + 20.0), flops=surface * 5000.0)
    if c["kind"] == "setup":
        return dict(bytes=cells * (2 * 19 * pdf + 2 + 12.0) + liquid * 19 * pdf, flops=surface * 4096 * 10.0)
    step = dict(bytes=liquid * (38 * pdf + 1) + surface * (38 * pdf + 40), flops=liquid * 250.0 + surface * 1500.0)
    if c.get("curv") == "mlp":
        step["flops"] += surface * 65e3
    # a window: the forward steps, the recomputed steps, and the reverse (the state and its adjoint)
    times = c["steps"] if c["kind"] == "steps" else 4 * c["window"]
    return dict(bytes=step["bytes"] * times, flops=step["flops"] * times)


# ---- the method in 64 bits, on lists of cells -----------------------------------------
class _Exact:
    def __init__(self, c, phi, obs, tau, sigma, trt):
        self.n = (c["nx"], c["ny"], c["nz"])
        self.t = _initial_types(phi, obs).view(-1)
        self.phi = torch.where(self.t.view(phi.shape) == LIQ, 1.0, torch.where(self.t.view(phi.shape) == IF, phi, 0.0)).view(-1)
        self.m = self.phi.clone()
        self.kappa = torch.zeros_like(self.phi)
        self.we = 1 / tau
        self.wo = 1 / (0.5 + 3 / 16 / (tau - 0.5)) if trt else self.we
        self.sigma, self.p0 = sigma, None

    def at(self, i, dx, dy, dz):
        """Index of the cells at an offset from the cells i (periodic)."""
        nx, ny, nz = self.n
        x, y, z = i % nx, i // nx % ny, i // (nx * ny)
        return (x + dx) % nx + nx * ((y + dy) % ny + ny * ((z + dz) % nz))

    def set_pdfs(self, f, store):
        self.store = store
        f = f.view(19, -1).double()
        self.f = f if store == "f32" else f / 2.0 ** SHIFT + torch.tensor(W, device=DEV, dtype=torch.float64).view(19, 1)
        self.old = torch.tensor(W, device=DEV, dtype=torch.float64).view(19, 1).repeat(1, f.shape[1])

    def stored(self):
        if self.store == "f32":
            return self.f
        return (self.f - torch.tensor(W, device=DEV, dtype=torch.float64).view(19, 1)) * 2.0 ** SHIFT

    def gas_volume(self):
        return float((self.t != OBS).sum() - (self.t == LIQ).sum()) - float(self.phi[self.t == IF].sum())

    def unit(self, field, i):
        """Unit Parker-Youngs gradient of a field at the cells i, and where it is not zero."""
        n = torch.zeros(3, i.numel(), dtype=torch.float64, device=DEV)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    v = field[self.at(i, dx, dy, dz)]
                    w = [2 if a == 0 else 1 for a in (dx, dy, dz)]
                    n[0] += dx * w[1] * w[2] * v
                    n[1] += dy * w[0] * w[2] * v
                    n[2] += dz * w[0] * w[1] * v
        ln = n.norm(dim=0)
        ok = ln >= 1e-12
        return torch.where(ok, n / ln.clamp(min=1e-300), 0.0), ok

    # interface normals (towards the liquid) and PLIC offsets of the cells i
    def normals(self, i):
        n, ok = self.unit(self.phi, i)
        s = n.abs().sum(0)
        m = (n.abs() / s.clamp(min=1e-300)).sort(dim=0).values
        phi = self.phi[i]
        lo, hi = torch.zeros_like(phi), torch.ones_like(phi)
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            less = self._volume(m, mid) < phi
            lo, hi = torch.where(less, mid, lo), torch.where(less, hi, mid)
        a = s * (0.5 - 0.5 * (lo + hi))
        a = torch.where(phi <= 0, 0.5 * s, torch.where(phi >= 1, -0.5 * s, a))
        return n, torch.where(ok, a, 0.0), ok

    @staticmethod
    def _volume(m, al):
        """Volume of {z in the unit cube: m.z <= al}, 0 <= m1 <= m2 <= m3, sum 1; by dimension where components vanish."""
        p = lambda v, k: v.clamp(min=0) ** k  # noqa: E731
        m1, m2, m3 = m.clamp(min=1e-5)
        v3 = p(al, 3) + sum(p(al - x - y, 3) for x, y in ((m1, m2), (m1, m3), (m2, m3))) - sum(p(al - x, 3) for x in (m1, m2, m3))
        v3 = (v3 - p(al - m1 - m2 - m3, 3)) / (6 * m1 * m2 * m3)
        b = al - 0.5 * m[0]
        v2 = (p(b, 2) - p(b - m2, 2) - p(b - m3, 2) + p(b - m2 - m3, 2)) / (2 * m2 * m3)
        v1 = (al - 0.5 * (m[0] + m[1])) / m3
        return torch.where(m[0] >= 1e-5, v3, torch.where(m[1] >= 1e-5, v2, v1)).clamp(0, 1)

    def lsqr(self, i):
        """Curvature of the least-squares paraboloid through the PLIC points of the 3x3x3 block."""
        n, a, ok = self.normals(i)
        pos = torch.full((self.t.numel(),), -1, dtype=torch.int64, device=DEV)
        pos[i] = torch.arange(i.numel(), device=DEV)
        k = torch.argmin(n.abs(), dim=0)
        e = torch.nn.functional.one_hot(k, 3).T.double()
        tu = torch.linalg.cross(e, n, dim=0)
        tu = tu / tu.norm(dim=0).clamp(min=1e-300)
        tv = torch.linalg.cross(n, tu, dim=0)
        rows, rhs, used = [], [], torch.zeros_like(k)
        for t in range(27):
            if t == 13:
                continue
            o = torch.tensor([t % 3 - 1, t // 3 % 3 - 1, t // 9 - 1], device=DEV, dtype=torch.float64).view(3, 1)
            j = pos[self.at(i, *(int(v) for v in o.view(-1)))]
            use = (j >= 0) & ok[j.clamp(min=0)]
            j = j.clamp(min=0)
            d = o + a[j] * n[:, j] - a * n
            u, v, h = (d * tu).sum(0), (d * tv).sum(0), (d * n).sum(0)
            rows.append(torch.stack([u * u, v * v, u * v, u, v]) * use)
            rhs.append(h * use)
            used += use
        A, b = torch.stack(rows).permute(2, 0, 1), torch.stack(rhs).T.unsqueeze(2)
        full, sound = self._fit(A, b)
        iso, sound3 = self._fit(torch.stack([A[..., 0] + A[..., 1], A[..., 3], A[..., 4]], 2), b)
        z = torch.zeros_like(iso[:, 0])
        sol = torch.where((sound & (used >= 5)).unsqueeze(1), full, torch.stack([iso[:, 0], iso[:, 0], z, iso[:, 1], iso[:, 2]], 1))
        fine = ok & ((sound & (used >= 5)) | (sound3 & (used >= 3)))
        A_, B_, C_, H, I = sol.unbind(1)
        g = 1 + H * H + I * I
        return torch.where(fine, (A_ * (1 + I * I) + B_ * (1 + H * H) - C_ * H * I) / g ** 1.5, 0.0)

    @staticmethod
    def _fit(A, b):
        G = A.mT @ A
        L, bad = torch.linalg.cholesky_ex(G)
        dg = torch.diagonal(L, dim1=1, dim2=2).abs()
        sound = (bad == 0) & (dg.amin(1) > 1e-6 * dg.amax(1))
        G = torch.where(sound.view(-1, 1, 1), G, torch.eye(G.shape[1], dtype=G.dtype, device=DEV))
        L = torch.linalg.cholesky_ex(G)[0]
        x = torch.cholesky_solve(A.mT @ b, L)
        x = x + torch.cholesky_solve(A.mT @ (b - A @ x), L)  # refined once
        return x.squeeze(2), sound

    def fd(self, i):
        """-1/2 div of the unit normals of the K8-smoothed fill level, central differences."""
        nz, ny, nx = self.n[2], self.n[1], self.n[0]
        phi = torch.where(self.t == OBS, 0.0, self.phi).view(nz, ny, nx)
        k8 = {0: 1.0, 1: 0.31640625, 2: 0.0625, 3: 0.00390625}
        sm = torch.zeros_like(phi)
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    sm += k8[dx * dx + dy * dy + dz * dz] * torch.roll(phi, (dz, dy, dx), (0, 1, 2))
        sm = (sm / 3.6796875).view(-1)
        div = torch.zeros(i.numel(), dtype=torch.float64, device=DEV)
        for ax in range(3):
            for sg in (1, -1):
                o = [sg if k == ax else 0 for k in range(3)]
                div += sg * self.unit(sm, self.at(i, *o))[0][ax]
        return -0.25 * div

    def mlp(self, i, kls, net):
        """The network's value where it lies within 5 % of the least-squares one."""
        p = [torch.arange(125, device=DEV) // w % 5 - 2 for w in (25, 5, 1)]
        nx, ny, nz = self.n
        x, y, z = ((v.view(-1, 1) + o.view(1, -1)) % m for v, o, m in
                   ((i % nx, p[0], nx), (i // nx % ny, p[1], ny), (i // (nx * ny), p[2], nz)))
        s = self.phi[x + nx * (y + ny * z)]
        c = s.view(-1, 5, 5, 5)[:, 1:4, 1:4, 1:4]
        w = torch.tensor([1.0, 2.0, 1.0], dtype=torch.float64, device=DEV)
        g = torch.tensor([-1.0, 0.0, 1.0], dtype=torch.float64, device=DEV)
        n = torch.stack([torch.einsum("nabc,a,b,c->n", c, *v) for v in ((g, w, w), (w, g, w), (w, w, g))], 1)
        order = torch.argsort(-n.abs(), dim=1, stable=True)
        wt = torch.zeros_like(order).scatter_(1, order, torch.tensor([25, 5, 1], device=DEV).expand_as(order))
        to = torch.zeros_like(s, dtype=torch.int64)
        for k in range(3):
            r = (p[k] + 2).view(1, -1)
            to += torch.where(n[:, k: k + 1] < 0, 4 - r, r) * wt[:, k: k + 1]
        X = torch.zeros(s.shape[0], 128, dtype=torch.float64, device=DEV)
        X.scatter_(1, to, (2 * s - 1).bfloat16().double())
        k = _forward(net, X)
        return torch.where((k - kls).abs() <= 0.05 * kls.abs(), k, kls)

    def step(self, curv, net):
        i = (self.t == IF).nonzero().view(-1)
        kap = self.fd(i) if curv == "fd" else self.lsqr(i)
        if curv == "mlp":
            kap = self.mlp(i, kap, net)
        self.kappa[i] = kap
        pg = 1 / 3 if self.p0 is None else self.p0[0] * self.p0[1] / self.gas_volume()
        f, new = self.f, self.old
        # liquid cells
        for part in (self.t == LIQ).nonzero().view(-1).split(1 << 21):
            v = []
            for q in range(19):
                s = self.at(part, -CX[q], -CY[q], -CZ[q])
                v.append(torch.where(self.t[s] == OBS, f[OPP[q], part], f[q, s]))
            self._collide(v)
            for q in range(19):
                new[q, part] = v[q]
        # interface cells
        own = f[:, i]
        r0 = own.sum(0)
        u = [sum(cc[q] * own[q] for q in range(19)) / r0 for cc in (CX, CY, CZ)]
        rho_b = 3 * pg + 6 * self.sigma * kap
        v, dm = [own[0]], torch.zeros_like(r0)
        for q in range(1, 19):
            s = self.at(i, -CX[q], -CY[q], -CZ[q])
            ts, fin = self.t[s], f[q, s]
            fluid = (ts == LIQ) | (ts == IF)
            rec = _feq(q, rho_b, u) + _feq(OPP[q], rho_b, u) - own[OPP[q]]
            v.append(torch.where(fluid, fin, torch.where(ts == OBS, own[OPP[q]], rec)))
            kq = torch.where(ts == LIQ, 1.0, 0.5 * (self.phi[i] + self.phi[s]))
            dm += torch.where(fluid, kq * (fin - own[OPP[q]]), 0.0)
        rho = self._collide(v)
        for q in range(19):
            new[q, i] = v[q]
        self.m[i] += dm
        self._convert(i, rho, new)
        self.f, self.old = new, f

    def _collide(self, v):
        rho = sum(v)
        u = [sum(cc[q] * v[q] for q in range(19)) / rho for cc in (CX, CY, CZ)]
        fe = [_feq(q, rho, u) for q in range(19)]
        v[0] = v[0] - self.we * (v[0] - fe[0])
        for q in range(1, 19, 2):
            p, m = 0.5 * (v[q] + v[q + 1]), 0.5 * (v[q] - v[q + 1])
            ep, em = 0.5 * (fe[q] + fe[q + 1]), 0.5 * (fe[q] - fe[q + 1])
            a, b = self.we * (p - ep), self.wo * (m - em)
            v[q], v[q + 1] = v[q] - a - b, v[q + 1] - a + b
        return rho

    def _around(self, i):
        return torch.stack([self.at(i, CX[q], CY[q], CZ[q]) for q in range(1, 19)])

    def _convert(self, i, rho, new):
        t, m = self.t, self.m
        full = torch.zeros(t.numel(), dtype=torch.float64, device=DEV)
        full[i] = rho
        rho = full
        fill = i[m[i] > 1.001 * rho[i]]
        empty = i[m[i] < -0.001 * rho[i]]
        filling = torch.zeros_like(t, dtype=torch.bool)
        filling[fill] = True
        empty = empty[~filling[self._around(empty)].any(0)] if empty.numel() else empty
        leaving = filling.clone()
        leaving[empty] = True
        born = torch.zeros_like(filling)
        a, b = self._around(fill).reshape(-1), self._around(empty).reshape(-1)
        gas, liq = a[t[a] == GAS].unique(), b[t[b] == LIQ].unique()
        born[gas] = born[liq] = True
        if gas.numel():
            s = self._around(gas)
            fluid = (t[s] == LIQ) | (t[s] == IF)
            r = sum(new[q][s] for q in range(19))
            u = [torch.where(fluid, sum(cc[q] * new[q][s] for q in range(19)) / r, 0.0).sum(0) / fluid.sum(0) for cc in (CX, CY, CZ)]
            rb = torch.where(fluid, r, 0.0).sum(0) / fluid.sum(0)
            for q in range(19):
                new[q, gas] = _feq(q, rb, u)
            m[gas], rho[gas] = 0.0, rb
        m[liq] = rho[liq] = new[:, liq].sum(0)
        takes = ((t == IF) & ~leaving) | born
        share = torch.zeros_like(rho)
        for cells, ex in ((fill, m[fill] - rho[fill]), (empty, m[empty])):
            cnt = takes[self._around(cells)].sum(0)
            share[cells] = torch.where(cnt > 0, ex / cnt.clamp(min=1), 0.0)
        m[fill], m[empty] = rho[fill], 0.0
        stay = torch.cat([i[~leaving[i]], gas, liq])
        m[stay] += torch.where(leaving[self._around(stay)], share[self._around(stay)], 0.0).sum(0)
        self.phi[stay] = m[stay] / rho[stay]
        t[stay], t[fill], t[empty] = IF, LIQ, GAS
        self.phi[fill], self.phi[empty] = 1.0, 0.0


def _forward(net, X):
    gelu = torch.nn.functional.gelu
    b = lambda v: torch.as_tensor(v).bfloat16().double().to(DEV)  # noqa: E731
    d = lambda v: torch.as_tensor(v).double().to(DEV)  # noqa: E731
    h = gelu(X @ b(net["W1"]).T + d(net["b1"]))
    return gelu(h @ b(net["W2"]).T + d(net["b2"])) @ b(net["w3"]) + d(net["b3"])


def exact(case, seed):
    c = case
    if c["kind"] == "steps":
        if c["setup"] == "cap" or c["curv"] == "tr":
            return None  # contact-line fits and the triangle fan have no short plain form
        g = _geometry(c, seed)
        phi, obs = _fill(c, g).float().double(), _walls(c)
        if obs is not None:
            phi[obs > 0] = 0
        e = _Exact(c, phi, obs, c["tau"], c["sigma"], c["trt"])
        e.set_pdfs(_initial_pdfs(c, g, seed, e.t.view(_grid(c))), c["storage"])
        if c["setup"] == "bubble":
            e.p0 = (1 / 3, e.gas_volume())
        for _ in range(c["steps"]):
            e.step(c["curv"], _network() if c["curv"] == "mlp" else None)
        s = _grid(c)
        return dict(f=e.stored().view((19,) + s), flags=None, mass=e.m.view(s), phi=e.phi.view(s), kappa=e.kappa.view(s))
    if c["kind"] == "curvature":
        e = _Exact(c, _fill(c, _geometry(c, seed)).float().double(), None, 1.0, 0.0, False)
        i = (e.t == IF).nonzero().view(-1)
        out = []
        for k in (e.lsqr(i), e.fd(i)):
            full = torch.zeros_like(e.phi)
            full[i] = k
            out.append(full.view(_grid(c)))
        return out + [None]
    if c["kind"] == "train":
        return _exact_train(c, seed)
    if c["kind"] == "stencils":
        return dict(X=None, target=_exact_targets(_ellipsoids(c, seed)))
    if c["kind"] == "setup":
        phi = _fill(c, _geometry(c, seed)).float().double()
        obs = None
        if c["shape"] in ("cap", "pool"):
            obs = torch.zeros(_grid(c), dtype=torch.uint8, device=DEV)
            obs[0] = obs[-1] = 1
            phi[obs > 0] = 0
        e = _Exact(c, phi, obs, 1.0, 0.0, False)
        s = _grid(c)
        w = torch.tensor(W, dtype=torch.float64, device=DEV) if c["storage"] == "f32" else torch.zeros(19, dtype=torch.float64, device=DEV)
        mass = e.m.clone()
        return dict(f=w.view(19, 1, 1, 1).expand((19,) + s), flags=None, mass=mass.view(s), phi=e.phi.view(s),
                    kappa=e.kappa.view(s), total=float(mass.sum()))
    return None  # the reverse of the wall-bounded window has no short plain form


def _exact_train(c, seed):
    """The epoch in 64 bits: BF16 weights in the passes, FP64 elsewhere, Adam on the masters."""
    net = _midway()
    keys = ("W1", "W2", "w3", "b1", "b2", "b3")
    w = torch.cat([torch.as_tensor(net[k]).double().reshape(-1) for k in keys]).to(DEV)
    r = torch.Generator(device=DEV).manual_seed(seed)
    m, v = (x.double() for x in _moments(r))
    X, t = _sphere_stencils(seed, c["rows"])
    Xh, _ = _sphere_stencils(seed + 1, c["held"])
    perm = torch.randperm(c["rows"], generator=r, device=DEV)
    gelu, losses = torch.nn.functional.gelu, []

    def forward(p, x):
        W1, W2, w3, b1, b2, b3 = torch.split(p, [16384, 16384, 128, 128, 128, 1])
        return gelu(gelu(x @ W1.view(128, 128).T + b1) @ W2.view(128, 128).T + b2) @ w3 + b3

    def used(p):
        return torch.cat([p[:32896].float().bfloat16().double(), p[32896:]])

    B = c["batch"]
    for b in range(c["rows"] // B):
        rows = perm[b * B: (b + 1) * B]
        p = used(w).requires_grad_()
        tt = t[rows].double()
        loss = ((forward(p, X[rows].double()) - tt) ** 2 / (tt * tt + 7e-5)).mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(loss.detach())
        k = 1000 + b + 1
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - LR * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return dict(master=w, m=m, v=v, losses=torch.stack(losses), held=forward(used(w), Xh.double()))


def _exact_targets(p):
    """Mean curvature of each ellipsoid at the surface point nearest the stencil's centre."""
    a, q, d, o = (torch.as_tensor(p[k]).double().to(DEV) for k in ("axes", "quat", "dir", "delta"))
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    s = d / (d / a).norm(dim=1, keepdim=True)  # the surface point in the body frame
    cen = o - (R @ s.unsqueeze(2)).squeeze(2)
    b = -(R.mT @ cen.unsqueeze(2)).squeeze(2)
    a2 = a * a
    lo, hi = -a2.amin(1), (b.abs() * a).norm(dim=1) + 1
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        out = ((a * b / (a2 + mid.unsqueeze(1))) ** 2).sum(1) > 1
        lo, hi = torch.where(out, mid, lo), torch.where(out, hi, mid)
    x = a2 * b / (a2 + (0.5 * (lo + hi)).unsqueeze(1))
    gr, hs = 2 * x / a2, 2 / a2
    g2 = (gr * gr).sum(1)
    H = (g2 * hs.sum(1) - (gr * gr * hs).sum(1)) / (2 * g2 ** 1.5)
    return torch.where(torch.as_tensor(p["invert"]).to(DEV) > 0, -H, H)
