"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (a
simulation at its first level, a batch, a denoiser with its currents), `run` makes one pass
through the public binding and returns what the pass computed, `work` counts the bytes and
operations a pass cannot do without, and `exact` restates a pass in plain FP64.

Kinds:
  march     Sim.step(steps), then the spectral state and the energies
  streamed  Sim.step_streamed(steps): the state goes through pinned host memory every s-step
  scan      Batch.step(steps): a parameter scan of independent 2-D runs
  chain     Sim.step(steps) with the learned current denoiser in the loop
  apply     Denoiser.apply on one current
  train     Denoiser.train_step (forward, backward, Adam) on one slab
"""
import math

import numpy as np
import torch

from paper_2509_16793_gb300 import gempic
from paper_2509_16793_gb300 import workloads as W


def listed():
    return [
        # one s-step of a small 3-D grid: the latency of a single call (parity-sized runs,
        # interactive use)
        dict(name="small3d_16x16x48_1step", kind="march", family="small3d", nx=16, ny=16, nz=48,
             ppc=2, precision=32, a0=1.5, steps=1, option=""),
        # FP64 verification of a 3-D run with a plasma channel and a refined zeta-step
        dict(name="small3d_32x32x96_fp64", kind="march", family="small3d", nx=32, ny=32, nz=96,
             ppc=2, precision=64, a0=1.5, steps=2, option="channel+refined"),
        # the 2-D slab workload in FP64 at its stability limit, many s-steps per call
        dict(name="lwfa2d_128x256_fp64", kind="march", family="lwfa2d", nx=128, ny=1, nz=256,
             ppc=4, precision=64, a0=1.0, steps=40, option=""),
        # a wide 2-D slab in FP32 with an odd number of slices
        dict(name="lwfa2d_512x1001_fp32", kind="march", family="lwfa2d", nx=512, ny=1, nz=1001,
             ppc=4, precision=32, a0=1.0, steps=32, option=""),
        # a 3-D laser looked at after every s-step, on a short window
        dict(name="lwfa3d_128x128x300_1step", kind="march", family="lwfa3d", nx=128, ny=128,
             nz=300, ppc=2, precision=32, a0=2.5, steps=1, option=""),
        # the flagship 3-D grid, several s-steps per call
        dict(name="lwfa3d_128x128x1024", kind="march", family="lwfa3d", nx=128, ny=128, nz=1024,
             ppc=2, precision=32, a0=1.5, steps=14, option=""),
        # beam-driven wake: a sampled bunch, electrons and mobile protons
        dict(name="pwfa3d_128x128x768", kind="march", family="pwfa3d", nx=128, ny=128, nz=768,
             ppc=2, precision=32, a0=0.0, steps=7, option=""),
        # the flagship grid with its state streamed through host memory
        dict(name="lwfa3d_streamed_1024", kind="streamed", family="lwfa3d", nx=128, ny=128,
             nz=1024, ppc=2, precision=32, a0=1.5, steps=14, option=""),
        # a parameter scan of uneven 2-D runs
        dict(name="scan_24_runs", kind="scan", runs=24, precision=32, steps=8),
        # a sparse 3-D run with the denoiser in the loop
        dict(name="denoised_128x128x512", kind="chain", family="lwfa3d", nx=128, ny=128, nz=512,
             ppc=1, precision=32, a0=1.5, steps=7, option=""),
        # the denoiser on a whole window's current
        dict(name="denoise_apply_128x128x512", kind="apply", nx=128, ny=128, nz=512),
        # one training step on a slab of half-slices
        dict(name="denoise_train_128x128x32", kind="train", nx=128, ny=128, nz=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small3d", "lwfa2d", "lwfa2d", "lwfa3d", "lwfa3d", "pwfa3d", "streamed",
                       "scan", "chain", "apply", "apply", "train"])
    if kind == "small3d":
        return dict(kind="march", family="small3d", nx=rng.choice([16, 32, 64]),
                    ny=rng.choice([16, 32, 64]), nz=_log(rng, 24, 160), ppc=rng.choice([1, 2, 3]),
                    precision=rng.choice([32, 64]), a0=round(rng.uniform(0.5, 1.5), 3),
                    steps=rng.choice([1, 2, 3]),
                    option=rng.choice(["", "channel", "refined", "channel+refined"]))
    if kind == "lwfa2d":
        fp64 = rng.random() < 0.5
        return dict(kind="march", family="lwfa2d",
                    nx=rng.choice([64, 128] if fp64 else [64, 128, 256, 512]), ny=1,
                    nz=_log(rng, 80, 256) if fp64 else _log(rng, 100, 1001),
                    ppc=rng.choice([2, 3, 4]), precision=64 if fp64 else 32,
                    a0=round(rng.uniform(0.5, 1.0), 3), steps=_log(rng, 1, 32),
                    option=rng.choice(["", "", "channel", "refined"]))
    if kind == "lwfa3d":
        return dict(kind="march", family="lwfa3d", nx=128, ny=128, nz=_log(rng, 100, 1024),
                    ppc=rng.choice([1, 2]), precision=32, a0=round(rng.uniform(0.6, 1.5), 3),
                    steps=_log(rng, 1, 14), option=rng.choice(["", "", "channel"]))
    if kind == "pwfa3d":
        return dict(kind="march", family="pwfa3d", nx=128, ny=128, nz=_log(rng, 400, 768), ppc=2,
                    precision=32, a0=0.0, steps=rng.randint(1, 7), option="")
    if kind == "streamed":
        return dict(kind="streamed", family="lwfa3d", nx=128, ny=128, nz=_log(rng, 150, 800),
                    ppc=rng.choice([1, 2]), precision=32, a0=round(rng.uniform(0.6, 1.5), 3),
                    steps=rng.randint(2, 14), option="")
    if kind == "scan":
        return dict(kind="scan", runs=rng.randint(4, 24), precision=32, steps=rng.randint(2, 8))
    if kind == "chain":
        return dict(kind="chain", family="lwfa3d", nx=128, ny=128, nz=_log(rng, 100, 512), ppc=1,
                    precision=32, a0=round(rng.uniform(0.6, 1.5), 3), steps=rng.randint(1, 7),
                    option="")
    # nets: the bench's rows of 128 voxels and other widths, odd volumes
    nx = rng.choice([128, 128, 16, 32, 64, 96])
    ny = rng.randint(1, 128)
    if kind == "apply":
        return dict(kind="apply", nx=nx, ny=ny, nz=_log(rng, 8, 512))
    return dict(kind="train", nx=nx, ny=ny, nz=_log(rng, 9, 32))


# ---- inputs ---------------------------------------------------------------------------------


def _workload(case, seed):
    nx, ny, nz, ppc, prec = case["nx"], case["ny"], case["nz"], case["ppc"], case["precision"]
    if case["family"] == "small3d":
        w = W.small_3d(nx=nx, ny=ny, nzeta=nz, ppc=ppc, precision=prec, a0=case["a0"])
    elif case["family"] == "lwfa2d":
        w = W.lwfa_2d_128x256(precision=prec)
        if prec == 32:                            # the limit itself amplifies FP32 rounding
            w = w.with_(delta=0.25 * w.delta)
        w = w.with_(nx=nx, nzeta=nz, species=[W.Species(-1.0, 1.0, w.species[0].density, ppc)],
                    laser=W.Laser(**{**w.laser.__dict__, "a0": case["a0"],
                                     "zeta_center": 0.6 * nz * w.h}))
    elif case["family"] == "pwfa3d":
        w = W.pwfa_3d_128x128x768(precision=prec)
        # a bunch of a fifth of the plasma density: a wake that does not break
        w = w.with_(nzeta=nz, beam=W.Beam(**{**w.beam.__dict__, "n_peak": 0.2, "seed": seed + 3,
                                             "zeta_center": nz * w.h - 3.0}))
    else:
        w = W.lwfa_3d_128x128x1024(precision=prec)
        w = w.with_(nzeta=nz, species=[W.Species(-1.0, 1.0, w.species[0].density, ppc)],
                    laser=W.Laser(**{**w.laser.__dict__, "a0": case["a0"],
                                     "zeta_center": nz * w.h - 2.0 * w.laser.duration}))
    if "channel" in case["option"]:
        w = w.with_(channel=W.Channel(n1_over_n0=0.25, radius=0.3 * nx * w.hx))
    if "refined" in case["option"]:
        w = w.with_(hz=W.refined_h(nz, w.h, 2.0))
    return w.with_(seed=seed)


def _scan(case, seed):
    """The runs of a scan: the recipe's grids and densities, drivers that do not break the wake,
    a quarter of the stability limit."""
    return [w.with_(seed=seed + i, delta=0.25 * w.delta,
                    laser=W.Laser(**{**w.laser.__dict__, "a0": 0.3 + 0.4 * w.laser.a0}))
            for i, w in enumerate(W.scan_2d(n=case["runs"], precision=case["precision"]))]


def _params(seed, last=0.2):
    """Weights of the denoiser's net, He-normal with a small last layer (as after training)."""
    g = np.random.default_rng(seed)
    P = {}
    for l, (ci, co, s) in enumerate(((3, 16, 1.0), (16, 16, 1.0), (16, 3, last)), start=1):
        P[f"W{l}"] = g.standard_normal((3, 3, 3, ci, co)) * math.sqrt(2.0 / (27 * ci)) * s
        P[f"b{l}"] = g.standard_normal(co) * 0.05
    return gempic.denoiser_params_to_vector(P)


NET_SCALE = 0.002        # |q n0| of the 3-D workloads


def _currents(case, seed):
    """(noisy, clean) currents [nz, 3, ny, nx]: a few smooth waves, and shot noise on top."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.arange(nz, device="cuda").view(-1, 1, 1, 1)
    y = torch.arange(ny, device="cuda").view(1, 1, -1, 1)
    x = torch.arange(nx, device="cuda").view(1, 1, 1, -1)
    c = torch.arange(3, device="cuda").view(1, -1, 1, 1)
    ph = torch.rand(3, generator=gen, device="cuda") * 6.28
    clean = NET_SCALE * (torch.cos(0.1 * z + ph[0] + c) * torch.cos(6.2831853 * x / nx + ph[1])
                         * torch.cos(6.2831853 * y / ny + ph[2]))
    noisy = clean + 0.5 * NET_SCALE * torch.randn((nz, 3, ny, nx), generator=gen, device="cuda")
    return noisy.contiguous(), clean.contiguous()


def _complex(w):
    return torch.complex128 if w.precision == 64 else torch.complex64


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("apply", "train"):
        s["den"] = gempic.Denoiser(_params(seed), NET_SCALE)
        s["j"], s["target"] = _currents(case, seed)
        s["out"] = torch.empty_like(s["j"])
        return s
    if kind == "scan":
        ws = _scan(case, seed)
        s["batch"] = gempic.Batch(ws)
        s["states"] = [torch.empty((6, w.nzeta, 1, w.nx // 2), dtype=_complex(w), device="cuda")
                       for w in ws]
        return s
    w = _workload(case, seed)
    s["sim"] = sim = gempic.Sim(w)
    if kind == "chain":
        s["den"] = gempic.Denoiser(_params(seed), NET_SCALE)
        sim.set_denoiser(s["den"])
    if kind == "streamed":
        s["host"] = torch.empty(sim.state_shape(), dtype=_complex(w), pin_memory=True)
        s["host_np"] = s["host"].numpy()
        sim.gempic_get_state(s["host_np"])
        return s
    sim.step(0)                                   # lays the laser and the first level
    s["state"] = torch.empty(sim.state_shape(), dtype=_complex(w), device="cuda")
    return s


def _energies(case, d):
    # (the flux of a neutral plasma is a sum of cancelling charges: rounding alone)
    keys = ("field_energy", "kinetic_energy", "charge_flux")
    return {k: float(d[k]) for k in (keys[:2] if case["family"] == "pwfa3d" else keys)}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        return s["den"].apply(s["j"], s["out"])
    if kind == "train":
        loss = s["den"].train_step(s["j"], s["target"], 1e-3, z_margin=3)
        return {"loss": loss, "params": s["den"].params()}
    if kind == "scan":
        b = s["batch"]
        b.step(case["steps"])
        return [v.state(t) for v, t in zip(b.sims, s["states"])]
    sim = s["sim"]
    if kind == "streamed":
        d = sim.step_streamed(case["steps"], s["host_np"])
        return {"state": s["host"], **_energies(case, d[-1])}
    sim.step(case["steps"])
    return {"state": sim.state(s["state"]), **_energies(case, sim.diagnostics())}


# ---- what a pass cannot do without ----------------------------------------------------------

PUSH_FLOP = 330          # gather 52, two-pass Boris 156, advance 22, Esirkepov and CIC 100
SOLVE_FLOP = 150         # closed form of one mode
NET_MACS = 27 * (3 * 16 + 16 * 16 + 16 * 3)


def _march_flops(nx, ny, nz, ppc):
    """One s-step: the pushes, the transverse transforms (two real rows as one complex one, nine
    columns of every kept kx) and the per-mode solves; 2-D has no column transforms and half
    the deposit."""
    fft = lambda n: 5.0 * n * math.log2(n) if n > 1 else 0.0
    rows = 5 * ny if ny > 1 else 5
    per_slice = rows * fft(nx) + 9 * (nx // 2) * fft(ny) + SOLVE_FLOP * (nx // 2) * ny
    push = PUSH_FLOP if ny > 1 else 230
    return nz * (per_slice + push * ppc * nx * ny)


def work(case):
    kind = case["kind"]
    if kind in ("apply", "train"):
        v = case["nx"] * case["ny"] * case["nz"]
        if kind == "apply":
            return {"bytes": 24 * v, "flops": 2 * NET_MACS * v}
        return {"bytes": 24 * v, "flops": 6 * NET_MACS * v}
    if kind == "scan":
        ws, n = _scan(case, 0), case["steps"]
        return {"bytes": n * sum(w.nx * w.nzeta * 48 for w in ws),
                "flops": n * sum(_march_flops(w.nx, 1, w.nzeta, 4) for w in ws)}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    eb = case["precision"] // 8
    ppc = case["ppc"] * (2 if case["family"] == "pwfa3d" else 1)
    per_step = nx * ny * nz * 6 * 2 * eb          # the state, read and written
    flops = _march_flops(nx, ny, nz, ppc)
    if kind == "chain":
        flops += _march_flops(nx, ny, nz, 0) + 2 * NET_MACS * nx * ny * nz
    if kind == "streamed":
        per_step *= 2                             # and through host memory
    return {"bytes": case["steps"] * per_step, "flops": case["steps"] * flops}


# ---- the same pass in plain FP64 ------------------------------------------------------------


def _splitmix(seed, c):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (c + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


class _Plain:
    """The slice scheme and the particles of one species of electrons under GT2, without stored
    particles: a run that would need them (one that traps before its last s-step) has no value."""

    def __init__(self, w):
        self.w, self.dev = w, "cuda"
        self.hz = torch.tensor(w.hz if w.hz is not None else np.full(w.nzeta, w.h)).tolist()
        f64 = dict(dtype=torch.float64, device=self.dev)
        kx = 2 * math.pi * torch.arange(w.nx // 2, **f64) / (w.nx * w.hx)
        ky = 2 * math.pi * torch.fft.fftfreq(w.ny, d=w.hy, **f64) if w.ny > 1 else torch.zeros(1, **f64)
        self.kx, self.ky = kx.view(1, -1), ky.view(-1, 1)
        self.keep = torch.ones((w.ny, w.nx // 2), **f64)
        if w.ny > 1:
            self.keep[w.ny // 2] = 0.0
        shape = (w.nzeta, w.ny, w.nx // 2)
        self.S = torch.zeros((6, *shape), dtype=torch.complex128, device=self.dev)
        self.x = torch.arange(w.nx, **f64) * w.hx - 0.5 * w.nx * w.hx
        self.y = torch.arange(w.ny, **f64) * w.hy - (0.5 * w.ny * w.hy if w.ny > 1 else 0.0)
        self.k = 0
        if w.laser is not None:
            L = w.laser
            zc = np.concatenate(([0.0], np.cumsum(self.hz)))
            tr = torch.exp(-(self.y.view(-1, 1) ** 2 + self.x.view(1, -1) ** 2) / L.waist ** 2)
            tr = self.spectrum(tr)
            for n in range(w.nzeta):
                ph = zc[n] - L.zeta_center
                self.S[L.pol, n] = 2.0 * L.a0 * math.cos(ph) * math.exp(-ph * ph / L.duration ** 2) * tr
        self.march(0.0, False)

    def spectrum(self, a):
        return torch.fft.rfft2(a)[..., :-1] * self.keep

    def real(self, a):
        return torch.fft.irfft2(torch.nn.functional.pad(a, (0, 1)), s=(self.w.ny, self.w.nx))

    def layer(self):
        w, sp = self.w, self.w.species[0]
        n = w.nx * w.ny * sp.ppc
        g = np.arange(n, dtype=np.uint64)
        c = (np.uint64(self.k * n) + g) * np.uint64(2)
        u = lambda i: torch.tensor((_splitmix(w.seed, c + np.uint64(i)) >> np.uint64(40))
                                   .astype(np.float64) / 16777216.0, device=self.dev)
        cell = torch.arange(n, device=self.dev) // sp.ppc
        X = cell % w.nx + u(0)
        Y = cell // w.nx + (u(1) if w.ny > 1 else torch.zeros_like(X))
        q = torch.full_like(X, sp.charge * sp.density / sp.ppc)      # Q / (hx hy Delta)
        if w.channel is not None:
            r2 = ((X - w.nx // 2) * w.hx) ** 2
            if w.ny > 1:
                r2 = r2 + ((Y - w.ny // 2) * w.hy) ** 2
            q = q * (1 + (w.channel.n1_over_n0 - 1) * torch.exp(-r2 / w.channel.radius ** 2))
        z = torch.zeros_like(X)
        return dict(X=X, Y=Y, ux=z, uy=z.clone(), uz=z.clone(), sig=z.clone(), q=q)

    def add(self, plane, X, Y, v):
        w = self.w
        plane.view(-1).index_add_(0, (Y.long() % w.ny) * w.nx + X.long() % w.nx, v)

    def push(self, p, E, h):
        """Push by one slab; the currents of the move and which particles used up their budget."""
        w, sp = self.w, self.w.species[0]
        D, qm = w.delta, sp.charge / sp.mass
        ix, iy = torch.floor(p["X"]), torch.floor(p["Y"])
        fx, fy = p["X"] - ix, p["Y"] - iy
        F = E.reshape(6, -1)
        at = lambda a, b: F[:, ((iy.long() + b) % w.ny) * w.nx + (ix.long() + a) % w.nx]
        if w.ny > 1:
            f = ((1 - fx) * (1 - fy) * at(0, 0) + fx * (1 - fy) * at(1, 0) + (1 - fx) * fy * at(0, 1)
                 + fx * fy * at(1, 1))
        else:
            f = (1 - fx) * at(0, 0) + fx * at(1, 0)
        u = torch.stack((p["ux"], p["uy"], p["uz"]))
        gam = lambda v: torch.sqrt(1 + (v * v).sum(0))
        gmu = lambda v, g: torch.where(v[2] > 0, (1 + v[0] ** 2 + v[1] ** 2) / (g + v[2]), g - v[2])

        def boris(dt):
            a = 0.5 * qm * dt
            um = u + a * f[:3]
            t = a / gam(um) * f[3:]
            up = um + torch.linalg.cross(um, t, dim=0)
            return um + torch.linalg.cross(up, 2 * t / (1 + (t * t).sum(0)), dim=0) + a * f[:3]

        g0 = gam(u)
        gm0 = gmu(u, g0)
        lim = torch.where(u[2] > 0, (D - p["sig"]) * gm0 / u[2].clamp_min(1e-300), math.inf).clamp_min(0)
        trap = lim < h
        hc = torch.where(trap, lim, torch.full_like(lim, h))
        ub = 0.5 * (u + boris(hc * g0 / gm0))
        gb = gam(ub)
        un = boris(hc * gb / gmu(ub, gb))
        gn = gam(un)
        hd = hc / gmu(un, gn)
        dx, dy, ds = hd * un[0], hd * un[1], hd * un[2]
        X1 = p["X"] + dx / w.hx
        Y1 = p["Y"] + dy / w.hy if w.ny > 1 else p["Y"]
        j = torch.zeros((3, w.ny, w.nx), dtype=torch.float64, device=self.dev)
        self.esirkepov(j, p["X"], p["Y"], X1, Y1, p["q"], dy, h)
        gx, gy = torch.floor(X1), torch.floor(Y1)
        ax, ay, vz = X1 - gx, Y1 - gy, p["q"] * ds / h
        if w.ny > 1:
            for a, wx in ((0, 1 - ax), (1, ax)):
                for b, wy in ((0, 1 - ay), (1, ay)):
                    self.add(j[2], gx + a, gy + b, wx * wy * vz)
        else:
            self.add(j[2], gx, gy, (1 - ax) * vz)
            self.add(j[2], gx + 1, gy, ax * vz)
        dt = hd * gn
        kin = (p["q"] * w.hx * w.hy * (sp.mass / sp.charge) * (gn - 1) * dt).sum()
        flux = (p["q"] * ~trap).sum() * w.hx * w.hy * h
        keep = ~trap
        q = dict(X=torch.remainder(X1, w.nx), Y=torch.remainder(Y1, w.ny), ux=un[0], uy=un[1],
                 uz=un[2], sig=p["sig"] + ds, q=p["q"])
        if bool(trap.any()):
            q = {k: v[keep] for k, v in q.items()}
        return q, j, kin, flux, int(trap.sum())

    def esirkepov(self, j, X0, Y0, X1, Y1, q, dy, h):
        w = self.w
        dX, dY = X1 - X0, Y1 - Y0
        m = torch.maximum(dX.abs(), dY.abs())
        ns = torch.where(m > 1, torch.ceil(m), torch.ones_like(m))
        for s in range(int(ns.max())):
            on = (s < ns).to(q.dtype)
            xa, xb = X0 + dX * (s / ns), X0 + dX * ((s + 1) / ns)
            bx = torch.floor(torch.minimum(xa, xb))
            Sx = [(torch.clamp(1 - (xa - bx - i).abs(), min=0), torch.clamp(1 - (xb - bx - i).abs(), min=0))
                  for i in range(3)]
            e0 = -(q * w.hx / h) * (Sx[0][1] - Sx[0][0]) * on
            ex = (e0, e0 - (q * w.hx / h) * (Sx[1][1] - Sx[1][0]) * on)
            mx = [0.5 * (a + b) for a, b in Sx]
            if w.ny == 1:
                vy = q * dy / ns / h * on
                for i in range(2):
                    self.add(j[0], bx + i, Y0, ex[i])
                for i in range(3):
                    self.add(j[1], bx + i, Y0, vy * mx[i])
                continue
            ya, yb = Y0 + dY * (s / ns), Y0 + dY * ((s + 1) / ns)
            by = torch.floor(torch.minimum(ya, yb))
            Sy = [(torch.clamp(1 - (ya - by - i).abs(), min=0), torch.clamp(1 - (yb - by - i).abs(), min=0))
                  for i in range(3)]
            e0 = -(q * w.hy / h) * (Sy[0][1] - Sy[0][0]) * on
            ey = (e0, e0 - (q * w.hy / h) * (Sy[1][1] - Sy[1][0]) * on)
            my = [0.5 * (a + b) for a, b in Sy]
            for a in range(2):
                for b in range(3):
                    self.add(j[0], bx + a, by + b, ex[a] * my[b])
                    self.add(j[1], bx + b, by + a, ey[a] * mx[b])

    def march(self, D, inject):
        w = self.w
        kx, ky = self.kx, self.ky
        K2 = kx * kx + ky * ky
        sx = torch.exp(-0.5j * kx * w.hx)
        sy = torch.exp(-0.5j * ky * w.hy) if w.ny > 1 else 1.0
        old, new = self.S, torch.zeros_like(self.S)
        zero = torch.zeros_like(old[0, 0])
        Rx, Ry, Lx, Ly, Ez, Bz = (zero,) * 6
        jpx = jpy = zero
        part = self.layer() if inject else None
        fields = torch.zeros((6, w.ny, w.nx), dtype=torch.float64, device=self.dev)
        kin = flux = fe = 0.0
        trapped = 0
        for n in range(w.nzeta - 1, -1, -1):
            h = self.hz[n]
            jx = jy = jz = zero
            if inject:
                part, j, dk, df, nt = self.push(part, fields, h)
                kin, flux, trapped = kin + dk, flux + df, trapped + nt
                J = self.spectrum(j)
                jx, jy, jz = J[0] * sx, J[1] * sy, J[2]
            if n + 1 < w.nzeta:
                Rx, Ry = Rx - 0.25 * D * (jx - jpx), Ry - 0.25 * D * (jy - jpy)
                new[0, n + 1], new[1, n + 1], new[2, n + 1], new[3, n + 1] = Rx, Ry, Ez, Bz
            new[4, n], new[5, n] = jx, jy
            m = max(n - 1, 0)
            Jx = old[4, m] + old[4, n] + 2 * jx
            Jy = old[5, m] + old[5, n] + 2 * jy
            ox, oy, oe, ob = old[0, n], old[1, n], old[2, n], old[3, n]
            c = 16 - h * h * K2
            nE = (c * Ez - 16 * h * jz - 1j * h * D * (kx * Jx + ky * Jy) - 2 * h * D * K2 * oe
                  + 2j * h * h * (kx * jx + ky * jy)
                  + 4j * h * (kx * (Rx + ox - 2 * Lx) + ky * (Ry + oy - 2 * Ly)))
            nB = (c * Bz + 2j * h * h * (kx * jy - ky * jx) + 1j * h * D * (kx * Jy - ky * Jx)
                  - 2 * h * D * K2 * ob + 4j * h * (ky * (Rx + ox + 2 * Lx) - kx * (Ry + oy + 2 * Ly)))
            Dd = 16 + h * (2 * D + h) * K2
            e, b = nE / Dd, nB / Dd
            Rx = ox + D * (0.5j * (kx * (e + oe) + ky * (b + ob)) - 0.25 * Jx)
            Ry = oy + D * (0.5j * (ky * (e + oe) - kx * (b + ob)) - 0.25 * Jy)
            Lx = Lx - 0.5 * h * (0.5j * (kx * (Ez + e) - ky * (Bz + b)) + jx)
            Ly = Ly - 0.5 * h * (0.5j * (ky * (Ez + e) + kx * (Bz + b)) + jy)
            Ez, Bz = e, b
            Rx, Ry, Lx, Ly, Ez, Bz = (v * self.keep for v in (Rx, Ry, Lx, Ly, Ez, Bz))
            jpx, jpy = jx, jy
            fields = self.real(torch.stack((0.5 * (Rx + Lx), 0.5 * (Ry + Ly), Ez, 0.5 * (Ly - Ry),
                                            0.5 * (Rx - Lx), Bz)))
            fe = fe + (fields * fields).sum() * h
        new[0, 0], new[1, 0], new[2, 0], new[3, 0] = Rx, Ry, Ez, Bz
        self.S = new
        self.k += 1 if inject else 0
        return trapped, {"field_energy": 0.5 * w.hx * w.hy * float(fe), "kinetic_energy": float(kin),
                         "charge_flux": float(flux)}


def _net(P, j):
    """The net's correction r for the normalised current [nz, 3, ny, nx], FP64, in planes."""
    x = j
    for l in (1, 2, 3):
        Wt, b = P[f"W{l}"], P[f"b{l}"]
        x = torch.nn.functional.pad(x, (0, 0, 0, 0, 0, 0, 1, 1))
        nz = x.shape[0] - 2
        acc = None
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3 - 1, t % 3 - 1
            s = torch.roll(x[dz:dz + nz], shifts=(-dy, -dx), dims=(2, 3))
            v = torch.einsum("zcyx,co->zoyx", s, Wt[dz, dy + 1, dx + 1])
            acc = v if acc is None else acc + v
        x = acc + b.view(1, -1, 1, 1)
        if l < 3:
            x = torch.relu(x)
    return x


def _net_params(seed):
    P, out, o = _params(seed), {}, 0
    for l, (ci, co) in enumerate(((3, 16), (16, 16), (16, 3)), start=1):
        n = 27 * ci * co
        out[f"W{l}"] = torch.tensor(P[o:o + n].astype(np.float64).reshape(3, 3, 3, ci, co), device="cuda")
        out[f"b{l}"] = torch.tensor(P[o + n:o + n + co].astype(np.float64), device="cuda")
        o += n + co
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        j, P = _currents(case, seed)[0].double(), _net_params(seed)
        nz, out = case["nz"], torch.empty_like(j)
        for z in range(0, nz, 16):                # a group of planes and the net's reach around it
            a, b = max(0, z - 3), min(nz, z + 19)
            r = _net(P, j[a:b] / NET_SCALE)       # (planes within reach of a cut are not used)
            out[z:z + 16] = j[z:z + 16] + NET_SCALE * r[z - a:z - a + min(16, nz - z)]
        return out
    if kind == "train":
        noisy, clean = (t.double() / NET_SCALE for t in _currents(case, seed))
        P = _net_params(seed)
        for t in P.values():
            t.requires_grad_(True)
        e = (noisy + _net(P, noisy) - clean)[3:case["nz"] - 3]
        loss = (e * e).mean()
        loss.backward()
        new = [(P[k] - 1e-3 * P[k].grad / (P[k].grad.abs() + 1e-8)).detach().reshape(-1)
               for l in (1, 2, 3) for k in (f"W{l}", f"b{l}")]
        return {"loss": float(loss), "params": torch.cat(new)}
    # plain FP64 s-steps where they take seconds
    if kind not in ("march", "streamed") or case["family"] == "pwfa3d":
        return None
    if case["steps"] * case["nz"] > (11000 if case["ny"] == 1 else 4000):
        return None
    w = _workload(case, seed)
    sim, trapped, d = _Plain(w), 0, {}
    for _ in range(case["steps"]):
        if trapped:
            return None                           # later s-steps would need the stored set
        trapped, d = sim.march(w.delta, True)
    if trapped:
        d["kinetic_energy"] = None                # the stored set's energy is part of it
    return {"state": sim.S, **d}

