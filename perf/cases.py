"""Performance cases: the work that a user of this framework has it do, through
paper_2010_00409_gb300.psatd (contexts, batches, one-shots, the surrogate).

  steps     n PSATD steps of one box (complex64, complex128 or real float32 storage)
  batch     one persistent launch that steps many boxes of different sizes
  one_shot  pulse to focal plane in one exact step
  scan      the focal plane at several times, one exact step of its own each
  patch     a focal patch of the surrogate's training set (one-shot + P planes)
  job       a whole small run: pulse, steps, focal plane, diagnostics
  train     the surrogate's forward, loss and backward pass
  infer     the surrogate's forward pass

Every input comes from the seed; `exact` evaluates the same formulas in float64
(the pulse of Sec. 2.2 / 3.2.1 on the mapped layer, Eq. 3-4 per mode between 3D
DFTs, the trigonometric interpolant with the cut-out of Eq. 14-16, the network).
"""
import math

import numpy as np
import torch

from paper_2010_00409_gb300 import psatd
from paper_2010_00409_gb300 import workloads as W

C = 2.99792458e10
LAM = 800e-7

# 5-smooth lengths the solver takes, as far as the cases go
SMOOTH = [n for n in range(8, 1025)
          if any(n == 2 ** a * 3 ** b * 5 ** c for a in range(11) for b in range(7) for c in range(5))]


def listed():
    return [
        # the plain method's check run: 64^3, FP64, 20 steps of the Courant value
        {"name": "steps_64_f64", "do": "steps", "storage": "c128", "nx": 64, "ny": 64, "nz": 64, "steps": 20},
        # the tight-focus box on real storage (the solver's main configuration), a burst of steps
        {"name": "steps_256_real", "do": "steps", "storage": "real", "nx": 256, "ny": 256, "nz": 256, "steps": 8},
        # the same box on complex storage, the default of a context
        {"name": "steps_256_c64", "do": "steps", "storage": "c64", "nx": 256, "ny": 256, "nz": 256, "steps": 4},
        # one box of a parameter sweep by itself: mixed-radix lengths, unequal axes
        {"name": "steps_ragged_c64", "do": "steps", "storage": "c64", "nx": 180, "ny": 135, "nz": 150, "steps": 4},
        # a large multi-octave box: 512-point axes, 6.4 GB of fields
        {"name": "steps_512_c64", "do": "steps", "storage": "c64", "nx": 512, "ny": 512, "nz": 512, "steps": 1},
        # a sweep of pulse realisations on uneven layers, stepped together
        {"name": "batch_16_c64", "do": "batch", "boxes": 16, "sweep": 0, "steps": 2},
        # one focal field of the tight-focus box
        {"name": "one_shot_256_real", "do": "one_shot", "storage": "real", "nx": 256, "ny": 256, "nz": 256, "plane": 128},
        # the focal plane at four times around the focus
        {"name": "scan_96_c64", "do": "scan", "storage": "c64", "nx": 96, "ny": 108, "nz": 108, "plane": 64, "times": 4},
        # one sample of the surrogate's training set
        {"name": "patch_128_c64", "do": "patch", "storage": "c64", "nx": 128, "ny": 128, "nz": 128, "plane": 64},
        # a whole small run, bound by launches and latency
        {"name": "job_64_c64", "do": "job", "storage": "c64", "nx": 64, "ny": 64, "nz": 64, "steps": 16, "plane": 64},
        # the surrogate's training step at its usual size
        {"name": "train_8", "do": "train", "batch": 8, "patch": 64, "width": 32, "layers": 4, "modes": 12, "hidden": 64},
        # the surrogate asked for one focal field
        {"name": "infer_1", "do": "infer", "batch": 1, "patch": 64, "width": 32, "layers": 4, "modes": 12, "hidden": 64},
    ]


def _near(rng, lo, hi):
    """A 5-smooth length, log-uniform in [lo, hi]."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in SMOOTH if lo <= n <= hi), key=lambda n: abs(math.log(n / v)))


def draw(rng):
    do = rng.choice(["steps", "steps", "steps", "batch", "one_shot", "scan", "patch", "job", "train", "infer"])
    if do == "steps":
        storage = rng.choice(["c64", "c64", "c128", "real"])
        if storage == "real":
            return {"do": do, "storage": storage, "nx": 256, "ny": 256, "nz": rng.choice([64, 128, 256]),
                    "steps": rng.randint(1, 8)}
        most = 2.0 ** (22 if storage == "c128" else 26.5)
        while True:
            c = {"do": do, "storage": storage, "nx": _near(rng, 16, 1024), "ny": _near(rng, 8, 512),
                 "nz": _near(rng, 8, 512), "steps": rng.randint(1, 8)}
            if 2 ** 11 <= c["nx"] * c["ny"] * c["nz"] and c["nx"] * c["ny"] * c["nz"] * c["steps"] <= most:
                return c
    if do == "batch":
        return {"do": do, "boxes": rng.randint(3, 16), "sweep": rng.randint(1, 1000), "steps": rng.randint(1, 2)}
    if do in ("train", "infer"):
        return {"do": do, "batch": rng.randint(1, 8), "patch": rng.choice([32, 40, 48, 64]),
                "width": rng.choice([16, 20, 24, 32]), "layers": rng.randint(2, 4), "modes": rng.randint(6, 12),
                "hidden": rng.choice([32, 48, 64])}
    storage = rng.choice(["c64", "real"]) if do == "one_shot" else "c64"
    plane = rng.choice([32, 48, 64, 96, 128]) if do != "patch" else rng.choice([24, 32, 48, 64])
    if storage == "real":
        c = {"do": do, "storage": storage, "nx": 256, "ny": 256, "nz": rng.choice([128, 256]), "plane": plane}
    else:
        c = {"do": do, "storage": storage, "nx": _near(rng, 64, 256), "plane": plane}
        c["ny"] = c["nz"] = _near(rng, 64, 256 if do == "one_shot" else 160)
    if do == "scan":
        c["times"] = rng.randint(2, max(2, min(6, 10_000_000 // (c["nx"] * c["ny"] * c["nz"]))))
    if do == "job":
        c["steps"] = rng.randint(4, 24)
    return c


# ---------------------------------------------------------------------------
# geometry and the pulse, in float64

class Box:
    """A periodic layer with its mapping and a Gaussian pulse (the f-number, CEP,
    ellipticity and polarisation of the seed)."""

    def __init__(self, nx, ny, nz, f, rng, R0=20.0, L=9.0):
        lam = LAM
        self.Nx, self.Ny, self.Nz = nx, ny, nz
        self.theta = math.atan(1.0 / (2.0 * f))
        self.eps = 0.2
        support = 2 * self.theta + 0.5 * self.eps
        self.R0, self.L = R0 * lam, L * lam
        r_min, r_max = self.R0 - 0.5 * self.L, self.R0 + 0.5 * self.L
        D = (1.05 + 0.02 * rng.random()) * (r_max - r_min * math.cos(support))
        H = r_max * math.sin(min(support, math.pi / 2)) * (1.0 + 0.01 * rng.random()) + lam
        self.dx, self.dy, self.dz = D / nx, 2 * H / ny, 2 * H / nz
        self.x_min, self.y_min, self.z_min = -r_min - D, -H, -H
        self.lam, self.ncyc, self.P0 = lam, 2.0, 1e7
        self.cep = 2 * math.pi * rng.random()
        self.ell = rng.random()
        self.psi = math.pi * rng.random()
        self.T = self.R0 / C

    @property
    def cells(self):
        return self.Nx * self.Ny * self.Nz

    def dt(self):
        """The Courant value, rounded so that a step lands on the focus."""
        d = 1.0 / (C * math.sqrt(1 / self.dx ** 2 + 1 / self.dy ** 2 + 1 / self.dz ** 2))
        return self.T / math.ceil(self.T / d)

    def grid(self):
        return W.GridSpec(self.Nx, self.Ny, self.Nz, self.dx, self.dy, self.dz, self.x_min, self.y_min, self.z_min, C)

    def mapping(self):
        return W.MappingSpec(self.R0, self.L)

    def pulse(self):
        return W.PulseSpec(kind=W.GAUSSIAN, lam=self.lam, theta=self.theta, eps=self.eps, P0=self.P0,
                           n_cycles=self.ncyc, cep=self.cep, ellipticity=self.ell, pol_angle=self.psi, div_project=1)

    def field(self, out):
        """The pulse's E and B on the layer into out [6, Nz, Ny, Nx] (any real or
        complex type), slab by slab in float64; replicas along x summed."""
        dev = out.device
        f64 = dict(dtype=torch.float64, device=dev)
        th, R0, L, lam = self.theta, self.R0, self.L, self.lam
        amp = math.sqrt(4 * self.P0 / (C * R0 * R0 * (th ** 2 / 4 - th ** 4 / 48 + th ** 6 / 960)))
        D = self.Nx * self.dx
        x = self.x_min + self.dx * torch.arange(self.Nx, **f64)
        y = (self.y_min + self.dy * torch.arange(self.Ny, **f64))[None, :, None]
        r_max = R0 + 0.5 * L
        ms = range(math.floor((-r_max - (self.x_min + D)) / D), math.ceil((r_max - self.x_min) / D) + 1)
        lim, e = 2 * th, self.eps
        step = max(1, (1 << 23) // (self.Nx * self.Ny))
        cp, sp = math.cos(self.psi), math.sin(self.psi)
        for z0 in range(0, self.Nz, step):
            z = (self.z_min + self.dz * torch.arange(z0, min(self.Nz, z0 + step), **f64))[:, None, None]
            acc = torch.zeros((6, z.shape[0], self.Ny, self.Nx), **f64)
            for m in ms:
                X = (x + m * D)[None, None, :]
                if float(X.min()) > 0 or float(X.max()) < -r_max:
                    continue                                    # no point of the sector x < 0, R <= R_max
                R = torch.sqrt(X * X + y * y + z * z)
                zeta = R - R0
                al = torch.atan2(torch.sqrt(y * y + z * z), -X)
                ts = torch.where(al <= lim - 0.5 * e, 1.0, torch.cos(math.pi * (al - lim + 0.5 * e) / (2 * e)) ** 2)
                ts = torch.where((al <= lim + 0.5 * e) & (zeta.abs() <= 0.5 * L) & (R > 0), ts, 0.0)
                env = amp * R0 / R * ts * torch.exp(-(al / th) ** 2 - zeta ** 2 * math.log(4.0) / (self.ncyc * lam) ** 2)
                env = torch.where(R > 0, env, 0.0)
                for k, (d1, d2) in enumerate(((cp, sp), (-sp, cp))):
                    u = env * torch.sin(2 * math.pi / lam * zeta + self.cep + 0.5 * math.pi * k)
                    if k:
                        u = u * self.ell
                    a0, a1, a2 = d1 * z - d2 * y, d2 * X, -d1 * X      # d x R, d = (0, d1, d2)
                    b0, b1, b2 = y * a2 - z * a1, z * a0 - X * a2, X * a1 - y * a0
                    n1 = torch.sqrt(a0 * a0 + a1 * a1 + a2 * a2)
                    n0 = torch.sqrt(b0 * b0 + b1 * b1 + b2 * b2)
                    u0, u1 = torch.where(n0 > 0, u / n0, 0.0), torch.where(n1 > 0, u / n1, 0.0)
                    for q, v in enumerate((b0 * u0, b1 * u0, b2 * u0, a0 * u1, a1 * u1, a2 * u1)):
                        acc[q] += v
            out[:, z0:z0 + z.shape[0]] = acc
        return out


def _box(case, seed):
    return Box(case["nx"], case["ny"], case["nz"], 1.0, np.random.default_rng(seed))


def _sweep_boxes(case, seed):
    """Realisations of a sweep: f-number in [0.5, 2], R0 = max(20, 10 f^2) lambda,
    lengths from the solver's usual ones for 8 points per wavelength along x and
    the pulse's transverse support across (the sizes depend on the case alone)."""
    sizes = (96, 100, 108, 120, 128, 135, 144, 150, 160, 162, 180, 192)
    shape, rng = np.random.default_rng(case["sweep"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["boxes"]):
        f = shape.uniform(0.5, 2.0)
        th = math.atan(1.0 / (2.0 * f))
        sup, R0 = 2 * th + 0.1, max(20.0, 10.0 * f * f)
        nx = 8 * 1.05 * (R0 + 4.5 - (R0 - 4.5) * math.cos(sup))
        nt = 2 * ((R0 + 4.5) * math.sin(min(sup, math.pi / 2)) + 1) * 2.6 * math.sin(min(sup, math.pi / 2))
        up = [next((s for s in sizes if s >= n), sizes[-1]) for n in (nx, nt)]
        out.append(Box(up[0], up[1], up[1], f, rng, R0=R0))
    return out


def _plane(box, case, n=None):
    h = 1.5 * box.lam
    n = n or case["plane"]
    return n, n, -h, h, -h, h


def _times(box, case):
    return [box.T + (k - case["times"] // 2) * 0.25 * box.lam / C for k in range(case["times"])]


def _context(box, case, stream=None):
    real = case.get("storage") == "real"
    return psatd.Context(box.grid(), box.mapping(), box.dt(), 64 if case.get("storage") == "c128" else 32,
                         stream=stream, real=real)


# ---------------------------------------------------------------------------
# the surrogate's weights and data

def _fno_shapes(case):
    c, m, n_in = case["width"], case["modes"], 6 + 3
    modes = 4 * m ** 3
    s = [("lw", (c, n_in)), ("lb", (c,))]
    for l in range(case["layers"]):
        s += [("R%d" % l, (2, modes, c, c)), ("W%d" % l, (c, c)), ("b%d" % l, (c,))]
    return s + [("q1w", (case["hidden"], c)), ("q1b", (case["hidden"],)), ("q2w", (3, case["hidden"])), ("q2b", (3,))]


def _fno_inputs(case, seed):
    """Flat weights (as the model lays them out), pulse parameters in [-1, 1] and a
    smooth focal-spot-like target per sample."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    parts = []
    for name, s in _fno_shapes(case):
        if name[0] == "R":
            parts.append((u(s) / case["width"] ** 2).reshape(-1))
        elif len(s) == 1:
            parts.append(0.1 * (2 * u(s) - 1))
        else:
            parts.append(((2 * u(s) - 1) / math.sqrt(s[1])).reshape(-1))
    B, P = case["batch"], case["patch"]
    prm = 2 * u(B, 6) - 1
    x = -2 + 4 * torch.arange(P, device="cuda", dtype=torch.float32) / P
    r2 = x[:, None, None] ** 2 + x[None, :, None] ** 2
    k = 1 + 0.2 * prm[:, 1]
    env = torch.exp(-r2[None] - (x ** 2)[None, None, None, :] * (0.5 + 0.2 * prm[:, 2])[:, None, None, None])
    ph = 2 * math.pi * k[:, None, None, None] * x[None, None, None, :] + prm[:, 0, None, None, None]
    w = torch.stack([prm[:, 3], 1 + 0.3 * prm[:, 4], prm[:, 5]], 1)
    tgt = (w[:, :, None, None, None] * (env * torch.sin(ph))[:, None]).contiguous()
    return torch.cat(parts), prm.contiguous(), tgt


# ---------------------------------------------------------------------------

def prepare(case, seed):
    do = case["do"]
    s = {"case": case}
    if do in ("train", "infer"):
        theta, s["prm"], s["target"] = _fno_inputs(case, seed)
        s["net"] = psatd.Fno(6, width=case["width"], layers=case["layers"], patch=case["patch"], modes=case["modes"],
                             hidden=case["hidden"], out_channels=3, max_batch=case["batch"], seed=0)
        s["net"].params.copy_(theta)
        return s
    if do == "batch":
        boxes = _sweep_boxes(case, seed)
        s["stream"] = torch.cuda.Stream()
        with torch.cuda.stream(s["stream"]):
            s["ctx"] = [_context(b, case, s["stream"]) for b in boxes]
            for b, c in zip(boxes, s["ctx"]):
                b.field(c.fields)
        # boxes step to their own focus: the counts differ
        s["counts"] = [case["steps"] + (k & 1) for k in range(case["boxes"])]
        torch.cuda.synchronize()
        return s
    box = s["box"] = _box(case, seed)
    ctx = s["ctx"] = _context(box, case)
    if do == "steps":
        box.field(ctx.fields)
        return s
    n = case["plane"]
    if do == "patch":
        s["plane"] = torch.empty((3, n, n), dtype=torch.complex64, device="cuda")
        s["out"] = torch.empty((3, n, n, n), dtype=torch.float32, device="cuda")
    elif do != "job":
        s["out"] = [torch.empty((3, n, n), dtype=torch.complex64, device="cuda")
                    for _ in range(case.get("times", 1))]
    return s


def _held(net, view):
    """A view of the model's own memory, which lives as long as the model: the
    view keeps the model, as a program that reads the result later has to."""
    view.owner = net
    return view


def run(s):
    case = s["case"]
    do = case["do"]
    if do == "train":
        s["net"].loss_backward(s["prm"], s["target"], want_loss=False)
        return {"grads": _held(s["net"], s["net"].grads), "out": _held(s["net"], s["net"].output(case["batch"]))}
    if do == "infer":
        return _held(s["net"], s["net"].forward(s["prm"]))
    if do == "batch":
        psatd.multi_advance(s["ctx"], s["counts"])
        return [c.fields for c in s["ctx"]]
    box, ctx = s["box"], s["ctx"]
    if do == "steps":
        ctx.advance(case["steps"])
        return ctx.fields
    if do in ("one_shot", "scan"):
        for T, out in zip(_times(box, case) if do == "scan" else [box.T], s["out"]):
            ctx.focal_one_shot(box.pulse(), T, 0.0, *_plane(box, case), out=out)
        return s["out"]
    if do == "patch":
        h, n = 2 * box.lam, case["plane"]
        for i in range(n):
            x = -h + 2 * h * i / n
            if i == 0:
                ctx.focal_one_shot(box.pulse(), box.T, x, n, n, -h, h, -h, h, out=s["plane"])
            else:
                ctx.sample_focal_plane(x, n, n, -h, h, -h, h, out=s["plane"])
            s["out"][:, :, :, i] = s["plane"].real
        return s["out"]
    # job: the pulse, some steps, the plane through the layer's middle and the diagnostics, on the host
    ctx.init_pulse(box.pulse())
    ctx.advance(case["steps"])
    plane = ctx.sample_focal_plane(_job_x(box, case), *_plane(box, case))
    d = ctx.diagnostics()
    return {"plane": plane, "fields": ctx.fields,
            "numbers": [d[k] for k in ("energy", "energy_E", "energy_B", "max_E_hat", "max_B_hat")]}


def _job_x(box, case):
    """Where the pulse's centre on the axis is after the steps."""
    return -box.R0 + C * case["steps"] * box.dt()


def work(case):
    """Bytes: the fields read and written once per step (a step leaves its result in
    storage), a plane or patch written once; transforms at 5 N log2 N flops."""
    do = case["do"]
    if do in ("train", "infer"):
        B, P, c, L, h = case["batch"], case["patch"], case["width"], case["layers"], case["hidden"]
        m, nv = case["modes"], case["patch"] ** 3
        spec = 8 * m ** 3 * c * c * L
        point = 2.0 * B * nv * (9 * c + L * c * c + c * h + 3 * h)
        fft = 2 * L * B * c * 2.5 * nv * math.log2(nv)
        io = 4.0 * (spec + B * 3 * nv)
        return {"bytes": io, "flops": point + fft + 8.0 * 4 * m ** 3 * B * c * c * L} if do == "infer" else \
            {"bytes": 2 * io + 4.0 * B * 3 * nv, "flops": 3 * (point + fft)}
    if do == "batch":
        boxes = _sweep_boxes(case, 0)
        n = sum((case["steps"] + (k & 1)) * b.cells for k, b in enumerate(boxes))
        lg = max(math.log2(b.cells) for b in boxes)
        return {"bytes": 96.0 * n, "flops": n * (60 * lg + 80)}
    cells = case["nx"] * case["ny"] * case["nz"]
    lg = math.log2(cells)
    per = {"c64": 96.0, "c128": 192.0, "real": 48.0}[case["storage"]]
    half = 0.5 if case["storage"] == "real" else 1.0
    if do == "steps":
        return {"bytes": per * cells * case["steps"], "flops": half * cells * case["steps"] * (60 * lg + 80)}
    n = case["plane"]
    one = half * cells * (30 * lg + 80)
    if do == "one_shot" or do == "scan":
        k = case.get("times", 1)
        return {"bytes": k * 24.0 * n * n, "flops": k * (one + half * 24.0 * cells)}
    if do == "patch":
        return {"bytes": 12.0 * n ** 3, "flops": one + 24.0 * n * cells}
    return {"bytes": (case["steps"] + 1) * per * cells, "flops": cells * (case["steps"] + 1) * (60 * lg + 80)}


# ---------------------------------------------------------------------------
# the same in float64

def _k(box):
    f64 = dict(dtype=torch.float64, device="cuda")
    k = [2 * math.pi * torch.fft.fftfreq(n, d, **f64)
         for n, d in ((box.Nx, box.dx), (box.Ny, box.dy), (box.Nz, box.dz))]
    return k[0][None, None, :], k[1][None, :, None], k[2][:, None, None]


def _dot(a, v):
    return a[0] * v[0] + a[1] * v[1] + a[2] * v[2]


def _update(F, box, t, real, project):
    """Eq. 3-4 for one step t on the spectra F (six complex128 [Nz, Ny, Nx], in
    place), slab by slab along z; the fields of real storage take the mean over
    the two mirrored wave numbers of a Nyquist plane."""
    kx, ky, kz = _k(box)
    step = max(1, (1 << 24) // (box.Nx * box.Ny))
    for z0 in range(0, box.Nz, step):
        sl = slice(z0, min(box.Nz, z0 + step))
        kk = (kx, ky, kz[sl])
        km = torch.sqrt(kk[0] ** 2 + kk[1] ** 2 + kk[2] ** 2)
        inv = torch.where(km > 0, 1.0 / km, 0.0)
        n = [k * inv for k in kk]
        m, a = n, n
        if real:
            nyq = [(2 * torch.arange(N, device="cuda") == N) for N in (box.Nx, box.Ny, box.Nz)]
            nyq = [nyq[0][None, None, :], nyq[1][None, :, None], nyq[2][sl, None, None]]
            m = [torch.where(q, -v, v) for q, v in zip(nyq, n)]
            a = [torch.where(q, 0.0, v) for q, v in zip(nyq, n)]
        E, B = [F[q][sl] for q in range(3)], [F[q][sl] for q in range(3, 6)]

        def across(V):
            p, q = _dot(n, V), _dot(m, V)
            return [v - 0.5 * (x * p + y * q) for v, x, y in zip(V, n, m)]
        if project:
            B = across(B)
            if real:
                E = across(E)
        cs, sn = torch.cos(C * km * t), torch.sin(C * km * t)
        Et = across(E)
        cB = [a[1] * B[2] - a[2] * B[1], a[2] * B[0] - a[0] * B[2], a[0] * B[1] - a[1] * B[0]]
        cE = [a[1] * E[2] - a[2] * E[1], a[2] * E[0] - a[0] * E[2], a[0] * E[1] - a[1] * E[0]]
        for q in range(3):
            F[q][sl] = cs * Et[q] + 1j * sn * cB[q]
            F[q + 3][sl] = cs * B[q] - 1j * sn * cE[q]


def _start(box, kind):
    """The pulse as storage of `kind` holds it, as six complex128 tensors."""
    dt = {"c64": torch.complex64, "c128": torch.complex128, "real": torch.float32}.get(kind, torch.float64)
    f = box.field(torch.empty((6, box.Nz, box.Ny, box.Nx), dtype=dt, device="cuda"))
    return [f[q].to(torch.complex128) for q in range(6)]


def _steps(F, box, t, n, real):
    for _ in range(n):
        for q in range(6):
            F[q] = torch.fft.fftn(F[q])
        _update(F, box, t, real, False)
        for q in range(6):
            F[q] = torch.fft.ifftn(F[q])
            if real:
                F[q] = F[q].real.to(torch.complex128)
    return F


def _phases(box, axis, at):
    n, d, lo = ((box.Nx, box.dx, box.x_min), (box.Ny, box.dy, box.y_min), (box.Nz, box.dz, box.z_min))[axis]
    k = 2 * math.pi * torch.fft.fftfreq(n, d, dtype=torch.float64, device="cuda")
    return torch.exp(1j * k[None, :] * (torch.as_tensor(at, dtype=torch.float64, device="cuda") - lo)[:, None])


def _cut(box, t, x, y, z):
    """I_S of Eq. 15-16 at the points (x scalar; y [ny]; z [nz]) -> [nz, ny]."""
    R = torch.sqrt(x * x + y[None, :] ** 2 + z[:, None] ** 2)
    r_min, r_max = box.R0 - 0.5 * box.L, box.R0 + 0.5 * box.L
    l, r = -r_max + C * t, -r_min + C * t
    zero = torch.zeros_like(R, dtype=torch.bool)
    if r < 0:
        zero |= (R >= -l) | (R < -r) | (x > 0)
    if l <= 0 <= r:
        zero |= (R > box.L) if x < 0 else (R > r)
    if l > 0:
        zero |= (R <= l) | (R > r) | (x < 0)
    return (~zero).to(torch.float64)


def _planes(G, box, t, xs, n, lo, hi):
    """Components 0..2 of the interpolant of the spectrum G (with its 1/N) on the
    planes x = xs: [3, len(xs), nz, ny]."""
    at = lo + (hi - lo) * np.arange(n) / n
    wx, wy, wz = _phases(box, 0, xs), _phases(box, 1, at), _phases(box, 2, at)
    y = torch.as_tensor(at, dtype=torch.float64, device="cuda")
    cut = torch.stack([_cut(box, t, float(x), y, y) for x in xs])
    res = []
    for q in range(3):
        g = torch.tensordot(G[q], wx, ([2], [1]))          # [Nz, Ny, X]
        h = torch.tensordot(g, wy, ([1], [1]))             # [Nz, X, ny]
        res.append(torch.einsum("lxp,ql->xqp", h, wz) * cut / box.cells)
    return torch.stack(res)


def _one_step(box, case, T, project=True):
    F = _start(box, None)
    for q in range(6):
        F[q] = torch.fft.fftn(F[q])
    _update(F, box, T, case["storage"] == "real", project)
    return F


def _network(case, theta, prm):
    B, P, c, m = case["batch"], case["patch"], case["width"], case["modes"]
    p, at = {}, 0
    for name, s in _fno_shapes(case):
        n = math.prod(s)
        p[name] = theta[at:at + n].view(s)
        at += n
    x = -1 + 2 * torch.arange(P, dtype=torch.float64, device="cuda") / P
    grid = [x[None, None, :].expand(P, P, P), x[None, :, None].expand(P, P, P), x[:, None, None].expand(P, P, P)]
    feat = torch.cat([prm[:, :, None, None, None].expand(B, 6, P, P, P), torch.stack(grid)[None].expand(B, 3, P, P, P)], 1)
    mix = lambda w, v: torch.einsum("oi,bizyx->bozyx", w, v)  # noqa: E731
    bias = lambda b: b[None, :, None, None, None]  # noqa: E731
    v = mix(p["lw"], feat) + bias(p["lb"])
    keep = torch.cat([torch.arange(m), torch.arange(P - m, P)]).cuda()
    for l in range(case["layers"]):
        s = torch.fft.rfftn(v, dim=(-3, -2, -1))[..., :m].index_select(2, keep).index_select(3, keep)
        r = torch.complex(p["R%d" % l][0], p["R%d" % l][1]).view(2 * m, 2 * m, m, c, c)
        s = torch.einsum("bizyx,zyxio->bozyx", s, r)
        full = torch.zeros((B, c, P, 2 * m, m), dtype=s.dtype, device="cuda").index_copy(2, keep, s)
        full = torch.zeros((B, c, P, P, m), dtype=s.dtype, device="cuda").index_copy(3, keep, full)
        full = torch.nn.functional.pad(torch.view_as_real(full), (0, 0, 0, P // 2 + 1 - m))
        z = torch.fft.irfftn(torch.view_as_complex(full.contiguous()), s=(P, P, P), dim=(-3, -2, -1))
        z = z + mix(p["W%d" % l], v) + bias(p["b%d" % l])
        v = torch.nn.functional.gelu(z) if l + 1 < case["layers"] else z
    h = torch.nn.functional.gelu(mix(p["q1w"], v) + bias(p["q1b"]))
    return mix(p["q2w"], h) + bias(p["q2b"])


def exact(case, seed):
    do = case["do"]
    if do in ("train", "infer"):
        theta, prm, tgt = (t.to(torch.float64) for t in _fno_inputs(case, seed))
        if do == "infer":
            return _network(case, theta, prm)
        theta.requires_grad_(True)
        out = _network(case, theta, prm)
        ((out - tgt) ** 2).mean().backward()
        return {"grads": theta.grad, "out": out.detach()}
    if do == "batch":
        return [torch.stack(_steps(_start(b, "c64"), b, b.dt(), case["steps"] + (k & 1), False))
                for k, b in enumerate(_sweep_boxes(case, seed))]
    box = _box(case, seed)
    real = case["storage"] == "real"
    if do == "steps":
        F = torch.stack(_steps(_start(box, case["storage"]), box, box.dt(), case["steps"], real))
        return F.real if real else F
    if do in ("one_shot", "scan"):
        n, _, lo, hi, _, _ = _plane(box, case)
        return [_planes(_one_step(box, case, T), box, T, [0.0], n, lo, hi)[:, 0]
                for T in (_times(box, case) if do == "scan" else [box.T])]
    if do == "patch":
        h, n = 2 * box.lam, case["plane"]
        xs = [-h + 2 * h * i / n for i in range(n)]
        return _planes(_one_step(box, case, box.T), box, box.T, xs, n, -h, h).real.permute(0, 2, 3, 1).contiguous()
    t = case["steps"] * box.dt()
    F = _one_step(box, case, t)
    n, _, lo, hi, _, _ = _plane(box, case)
    plane = _planes(F, box, t, [_job_x(box, case)], n, lo, hi)[:, 0]
    hat = [math.sqrt(float(sum(F[q].abs() ** 2 for q in qs).max())) for qs in ((0, 1, 2), (3, 4, 5))]
    f = torch.stack([torch.fft.ifftn(v) for v in F])
    e = [float(f[q].abs().square().sum()) for q in range(6)]
    return {"plane": plane.cpu().numpy(), "fields": f, "numbers": [sum(e), sum(e[:3]), sum(e[3:])] + hat}
