"""Performance cases: what a user of this framework has it do, through `aewave.Solver`.

Each case is one call (or the pair of calls a program makes together) on inputs of the
kind the path meets: wave speeds are smooth Gaussian random fields in 1.5-3 km/s, the
observed data come from a model with a +5% bump, sources are 25 Hz Ricker forces at the
grid's centre, receivers lie on the plane k = 1.  Grids, step counts and receiver counts
are those of the repository's configurations, tests and benchmark, plus a ragged grid.

The module also holds a plain torch restatement of the discretisation, used for two
things only: the observed data of `prepare` (FP32) and the values of `exact` (FP64).
"""
import math
import os

import numpy as np
import torch

from paper_2304_04781_gb300 import aewave

H = 10.0            # grid spacing [m]
CMAX = 3000.0       # dt = 0.5 H / CMAX
F0 = 25.0           # Ricker peak frequency [Hz]
DT = 0.5 * H / CMAX
THETA = 6400.0      # prior length scale [m^2], as in the MAP benchmark
SIGMA = 50.0        # source smoothing of the MAP problem [m]
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(aewave.__file__)), "weights")


# ---------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------
def listed():
    return [
        # the smallest solve: seismograms of one shot on the 32^3 grid of the tests
        {"name": "forward_32", "kind": "forward", "nz": 32, "ny": 32, "nx": 32, "nt": 200,
         "nrec": 16},
        # observed data of the largest grid, part of its time axis
        {"name": "forward_512x512x256", "kind": "forward", "nz": 256, "ny": 512, "nx": 512,
         "nt": 240, "nrec": 256},
        # one misfit gradient with every state kept, the 128^3 configuration
        {"name": "gradient_full_128", "kind": "gradient", "storage": "full", "nz": 128, "ny": 128,
         "nx": 128, "nt": 1000, "nrec": 64},
        # one gradient with 20 checkpoint slots on a grid that fills no tile evenly
        {"name": "gradient_revolve_ragged", "kind": "gradient", "storage": "revolve", "nz": 72,
         "ny": 100, "nx": 148, "nt": 500, "nrec": 64},
        # the headline: one gradient with the history compressed by the time codec
        {"name": "gradient_ae_256", "kind": "gradient", "storage": "ae", "nz": 256, "ny": 256,
         "nx": 256, "nt": 2000, "nrec": 128},
        # one Gauss-Newton Hessian-vector product of a Newton or subspace iteration
        {"name": "hessvec_ae_128", "kind": "hessvec", "storage": "ae", "newton": False, "nz": 128,
         "ny": 128, "nx": 128, "nt": 1000, "nrec": 64},
        # a whole MAP solve at a size where a user tries settings out
        {"name": "map_64", "kind": "map", "storage": "full", "nz": 64, "ny": 64, "nx": 64,
         "nt": 400, "nrec": 64, "iters": 2, "cg": 4},
        # one window of 16 strain states to latents and back (the codec alone, FP32 slices)
        {"name": "window_256", "kind": "window", "nz": 256, "ny": 256, "nx": 256, "steps": 16},
        # one state's 8^3 blocks to latents and back to strain, the space codec
        {"name": "state_256", "kind": "state", "nz": 256, "ny": 256, "nx": 256, "nlat": 64},
        # a stretch of codec training at the paper's batch, then the weights taken out
        {"name": "train_time_512", "kind": "train", "codec": "time", "batch": 512, "steps": 32},
        # one sample of the prior (or one application of its covariance's root)
        {"name": "prior_solve_256", "kind": "prior", "nz": 256, "ny": 256, "nx": 256},
        # training data of one draw: every tenth state's blocks (Algorithm 1)
        {"name": "snapshots_128", "kind": "snapshots", "nz": 128, "ny": 128, "nx": 128,
         "nt": 1000, "every": 10},
    ]


def draw(rng):
    def size(lo, hi, unit):
        """A multiple of `unit`, its logarithm spread evenly over lo .. hi."""
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return max(unit, min(int(hi), int(round(v / unit)) * unit))

    def grid(lo, hi, unit):
        return {"nz": size(lo, hi, unit), "ny": size(lo, hi, unit), "nx": size(lo, hi, unit)}

    def steps(g, lo, hi, budget):
        """Step count within `budget` node updates."""
        n = g["nz"] * g["ny"] * g["nx"]
        return max(16, min(size(lo, hi, 1), int(budget // n)))

    kind = rng.choice(["forward", "gradient", "gradient", "gradient", "hessvec", "map", "window",
                       "state", "train", "prior", "snapshots"])
    nrec = rng.choice([16, 64, 128, 256])
    if kind == "forward":
        g = grid(32, 512, 4)
        g["nz"] = min(g["nz"], 256)
        return {"kind": kind, **g, "nt": steps(g, 100, 1000, 1.6e10), "nrec": nrec}
    if kind in ("gradient", "hessvec"):
        storage = rng.choice(["full", "revolve", "ae"])
        g = grid(32, 256, 8 if storage == "ae" else 4)
        c = {"kind": kind, "storage": storage, **g, "nt": steps(g, 100, 1500, 3.0e9), "nrec": nrec}
        if kind == "hessvec":
            c["newton"] = storage != "revolve" and rng.random() < 0.25
        return c
    if kind == "map":
        g = grid(48, 96, 8)
        return {"kind": kind, "storage": rng.choice(["full", "ae"]), **g,
                "nt": steps(g, 250, 500, 4e8), "nrec": 64, "iters": 2, "cg": rng.choice([2, 3, 4])}
    if kind == "window":
        return {"kind": kind, **grid(32, 256, 8), "steps": rng.choice([16, 16, rng.randint(1, 15)])}
    if kind == "state":
        return {"kind": kind, **grid(32, 256, 8), "nlat": rng.choice([32, 64])}
    if kind == "train":
        return {"kind": kind, "codec": rng.choice(["time", "space"]), "batch": size(64, 512, 8),
                "steps": rng.randint(8, 32)}
    if kind == "prior":
        return {"kind": kind, **grid(32, 256, 4)}
    g = grid(32, 128, 8)
    return {"kind": kind, **g, "nt": steps(g, 200, 1000, 2.1e9), "every": rng.randint(8, 25)}


def shape_of(case):
    return (case["nz"], case["ny"], case["nx"])


def work(case):
    """Bytes: inputs once, outputs once, and for the gradient and Hessian calls the
    history that the storage mode keeps (strain fields, or latents) once each way.
    Operations: 17 per node of a forward step, 20 of an adjoint step, the codec's
    products, the prior operator's and its solver's 30 per node and iteration."""
    k = case["kind"]
    if k == "train":
        nh, nl = (1024, 512) if case["codec"] == "time" else (512, 64)
        p = 2 * (2048 * nh + nh * nl) + 2 * nh + nl + 2048
        b = case["batch"] * case["steps"]
        # two copies of the weights' bytes in, two out: the weights and two moments
        return {"bytes": b * 2048 * 2 + 24.0 * p,
                "flops": 2.0 * b * (2 * (2048 * nh + nh * nl) * 3 - 2048 * nh)}
    n = float(case["nz"] * case["ny"] * case["nx"])
    if k == "window":
        vec = n / 128
        return {"bytes": (case["steps"] + 16) * n * 4 + vec * (512 * 2 + 4),
                "flops": vec * 2 * 2.0 * (2048 * 1024 + 1024 * 512)}
    if k == "state":
        b, nl = n / 512, case["nlat"]
        return {"bytes": 20 * n + b * (nl * 2 + 16),
                "flops": b * 2.0 * (2048 * 512 + 512 * nl + nl * 512 + 512 * 512)}
    if k == "prior":
        return {"bytes": 8 * n, "flops": 30 * n * 160}
    nt = case["nt"]
    if k == "snapshots":
        got = (nt - 1) // case["every"]
        return {"bytes": 4 * n + got * n * 8, "flops": 17 * n * nt}
    d = 12.0 * (nt + 1) * case["nrec"]
    if k == "forward":
        return {"bytes": 4 * n + d, "flops": 17 * n * nt}
    ae = case.get("storage") == "ae"
    hist = {"full": 8 * n * nt, "revolve": 0.0, "ae": 2 * 0.5 * n * nt}[case["storage"]]
    codec = 5.24e6 * n / 128 * nt / 16 if ae else 0.0   # one pass of encoder or decoder
    if k == "gradient":
        return {"bytes": 8 * n + d + hist, "flops": 37 * n * nt + 2 * codec}
    if k == "hessvec":
        adj = 2 if case["newton"] else 1
        return {"bytes": 8 * n + hist * adj, "flops": (20 + 20 * adj) * n * nt + 2 * adj * codec}
    solves = case["iters"] + 1                          # gradients of a MAP solve
    hv = case["iters"] * case["cg"]
    return {"bytes": (solves + hv) * hist + 12 * n + d,
            "flops": (solves * 37 + hv * 40) * n * nt + 2 * (solves + hv) * codec}


# ---------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------
def generator(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + what * 7919 + 17) & 0x7FFFFFFF)
    return g


def smooth_field(shape, corr, gen):
    """A Gaussian random field of correlation length `corr` [m], mean 0, variance 1."""
    w = torch.randn(shape, device="cuda", generator=gen)
    nz, ny, nx = shape
    kz, ky, kx = (2 * math.pi * f for f in (torch.fft.fftfreq(nz, d=H, device="cuda"),
                                            torch.fft.fftfreq(ny, d=H, device="cuda"),
                                            torch.fft.rfftfreq(nx, d=H, device="cuda")))
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
    z = torch.fft.irfftn(torch.fft.rfftn(w) * torch.exp(-k2 * corr * corr / 4), s=shape)
    z = z - z.mean()
    return z / z.std()


def speed_model(shape, seed):
    return (1500.0 + 1500.0 * torch.special.ndtr(smooth_field(shape, 80.0, generator(seed, 1)))).contiguous()


def bump_model(c):
    nz, ny, nx = c.shape
    ax = [torch.arange(s, device="cuda", dtype=torch.float32) for s in c.shape]
    r2 = ((ax[0] - nz / 4)[:, None, None] ** 2 + (ax[1] - ny / 2)[None, :, None] ** 2
          + (ax[2] - nx / 2)[None, None, :] ** 2)
    return c * (1.0 + 0.05 * torch.exp(-r2 / (2.0 * (nz / 8.0) ** 2)))


def direction(shape, seed):
    z = smooth_field(shape, 80.0, generator(seed, 2))
    return (z / z.abs().max()).contiguous()


def receivers(case):
    nx, ny, n = case["nx"], case["ny"], case.get("nrec", 16)
    rx, ry = {16: (4, 4), 64: (8, 8), 128: (16, 8), 256: (16, 16)}[n]
    out = np.zeros((n, 3), dtype=np.int32)
    for r in range(n):
        i, j = int((r % rx + 0.5) * nx / rx + 0.5), int((r // rx + 0.5) * ny / ry + 0.5)
        out[r] = (min(max(i, 1), nx - 2), min(max(j, 1), ny - 2), 1)
    return out


_loaded = {}


def committed_weights(name):
    if name not in _loaded:
        with np.load(os.path.join(WEIGHTS, name)) as z:
            _loaded[name] = {k: z[k] for k in ("W1", "b1", "W2", "b2", "W3", "b3", "W4", "b4")}
    return _loaded[name]


def glorot_weights(nh, nl, seed):
    g = generator(seed, 3)
    out = {}
    for i, (a, b) in enumerate(((2048, nh), (nh, nl), (nl, nh), (nh, 2048))):
        lim = math.sqrt(6.0 / (a + b))
        out["W%d" % (i + 1)] = ((torch.rand((a, b), device="cuda", generator=g) * 2 - 1) * lim).cpu().numpy()
        out["b%d" % (i + 1)] = np.zeros(b, np.float32)
    return out


def strain_window(shape, steps, seed):
    """`steps` consecutive strain states: six plane waves of the source's band under a smooth
    envelope that is 0 ahead of the wavefront."""
    g = generator(seed, 4)
    nz, ny, nx = shape
    env = torch.clamp(smooth_field(shape, 160.0, g) + 0.3, min=0.0)
    ax = [torch.arange(s, device="cuda", dtype=torch.float32) * H for s in shape]
    par = torch.rand((6, 5), generator=g, device="cuda").cpu().numpy()
    out = torch.zeros((steps, nz, ny, nx), device="cuda")
    for a, b, f, p, q in par:
        om = 2 * math.pi * F0 * (0.5 + f)
        k = om / (1800.0 + 900.0 * q)
        th, ph = math.acos(2 * a - 1), 2 * math.pi * b
        arg = (k * math.cos(th) * ax[0])[:, None, None] + (k * math.sin(th) * math.sin(ph) * ax[1])[None, :, None] \
            + (k * math.sin(th) * math.cos(ph) * ax[2])[None, None, :]
        for t in range(steps):
            out[t] += torch.cos(arg + (2 * math.pi * p - om * DT * t))
    out *= env
    out *= 1e-9      # the amplitude of the solver's strain for a unit force
    out[:, 0], out[:, -1], out[:, :, 0], out[:, :, -1] = 0, 0, 0, 0
    out[..., 0], out[..., -1] = 0, 0
    return out


def state_fields(shape, seed):
    return [(s * smooth_field(shape, 40.0, generator(seed, 10 + f))).contiguous()
            for f, s in enumerate((1.0, 2e-3, 5e-3, 1e-2))]


def training_vectors(n, seed):
    """n normalised window vectors in random order (BF16)."""
    v = window_vectors(strain_window((128, 128, 128), 16, seed))
    order = torch.randperm(v.shape[0], generator=generator(seed, 5), device="cuda")[:n]
    v = v[order]
    return over(v, pow2_scale(v.abs().amax(1))[:, None]).to(torch.bfloat16).contiguous()


def solver(case, storage, **kw):
    return aewave.Solver(shape_of(case), H, case.get("nt", 16), receivers(case), storage=storage, **kw)


def prepare(case, seed):
    k, s = case["kind"], {}
    if k == "train":
        nh, nl = (1024, 512) if case["codec"] == "time" else (512, 64)
        s["solver"] = aewave.Solver((32, 32, 32), H, 16, np.zeros((0, 3), np.int32), storage="revolve",
                                    n_checkpoints=0, codec=case["codec"])
        s["solver"].codec_set(glorot_weights(nh, nl, seed))
        s["batches"] = list(training_vectors(case["batch"] * case["steps"], seed).split(case["batch"]))
        return {"case": case, **s}
    shape = shape_of(case)
    if k == "window":
        s["solver"] = solver(case, "revolve", n_checkpoints=0, codec="time")
        s["solver"].codec_set(committed_weights("codec_time_512.npz"))
        s["e"] = strain_window(shape, case["steps"], seed)
    elif k == "state":
        s["solver"] = solver(case, "revolve", n_checkpoints=0, n_lat=case["nlat"])
        s["solver"].codec_set(committed_weights("codec_%d.npz" % case["nlat"]))
        s["fields"] = state_fields(shape, seed)
    elif k == "prior":
        s["solver"] = solver(case, "revolve", n_checkpoints=0)
        s["w"] = torch.randn(shape, device="cuda", generator=generator(seed, 6))
    elif k in ("forward", "snapshots"):
        s["solver"] = solver(case, "revolve", n_checkpoints=0)
        s["c"] = speed_model(shape, seed)
        s["vectors"] = s["solver"].nblocks * ((case["nt"] - 1) // case.get("every", 1))
    else:
        kw = {"ae": {"codec": "time"}, "full": {}, "revolve": {"n_checkpoints": 20}}[case["storage"]]
        sigma = SIGMA if k == "map" else 0.0
        s["c"] = speed_model(shape, seed)
        s["d_obs"] = Wave(case, bump_model(s["c"]), torch.float32, sigma).forward()[0]
        s["solver"] = solver(case, case["storage"], src_sigma=sigma, **kw)
        if case["storage"] == "ae":
            s["solver"].codec_set(committed_weights("codec_time_512.npz"))
        if k == "hessvec":
            s["dc"] = direction(shape, seed)
            s["solver"].gradient(s["c"], s["d_obs"])
        if k == "map":
            s["alpha"] = map_alpha(shape, s["d_obs"])
    return {"case": case, **s}


def map_alpha(shape, d_obs):
    """The regularisation's weight: noise of 1% of the data's rms, prior samples of 30 m/s."""
    noise = 0.01 * float(d_obs[1:].double().pow(2).mean().sqrt())
    return noise * float((prior_symbol(shape, 1.0) ** -2).mean().sqrt()) / 30.0


# ---------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------
def run(state):
    case, s = state["case"], state["solver"]
    k = case["kind"]
    if k == "forward":
        return s.forward(state["c"])
    if k == "gradient":
        J, g = s.gradient(state["c"], state["d_obs"])
        return {"J": np.float32(J), "g": g}     # the misfit of FP32 seismograms
    if k == "hessvec":
        return s.hessvec_full(state["dc"]) if case["newton"] else s.hessvec(state["dc"])
    if k == "map":
        c = state["c"].clone()
        hist = s.newton_cg(c, state["d_obs"], state["c"], state["alpha"], THETA,
                           newton_iters=case["iters"], cg_max=case["cg"])
        return {"c": c, "cost": np.array([h["cost"] for h in hist], np.float32),
                "cg": np.array([h["cg_iters"] for h in hist], np.int64)}
    if k == "window":
        lat, scale = s.codec_encode_window(state["e"])
        return {"lat": lat, "scale": scale, "e": s.codec_decode_window(lat, scale)}
    if k == "state":
        lat, bmax = s.codec_encode(state["fields"])
        return {"lat": lat, "bmax": bmax, "e": s.codec_decode_e(lat, bmax)}
    if k == "train":
        last = len(state["batches"]) - 1
        loss = None
        for i, b in enumerate(state["batches"]):
            loss = s.train_step(b, 1e-3, want_loss=i == last)
        return {"loss": np.float32(loss), "W": s.codec_get()}
    if k == "prior":
        x, its = s.prior_solve(state["w"], 1.0, THETA)
        return {"x": x, "its": its}
    v, m = s.snapshots(state["c"], case["every"], state["vectors"], with_scales=True)
    return {"vectors": v, "maxima": m}


# ---------------------------------------------------------------------------------
# the discretisation in plain torch
# ---------------------------------------------------------------------------------
class Wave:
    """The velocity-strain leapfrog scheme, its adjoint and its linearisation."""

    def __init__(self, case, c, dtype, sigma=0.0):
        self.shape, self.nt, self.dtype = tuple(c.shape), case["nt"], dtype
        self.c = c.to(dtype)
        self.m = self.c * self.c
        self.dth = DT / H
        nz, ny, nx = self.shape
        rec = receivers(case).astype(np.int64)
        self.rec = torch.from_numpy((rec[:, 2] * ny + rec[:, 1]) * nx + rec[:, 0]).cuda()
        t = np.arange(self.nt) * DT - 1.0 / F0
        sig = 1.0 / (math.sqrt(2.0) * math.pi * F0)
        self.wav = -(1.0 - t * t / sig ** 2) * np.exp(-t * t / (2 * sig ** 2))
        r = int(math.ceil(3.0 * sigma / H)) if sigma > 0 else 0
        o = torch.arange(-r, r + 1, device="cuda", dtype=torch.float64) * H
        r2 = o[:, None, None] ** 2 + o[None, :, None] ** 2 + o[None, None, :] ** 2
        w = torch.exp(-r2 / (2 * sigma * sigma)) if r else torch.ones_like(r2)
        self.src_w = (w / w.sum()).to(dtype)
        self.src = tuple(slice(n // 2 - r, n // 2 + r + 1) for n in self.shape)
        self.t = self.zeros()

    def zeros(self):
        return torch.zeros(self.shape, device="cuda", dtype=self.dtype)

    def faces(self, f, v, sign):
        """v += sign dt/h G f on the used faces."""
        for a in range(3):
            n = self.shape[a]
            d = torch.sub(f.narrow(a, 1, n - 1), f.narrow(a, 0, n - 1), out=self.t.narrow(a, 0, n - 1))
            v[a].narrow(a, 0, n - 1).add_(d, alpha=sign * self.dth)

    def div(self, v):
        """dt/h div v on interior nodes (a view of the work buffer)."""
        nz, ny, nx = self.shape
        i = (slice(1, -1),) * 3
        o = self.t[i]
        torch.sub(v[0][i], v[0][:-2, 1:-1, 1:-1], out=o)
        o.add_(v[1][i]).sub_(v[1][1:-1, :-2, 1:-1]).add_(v[2][i]).sub_(v[2][1:-1, 1:-1, :-2])
        return o.mul_(self.dth)

    def record(self, v, row):
        for a in range(3):   # components x, y, z
            row[:, a] = v[2 - a].reshape(-1)[self.rec]

    def solve(self, source, extra, keep):
        """(receiver rows, strain history): `source` adds the force, `extra(n)` is added to m e."""
        e, v, me = self.zeros(), [self.zeros() for _ in range(3)], self.zeros()
        d = torch.zeros((self.nt + 1, self.rec.numel(), 3), device="cuda", dtype=self.dtype)
        hist = []
        i = (slice(1, -1),) * 3
        for n in range(self.nt):
            if keep:
                hist.append(e.clone())
            torch.mul(self.m, e, out=me)
            if extra is not None:
                me += extra(n)
            self.faces(me, v, 1.0)
            if source:
                v[0][self.src].add_(self.src_w, alpha=DT * float(self.wav[n]))
            e[i] += self.div(v)
            self.record(v, d[n + 1])
        return d, hist

    def forward(self, keep=False):
        return self.solve(True, None, keep)

    def jvp(self, dm, hist, keep=False):
        return self.solve(False, lambda n: dm * hist[n], keep)

    def adjoint(self, resid, hist, keep=False, extra=None):
        """(dJ/dm, [dt q^n]) for a receiver residual; `extra(n)` is added in the mu update."""
        mu, lam, acc = self.zeros(), [self.zeros() for _ in range(3)], self.zeros()
        qs = [None] * self.nt
        i = (slice(1, -1),) * 3
        for n in range(self.nt - 1, -1, -1):
            for a in range(3):
                lam[2 - a].view(-1).index_add_(0, self.rec, resid[n + 1, :, a])
            self.faces(mu, lam, -1.0)
            q = self.div(lam).neg_()
            acc[i] += hist[n][i] * q
            mu[i] += self.m[i] * q
            if extra is not None:
                mu[i] += extra(n)[i]
            if keep:
                qs[n] = self.zeros()
                qs[n][i] = q
        return acc, qs

    def gradient(self, d_obs, hist=None):
        """(J, dJ/dc, residual, strain history); `hist` maps the stored history to the one read."""
        d, e = self.forward(keep=True)
        r = d - d_obs
        r[0] = 0
        e = hist(e) if hist else e
        return 0.5 * (r * r).sum(), 2 * self.c * self.adjoint(r, e)[0], r, e

    def hessvec(self, dc, e):
        dd, _ = self.jvp(2 * self.c * dc, e)
        return 2 * self.c * self.adjoint(dd, e)[0]

    def hessvec_full(self, dc, r, e, hist=None):
        dm = 2 * self.c * dc
        dd, de = self.jvp(dm, e, keep=True)
        de = hist(de) if hist else de
        a, q = self.adjoint(r, de, keep=True)
        b, _ = self.adjoint(dd, e, extra=lambda n: dm * q[n])
        g = sum(e[n] * q[n] for n in range(self.nt))
        return 2 * self.c * (a + b) + 2 * dc * g


def pow2_scale(mx):
    """2^max(e, -100) for mx = f 2^e with f in [0.5, 1); 0 for mx = 0."""
    s = torch.pow(2.0, torch.clamp(torch.frexp(mx)[1], min=-100).to(mx.dtype))
    return torch.where(mx > 0, s, torch.zeros_like(s))


def over(x, s):
    """x / s, and 0 where the scale is 0."""
    return x / torch.where(s > 0, s, torch.ones_like(s))


def window_vectors(e):
    """[16][nz][ny][nx] -> [vectors][2048], the order t, z, y, x over 2 x 8 x 8-node blocks."""
    t, nz, ny, nx = e.shape
    return e.reshape(t, nz // 2, 2, ny // 8, 8, nx // 8, 8).permute(1, 3, 5, 0, 2, 4, 6).reshape(-1, t * 128)


def window_fields(v, shape):
    nz, ny, nx = shape
    e = v.reshape(nz // 2, ny // 8, nx // 8, 16, 2, 8, 8).permute(3, 0, 4, 1, 5, 2, 6)
    return inside(e.reshape(16, nz, ny, nx))


def inside(e):
    """A copy with boundary nodes 0."""
    out = torch.zeros_like(e)
    out[..., 1:-1, 1:-1, 1:-1] = e[..., 1:-1, 1:-1, 1:-1]
    return out


def gelu(a):
    return torch.nn.functional.gelu(a)


def doubles(W):
    return {k: torch.from_numpy(np.asarray(v)).cuda().double() for k, v in W.items()}


def rows(f, x, n=16384):
    return torch.cat([f(p) for p in x.split(n)])


def code_window(W, e):
    """(latents, maxima, decoded fields) of one window of FP64 strain states."""
    shape = tuple(e.shape[1:])
    if e.shape[0] < 16:
        e = torch.cat([e, torch.zeros((16 - e.shape[0],) + shape, device="cuda", dtype=e.dtype)])
    x = window_vectors(e)
    mx = x.abs().amax(1)
    s = pow2_scale(mx)[:, None]
    z = rows(lambda y: gelu(y @ W["W1"] + W["b1"]) @ W["W2"] + W["b2"], over(x, s))
    out = rows(lambda y: gelu(y @ W["W3"] + W["b3"]) @ W["W4"] + W["b4"], z) * s
    return z, mx, window_fields(out, shape)


def coded_history(W):
    """The time codec applied to a strain history (e^0 stays 0)."""
    def of(hist):
        out = []
        for w in range(0, len(hist), 16):
            out += list(code_window(W, torch.stack(hist[w:w + 16]))[2][: len(hist) - w])
        out[0] = torch.zeros_like(out[0])
        return out
    return of


def block_vectors(fields):
    """4 x [nz][ny][nx] -> ([blocks][2048] normalised, maxima [blocks][4]), order z, field, y, x."""
    f = torch.stack(fields)
    _, nz, ny, nx = f.shape
    x = f.reshape(4, nz // 8, 8, ny // 8, 8, nx // 8, 8).permute(1, 3, 5, 2, 0, 4, 6).reshape(-1, 8, 4, 64)
    mx = x.abs().amax((1, 3))
    return over(x, pow2_scale(mx)[:, None, :, None]).reshape(-1, 2048), mx


def prior_symbol(shape, alpha):
    """Eigenvalues of A q = alpha (q - theta Lap q) on the cosine modes."""
    lam = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for a, n in enumerate(shape):
        s = (4.0 / (H * H)) * torch.sin(math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / (2 * n)) ** 2
        lam += s.reshape([n if b == a else 1 for b in range(3)])
    return alpha * (1.0 + THETA * lam)


def cosine_modes(n):
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    m = torch.cos(math.pi * i[:, None] * (i[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
    m[0] /= math.sqrt(2.0)
    return m


def prior_solution(w):
    """A^{-1} w in the cosine basis."""
    Cz, Cy, Cx = (cosine_modes(n) for n in w.shape)
    x = torch.einsum("ab,bjk->ajk", Cz, w)
    x = torch.einsum("ab,ibk->iak", Cy, x) @ Cx.T
    x = x / prior_symbol(w.shape, 1.0)
    x = torch.einsum("ba,bjk->ajk", Cz, x @ Cx)
    return torch.einsum("ba,ibk->iak", Cy, x)


def prior_apply(q, alpha):
    lap = torch.zeros_like(q)
    for a, n in enumerate(q.shape):
        d = q.narrow(a, 1, n - 1) - q.narrow(a, 0, n - 1)
        lap.narrow(a, 0, n - 1).add_(d)
        lap.narrow(a, 1, n - 1).sub_(d)
    return alpha * (q - THETA / (H * H) * lap)


def newton(case, c0, d_obs, alpha, hist):
    """Inexact Newton-CG with Armijo backtracking, as aew_newton_cg documents it."""
    dot = lambda a, b: float((a * b).sum())  # noqa: E731

    def at(c):
        w = Wave(case, c, torch.float64, SIGMA)
        J, g, _, e = w.gradient(d_obs, hist)
        return w, float(J), g, e

    c, out, its, g0 = c0.clone(), [], [], None
    w, Jm, gm, e = at(c)
    for _ in range(case["iters"]):
        a = prior_apply(c - c0, alpha)
        J, g = Jm + 0.5 * dot(a, a), gm + prior_apply(a, alpha)
        gn = math.sqrt(dot(g, g))
        g0 = gn if g0 is None else g0
        eta = min(0.5, math.sqrt(gn / g0))
        x, r = torch.zeros_like(c), -g
        p, rr, k = r.clone(), gn * gn, 0
        for k in range(1, case["cg"] + 1):
            Hp = w.hessvec(p, e) + prior_apply(prior_apply(p, alpha), alpha)
            pHp = dot(p, Hp)
            if not pHp > 0:
                k -= 1
                break
            x, r = x + rr / pHp * p, r - rr / pHp * Hp
            rn = dot(r, r)
            if math.sqrt(rn) <= eta * gn:
                break
            p, rr = r + rn / rr * p, rn
        x = -g if k == 0 else x
        slope, step = dot(g, x), 1.0
        out.append(J)
        its.append(k)
        for _ in range(10):
            ct = c + step * x
            if float(ct.min()) > 0 and float(ct.max()) * DT / H <= 1 / math.sqrt(3.0):
                got = at(ct)
                a = prior_apply(ct - c0, alpha)
                if got[1] + 0.5 * dot(a, a) <= J + 1e-4 * step * slope:
                    break
            step *= 0.5
        else:
            break
        c, (w, Jm, gm, e) = ct, got
    return {"c": c, "cost": torch.tensor(out, dtype=torch.float64), "cg": None}


def lamb_steps(W, batches):
    """LAMB on the mean squared error, the FP16 latent passed straight through."""
    names = ("W1", "b1", "W2", "b2", "W3", "b3", "W4", "b4")
    W = {k: v.requires_grad_(True) for k, v in doubles(W).items()}
    m = {k: torch.zeros_like(W[k]) for k in names}
    v = {k: torch.zeros_like(W[k]) for k in names}
    loss = None
    for t, y in enumerate(batches, 1):
        y = y.double()
        z = gelu(y @ W["W1"] + W["b1"]) @ W["W2"] + W["b2"]
        loss = ((gelu(z @ W["W3"] + W["b3"]) @ W["W4"] + W["b4"] - y) ** 2).mean()
        for k, g in zip(names, torch.autograd.grad(loss, [W[k] for k in names])):
            m[k] = 0.9 * m[k] + 0.1 * g
            v[k] = 0.999 * v[k] + 0.001 * g * g
            u = (m[k] / (1 - 0.9 ** t)) / ((v[k] / (1 - 0.999 ** t)).sqrt() + 1e-6)
            with torch.no_grad():
                wn, un = W[k].norm(), u.norm()
                W[k] -= 1e-3 * (wn / un if wn > 0 and un > 0 else 1.0) * u
    return {"loss": loss.detach(), "W": {k: W[k].detach() for k in names}}


def exact(case, seed):
    k = case["kind"]
    if k == "train":
        nh, nl = (1024, 512) if case["codec"] == "time" else (512, 64)
        return lamb_steps(glorot_weights(nh, nl, seed),
                          training_vectors(case["batch"] * case["steps"], seed).split(case["batch"]))
    shape = shape_of(case)
    nodes = case["nz"] * case["ny"] * case["nx"]
    if k == "window":
        e = strain_window(shape, case["steps"], seed).double()
        z, mx, out = code_window(doubles(committed_weights("codec_time_512.npz")), e)
        return {"lat": z, "scale": mx, "e": out}
    if k == "state":
        W = doubles(committed_weights("codec_%d.npz" % case["nlat"]))
        y, mx = block_vectors([f.double() for f in state_fields(shape, seed)])
        z = rows(lambda p: gelu(p @ W["W1"] + W["b1"]) @ W["W2"] + W["b2"], y)
        x = rows(lambda p: gelu(p @ W["W3"] + W["b3"]) @ W["W4"] + W["b4"], z)
        x = x.reshape(-1, 8, 4, 8, 8)[:, :, 0] * pow2_scale(mx[:, 0])[:, None, None, None]
        nz, ny, nx = shape
        x = x.reshape(nz // 8, ny // 8, nx // 8, 8, 8, 8).permute(0, 3, 1, 4, 2, 5).reshape(shape)
        return {"lat": z, "bmax": mx, "e": inside(x)}
    if k == "prior":
        w = torch.randn(shape, device="cuda", generator=generator(seed, 6))
        return {"x": prior_solution(w.double()), "its": None}
    c = speed_model(shape, seed)
    if k == "forward":
        if nodes * case["nt"] > 2.5e10:
            return None
        return Wave(case, c, torch.float64).forward()[0]
    if k == "snapshots":
        w, out = Wave(dict(case, nrec=16), c, torch.float64), []
        e, v, me = w.zeros(), [w.zeros() for _ in range(3)], w.zeros()
        for n in range(case["nt"]):
            if n and n % case["every"] == 0:
                out.append(block_vectors([e, v[2], v[1], v[0]]))
            torch.mul(w.m, e, out=me)
            w.faces(me, v, 1.0)
            v[0][w.src].add_(w.src_w, alpha=DT * float(w.wav[n]))
            e[1:-1, 1:-1, 1:-1] += w.div(v)
        return {"vectors": torch.cat([o[0] for o in out]), "maxima": torch.cat([o[1] for o in out])}
    # gradients and Hessian products read the whole history: FP64 within memory and time
    if nodes * case["nt"] > 3.1e9:
        return None
    sigma = SIGMA if k == "map" else 0.0
    d_obs = Wave(case, bump_model(c), torch.float32, sigma).forward()[0]
    hist = None
    if case["storage"] == "ae":
        hist = coded_history(doubles(committed_weights("codec_time_512.npz")))
    if k == "map":
        return newton(case, c.double(), d_obs.double(), map_alpha(shape, d_obs), hist)
    w = Wave(case, c, torch.float64)
    J, g, r, e = w.gradient(d_obs.double(), hist)
    if k == "gradient":
        return {"J": J, "g": g}
    dc = direction(shape, seed).double()
    return w.hessvec_full(dc, r, e, hist) if case["newton"] else w.hessvec(dc, e)
