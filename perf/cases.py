"""What the framework is timed on: its operators, through the calls a user's program makes.

Each case is one call (or one training step) of the public API on a workload of the kinds that the
repository's five configurations, its tests and its benchmark describe: 2D and 3D grids, single shots
and shot batches, one trial and many, every checkpoint storage type.  Long recordings are shortened in
time only (a pass costs the same per time step); the wave fields are developed all the same, because
the source peaks after a fifth of the recording or earlier.

Inputs are generated here from the seed alone, on the GPU, by plain torch.
"""
import math

import numpy as np
import torch

from paper_1101_3615_gb300 import Basis, Probe, apply_H_group, misfit

SNAPS = ("fp32", "fp16", "bf16")


def listed():
    return [
        # one shot, a few perturbations, a grid with no round size: the smallest modelling call (a
        # unit test, an interactive session); bounded by launches and latency
        dict(name="fwd2d_tiny", op="F", n="57x83", h=10.0, dt=1e-3, nt=200, pad=10, f0=25.0, ns=1, nb=3, snap="fp32"),
        # configuration 1 at full size: H on a 101 x 101 model, four shots, nt = 800
        dict(name="h2d_small", op="H", n="101x101", h=10.0, dt=1e-3, nt=800, pad=20, f0=15.0, ns=4, nb=1, snap="fp32"),
        # Krylov trial functions: a chain of H applications of one trial each, as in iterative inversion
        dict(name="krylov2d", op="krylov", n="201x241", h=8.0, dt=8e-4, nt=400, pad=20, f0=15.0, ns=6, nb=1,
             snap="fp32", iters=4),
        # migration of recorded data: F* on a ragged grid, two data sets, BF16 checkpoints
        dict(name="fadj2d_ragged", op="Fadj", n="243x389", h=8.0, dt=8e-4, nt=700, pad=17, f0=15.0, ns=12, nb=2,
             snap="bf16"),
        # configuration 2: H over 32 shots of a 501 x 501 model, one reference perturbation, FP16
        # checkpoints as in the benchmark
        dict(name="h2d_shots", op="H", n="501x501", h=8.0, dt=8e-4, nt=1000, pad=20, f0=12.0, ns=32, nb=1, snap="fp16"),
        # configuration 3: three models of different size probed together, several trials each
        dict(name="h2d_group", op="group", n="301x301,501x501,701x701", h=8.0, dt=8e-4, nt=400, pad=20, f0=15.0, ns=8,
             nb=4, snap="fp16"),
        # configuration 4: one training step, misfit and gradient through autograd on 1001 x 1001
        dict(name="grad2d", op="grad", n="1001x1001", h=5.0, dt=5e-4, nt=800, pad=20, f0=15.0, ns=8, nb=1, snap="fp16"),
        # 3D modelling of a batch of perturbations on a mid-sized cube
        dict(name="fwd3d_mid", op="F", n="128x128x128", h=10.0, dt=8e-4, nt=160, pad=20, f0=30.0, ns=4, nb=2,
             snap="fp32"),
        # H on a ragged 3D box with the default FP32 checkpoints, one trial
        dict(name="h3d_ragged", op="H", n="90x75x115", h=10.0, dt=8e-4, nt=240, pad=13, f0=25.0, ns=3, nb=1,
             snap="fp32"),
        # configuration 5, the benchmark's default: 256^3, BF16 checkpoints, four trials per call,
        # half of its shots
        dict(name="h3d_main", op="H", n="256x256x256", h=10.0, dt=8e-4, nt=60, pad=20, f0=40.0, ns=8, nb=4,
             snap="bf16"),
        # the randomized fit of the inverse on 3D pairs (60 terms, four pairs) ...
        dict(name="fit3d", op="fit", n="128x128x128", h=10.0, p=4, nspatial=5, nangular=3, nradial=4),
        # ... and the fitted preconditioner applied to a full-size image
        dict(name="precond3d", op="precond", n="256x256x256", h=10.0, p=1, nspatial=5, nangular=3, nradial=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["F", "F", "H", "H", "H", "Fadj", "grad", "group", "krylov", "fit", "precond"])
    nd = 3 if (op in ("F", "H", "Fadj", "fit", "precond") and rng.random() < 0.45) else 2
    if op in ("fit", "precond"):
        n = [_log(rng, 24, 200) for _ in range(3)] if nd == 3 else [_log(rng, 64, 1000) for _ in range(2)]
        case = dict(op=op, n=n, h=rng.choice([5.0, 8.0, 10.0]), p=rng.randint(1, 6) if op == "fit" else 1,
                    nspatial=rng.randint(1, 5), nangular=rng.randint(1, 4), nradial=rng.randint(1, 5))
        P = case["nspatial"] * case["nangular"] * case["nradial"]
        while op == "fit" and case["p"] * math.prod(n) * P * P > 3e10:  # the listed fit's Gram matrix
            n = case["n"] = [max(24, v * 4 // 5) for v in n]
            case["p"] = max(1, case["p"] - 1)
        if op == "fit" and case["p"] % 2 and all(v % 2 for v in n):
            case["p"] += 1  # 64-bit transforms of an odd number of values are not accepted
        return dict(case, n="x".join(map(str, n)))
    snap = rng.choice(SNAPS)
    pad = rng.randint(8, 24)
    if nd == 3:
        n = [_log(rng, 24, 200) for _ in range(3)]
        ns, nb, nt = _log(rng, 1, 9), rng.randint(1, 5), _log(rng, 60, 300)
    else:
        n = [_log(rng, 48, 1000) for _ in range(2)]
        ns, nb, nt = _log(rng, 1, 40), rng.randint(1, 9), _log(rng, 150, 1200)
    if op in ("grad", "krylov"):
        nb = 1

    def updates():
        return math.prod(x + 2 * pad for x in n) * ns * nt * (2 + 2 * nb) * {"group": 2, "krylov": 4}.get(op, 1)

    while updates() > 3e10:  # a quarter of the largest listed case's
        if ns > 1:
            ns = max(1, ns // 2)
        elif nt > 60:
            nt //= 2
        else:
            n = [max(16, x * 4 // 5) for x in n]
    names = "x".join(map(str, n))
    if op == "group":
        names += "," + "x".join(str(max(40, x * 3 // 4)) for x in n)
        if rng.random() < 0.5:
            names += "," + "x".join(str(max(33, x // 2 + 1)) for x in n)
    f0 = max(10.0, 2.5 / (nt * 8e-4))   # the wavelet peaks within the first 40 % of the recording
    case = dict(op=op, n=names, h=8.0 if nd == 2 else 10.0, dt=8e-4, nt=nt, pad=pad, f0=f0, ns=ns, nb=nb, snap=snap)
    if op == "krylov":
        case["iters"] = rng.randint(1, 4)
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["n"].split(",")]


def _gen(seed, k):
    g = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu")
    g.manual_seed(1000003 * (int(seed) % 1000003) + k)
    return g


def _background(shape, h, seed):
    """Flat layers, 1500 to 4500 m/s, smoothed over 80 m in depth: m0 = 1 / c^2 (float32, host)."""
    rng = np.random.default_rng([int(seed), shape[0]])
    depths = np.sort(rng.uniform(0, shape[0], size=12))
    speeds = rng.uniform(1500.0, 4500.0, size=13)
    c = speeds[np.searchsorted(depths, np.arange(shape[0]) + 0.5)]
    sig = 80.0 / h
    r = int(math.ceil(4 * sig))
    w = np.exp(-0.5 * (np.arange(-r, r + 1) / sig) ** 2)
    c = np.convolve(np.pad(c, r, mode="edge"), w / w.sum(), mode="valid")
    return np.broadcast_to((1.0 / c**2).reshape((-1,) + (1,) * (len(shape) - 1)), shape).astype(np.float32)


def _band(x, h, lo, hi):
    """Radial band-pass [lo, hi] cycles/m of the trailing axes."""
    dims = tuple(range(1, x.ndim))
    X = torch.fft.rfftn(x, dim=dims)
    nu2 = 0.0
    for i, a in enumerate(dims):
        f = (torch.fft.rfftfreq if a == dims[-1] else torch.fft.fftfreq)(x.shape[a], d=h, device=x.device)
        nu2 = nu2 + (f**2).reshape((-1,) + (1,) * (len(dims) - 1 - i))
    return torch.fft.irfftn(X * ((nu2 >= lo * lo) & (nu2 <= hi * hi)), s=x.shape[1:], dim=dims)


def _trials(shape, h, p, seed, level=1.0):
    """Random-sign band-limited trial functions, tapered over 10 edge cells, of given RMS."""
    g = _gen(seed, 1)
    x = torch.randn((p,) + tuple(shape), generator=g, device=g.device)
    lo, hi = 1.0 / (60.0 * h), 1.0 / (5.0 * h)
    x = _band(torch.sign(_band(x, h, lo, hi)), h, lo, hi)
    for a, n in enumerate(shape):
        m = min(10, n // 2)
        t = torch.ones(n, device=x.device)
        ramp = 0.5 - 0.5 * torch.cos(math.pi * (torch.arange(m, device=x.device) + 0.5) / m)
        t[:m] = ramp
        t[n - m:] = ramp.flip(0)
        x = x * t.reshape((-1,) + (1,) * (len(shape) - 1 - a))
    return (x * (level / x.pow(2).mean().sqrt())).float().contiguous()


def _ricker(nt, dt, f0):
    a = (math.pi * f0 * (np.arange(nt) * dt - 1.0 / f0)) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


def _acquisition(shape, ns):
    """Sources spread over the surface two cells down, receivers at every surface node."""
    n = len(shape)
    if n == 2:
        ix = np.round((np.arange(ns) + 0.5) * (shape[1] - 1) / ns).astype(np.int32)
        src = np.stack([np.full(ns, 2, np.int32), ix], 1)
        rec = np.stack([np.zeros(shape[1], np.int32), np.arange(shape[1], dtype=np.int32)], 1)
        return src, rec
    g = int(math.ceil(math.sqrt(ns)))
    k = np.arange(ns)
    src = np.stack([np.full(ns, 2), (k // g + 0.5) * (shape[1] - 1) / g, (k % g + 0.5) * (shape[2] - 1) / g], 1)
    yy, xx = np.meshgrid(np.arange(shape[1]), np.arange(shape[2]), indexing="ij")
    rec = np.stack([np.zeros(yy.size), yy.ravel(), xx.ravel()], 1)
    return np.round(src).astype(np.int32), rec.astype(np.int32)


def _gathers(case, shape, nb, seed):
    """Shot gathers [nb, ns, nt, nr]: reflections with hyperbolic moveout, random times and signs."""
    src, rec = _acquisition(shape, case["ns"])
    g = _gen(seed, 2)
    dev, h, nt, dt = g.device, case["h"], case["nt"], case["dt"]
    off = torch.tensor(((src[:, None, 1:] - rec[None, :, 1:]) ** 2).sum(-1) * h * h, device=dev, dtype=torch.float32)
    t = (torch.arange(nt, device=dev, dtype=torch.float32) * dt)[None, :, None]
    out = torch.zeros((nb, case["ns"], nt, rec.shape[0]), device=dev)
    for b in range(nb):
        for _ in range(6):
            t0, v, a = (torch.rand(3, generator=g, device=dev) * torch.tensor([0.6, 2500.0, 2.0], device=dev)).tolist()
            arr = torch.sqrt(((0.1 + t0) * nt * dt) ** 2 + off / (1500.0 + v) ** 2)[:, None, :]
            q = (math.pi * case["f0"] * (t - arr)) ** 2
            out[b] += (a - 1.0) * (1.0 - 2.0 * q) * torch.exp(-q)
    return out


def _probe(case, shape, seed):
    m0 = _background(shape, case["h"], seed)
    src, rec = _acquisition(shape, case["ns"])
    return Probe(m0, (case["h"],) * len(shape), case["dt"], case["nt"], case["pad"], src, rec,
                 _ricker(case["nt"], case["dt"], case["f0"]), snapshot_dtype=case["snap"]), m0


def _dm_level(m0):
    return 0.05 * float(m0.mean())


# spatial modes, angular indices of the symbol expansion in the order in which they are taken
_SPATIAL = {2: [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)],
            3: [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, 0, 1)]}
_ANGULAR = {2: [0, 2, -2, 4], 3: [0, 4, 5, 1]}


def _basis_args(case, nd):
    return dict(ndim=nd, spatial=_SPATIAL[nd][:case["nspatial"]], angular=_ANGULAR[nd][:case["nangular"]],
                nradial=case["nradial"], L=2 * math.pi / (15.0 * case["h"]), order=-1.0, fft_pad=16)


def _pairs(case, shape, seed):
    """Trials y and stand-ins for H y: a depth-weighted first-order filter of y plus noise."""
    y = _trials(shape, case["h"], case["p"], seed)
    dims = tuple(range(1, y.ndim))
    k2 = 0.0
    for i, a in enumerate(dims):
        f = (torch.fft.rfftfreq if a == dims[-1] else torch.fft.fftfreq)(y.shape[a], d=case["h"], device=y.device)
        k2 = k2 + (f**2).reshape((-1,) + (1,) * (len(dims) - 1 - i))
    x = torch.fft.irfftn(torch.fft.rfftn(y, dim=dims) * torch.sqrt(k2) * 15.0 * case["h"], s=y.shape[1:], dim=dims)
    z = torch.arange(shape[0], device=y.device).reshape((-1,) + (1,) * (len(shape) - 1)) / shape[0]
    g = _gen(seed, 3)
    x = x * (1.0 + 0.4 * torch.cos(2 * math.pi * z)) + 0.05 * torch.randn(x.shape, generator=g, device=g.device)
    return y, x.float().contiguous()


def _coeffs(case, seed):
    rng = np.random.default_rng([int(seed), 4])
    return rng.standard_normal(case["nspatial"] * case["nangular"] * case["nradial"])


def prepare(case, seed):
    shapes = _shapes(case)
    shape, op = shapes[0], case["op"]
    st = dict(case=case)
    if op in ("fit", "precond"):
        nd = len(shape)
        # a handle of that model (its acquisition plays no part in the fit)
        st["probe"], _ = _probe(dict(case, dt=5e-4, nt=2, pad=4, ns=1, snap="fp32", f0=15.0), shape, seed)
        st["basis"] = Basis(**_basis_args(case, nd))
        if op == "fit":
            st["y"], st["Hy"] = _pairs(case, shape, seed)
        else:
            st["coeffs"], st["img"] = _coeffs(case, seed), _trials(shape, case["h"], 1, seed)[0]
        return st
    st["probes"], st["dms"] = [], []
    for k, s in enumerate(shapes):
        p, m0 = _probe(case, s, seed + 17 * k)
        st["probes"].append(p)
        if op in ("F", "H", "group"):
            st["dms"].append(_trials(s, case["h"], case["nb"], seed + 17 * k, _dm_level(m0)))
        if op in ("Fadj", "grad"):
            st["data"] = _gathers(case, s, case["nb"], seed)
        if op == "grad":
            st["data"] = st["data"][0] * 1e-3
            st["m"] = (torch.tensor(m0, device="cuda") + 0.2 * _trials(s, case["h"], 1, seed, _dm_level(m0))[0]).contiguous()
        if op == "krylov":
            st["rhs"] = _trials(s, case["h"], 1, seed)[0]
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "fit":
        return st["probe"].fit(st["basis"], st["y"], st["Hy"])
    if op == "precond":
        return st["probe"].apply_precond(st["basis"], st["coeffs"], st["img"])
    p = st["probes"][0]
    if op == "F":
        return p.apply_F(st["dms"][0])
    if op == "H":
        return p.apply_H(st["dms"][0])
    if op == "Fadj":
        return p.apply_Fadj(st["data"])
    if op == "group":
        return apply_H_group(st["probes"], st["dms"])
    if op == "krylov":
        return p.krylov_trials(st["rhs"], case["iters"])
    m = st["m"].detach().requires_grad_(True)
    J = misfit(m, st["data"], p)
    (g,) = torch.autograd.grad(J, m)
    return J.detach(), g


def work(case):
    """Time stepping: each executed cell update reads two levels of its field and writes one (12 bytes;
    the working set of most cases exceeds the L2), besides the call's own inputs and outputs; the
    Laplacian is 8 adds and 9 fused multiply-adds in 2D, 12 and 13 in 3D, the update 6 more.  Fit and
    preconditioner: the transforms, and the Gram matrix of the fit, in 64-bit arithmetic."""
    shapes, op = _shapes(case), case["op"]
    if op in ("fit", "precond"):
        n, nd, p = math.prod(shapes[0]), len(shapes[0]), case["p"]
        nf = math.prod(v + 32 for v in shapes[0])
        mult = case["nangular"] * case["nradial"]
        P = mult * case["nspatial"]
        fft = 2.5 * nf * math.log2(nf)
        if op == "fit":
            return {"bytes": 8.0 * p * n + 8.0 * P, "flops": fft * p * (1 + mult) + 2.0 * p * n * P * (P + 1) / 2}
        return {"bytes": 8.0 * n + 8.0 * P, "flops": fft * (1 + case["nspatial"]) + 2.0 * n * case["nspatial"]}
    upd = io = 0.0
    nb, ns, steps = case["nb"], case["ns"], case["nt"] - 1
    for s in shapes:
        cells = math.prod(v + 2 * case["pad"] for v in s)
        sweeps = {"F": 1 + nb, "Fadj": 2 + nb, "H": 2 + 2 * nb, "group": 2 + 2 * nb, "grad": 4,
                  "krylov": 4 * case.get("iters", 0)}[op]
        nr = math.prod(s[1:])
        upd += float(cells) * ns * steps * sweeps
        io += 4.0 * nb * math.prod(s) * {"F": 1, "Fadj": 1, "krylov": 1 + 2 * case.get("iters", 0)}.get(op, 2)
        if op in ("F", "Fadj", "grad"):
            io += 4.0 * nb * ns * case["nt"] * nr
    nd = len(shapes[0])
    return {"bytes": 12.0 * upd + io, "flops": upd * (32.0 if nd == 2 else 44.0)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------
class _Wave:
    """The discrete scheme in FP64: 2nd order in time, 8th order in space, quadratic sponge."""

    W = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)

    def __init__(self, case, shape, seed, m=None):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        m0 = _background(shape, case["h"], seed)
        self.nd, self.h, self.dt, self.nt, self.pad = len(shape), case["h"], case["dt"], case["nt"], case["pad"]
        self.src, self.rec = (torch.tensor(a + self.pad, device=dev, dtype=torch.long) for a in _acquisition(shape, case["ns"]))
        self.w = _ricker(case["nt"], case["dt"], case["f0"]).astype(np.float64)
        mp = torch.tensor(np.pad(m0.astype(np.float64), self.pad, mode="edge"), device=dev)
        self.inner = tuple(slice(self.pad, self.pad + n) for n in shape)
        if m is not None:
            mp[self.inner] = m.double()
        self.s = self.dt**2 / mp
        cmax = 1.0 / math.sqrt(float(m0.astype(np.float64).min()))
        eta = torch.zeros(tuple(n + 2 * self.pad for n in shape), device=dev, dtype=torch.float64)
        for a, n in enumerate(shape):
            i = np.arange(n + 2 * self.pad)
            rho = np.maximum(np.maximum(self.pad - i, i - (self.pad + n - 1)), 0.0)
            e = 3.0 * cmax * math.log(1e3) / (2.0 * self.pad * self.h) * (rho / self.pad) ** 2
            eta += torch.tensor(e, device=dev).reshape((-1,) + (1,) * (self.nd - 1 - a))
        self.G, self.am = 1.0 / (1.0 + 0.5 * self.dt * eta), 1.0 - 0.5 * self.dt * eta
        self.shape, self.pshape, self.dev = shape, eta.shape, dev

    def lap(self, u):
        out = (self.nd * self.W[0]) * u
        for a in range(u.ndim - self.nd, u.ndim):
            n = u.shape[a]
            for k in range(1, 5):
                lo, hi = u.narrow(a, 0, n - k), u.narrow(a, k, n - k)
                out.narrow(a, k, n - k).add_(lo, alpha=self.W[k])
                out.narrow(a, 0, n - k).add_(hi, alpha=self.W[k])
        return out.div_(self.h**2)

    def step(self, u, prev, rhs):
        """G (2u - a- prev + s rhs); prev and rhs are consumed."""
        return rhs.mul_(self.s).add_(u, alpha=2.0).sub_(prev.mul_(self.am)).mul_(self.G)

    def zeros(self, *lead):
        return torch.zeros(tuple(lead) + tuple(self.pshape), device=self.dev, dtype=torch.float64)

    def sample(self, u):
        return u[(Ellipsis,) + tuple(self.rec.T)]

    def groups(self, nb, keep):
        """Shots a batch: at most about 16 GB of history and fields."""
        per = 8.0 * math.prod(self.pshape) * ((self.nt if keep else 0) + 6 + 5 * nb)
        k = max(1, int(16e9 // per))
        return [torch.arange(i, min(i + k, len(self.src))) for i in range(0, len(self.src), k)]

    def sweep(self, shots, dm=None, keep=False, sample_u=False):
        """Incident and Born fields of some shots: (data, Dtt history)."""
        ns, lead = len(shots), (0 if dm is None else dm.shape[0])
        if dm is not None:
            dmp = self.zeros(lead, 1)
            dmp[(Ellipsis,) + self.inner] = dm.double()[:, None]
            f, fp = self.zeros(lead, ns), self.zeros(lead, ns)
            d = torch.zeros(lead, ns, self.nt, len(self.rec), device=self.dev, dtype=torch.float64)
        elif sample_u:
            d = torch.zeros(ns, self.nt, len(self.rec), device=self.dev, dtype=torch.float64)
        else:
            d = None
        hist = self.zeros(self.nt - 1, ns) if keep else None
        u, up = self.zeros(ns), self.zeros(ns)
        at = (torch.arange(ns, device=self.dev),) + tuple(self.src[shots.to(self.dev)].T)
        for n in range(self.nt - 1):
            rhs = self.lap(u)
            rhs[at] += float(self.w[n]) / self.h**self.nd
            un = self.step(u, up.clone(), rhs)
            if keep or dm is not None:
                dtt = torch.add(un, up).sub_(u, alpha=2.0).div_(self.dt**2)
                if keep:
                    hist[n] = dtt
                if dm is not None:
                    f, fp = self.step(f, fp, self.lap(f).sub_(dmp * dtt)), f
                    d[:, :, n + 1] = self.sample(f)
            up, u = u, un
            if sample_u:
                d[:, n + 1] = self.sample(u)
        return d, hist

    def migrate(self, hist, r):
        """- sum_n Dtt u^{n-1} mu^n of data r [nb, ns, nt, nr], summed over these shots."""
        nb, ns = r.shape[:2]
        m1, m2, img = self.zeros(nb, ns), self.zeros(nb, ns), self.zeros(nb)
        flat = self.rec[:, 0]
        for a in range(1, self.nd):
            flat = flat * self.pshape[a] + self.rec[:, a]
        for n in range(self.nt - 1, 0, -1):
            rhs = self.lap(m1)
            rhs.view(nb, ns, -1).index_add_(2, flat, r[:, :, n].double())
            m1, m2 = self.step(m1, m2, rhs), m1
            for j in range(ns):
                img.sub_(hist[n - 1, j] * m1[:, j])
        return img[(Ellipsis,) + self.inner]

    def H(self, dm):
        out = 0.0
        for sh in self.groups(dm.shape[0], True):
            d, hist = self.sweep(sh, dm, keep=True)
            out = out + self.migrate(hist, d)
            del d, hist
        return out


def _multipliers(case, shape, dev):
    """The k-space factors of the expansion, angular-major, and the spatial factors."""
    nd, fs = len(shape), [n + 32 for n in shape]
    ks = []
    for a, N in enumerate(fs):
        f = (torch.fft.rfftfreq if a == nd - 1 else torch.fft.fftfreq)(N, d=case["h"], device=dev, dtype=torch.float64)
        ks.append((2 * math.pi * f).reshape((-1,) + (1,) * (nd - 1 - a)))
    kn = torch.sqrt(sum(k**2 for k in ks))
    ok = kn > 0
    for a, N in enumerate(fs):
        if N % 2 == 0:
            i = [slice(None)] * nd
            i[a] = N // 2
            ok[tuple(i)] = False
    safe = torch.where(kn > 0, kn, torch.ones_like(kn))
    b = _basis_args(case, nd)
    t = torch.arccos(((safe - b["L"]) / (safe + b["L"])).clamp(-1, 1))
    out = []
    for q in b["angular"]:
        if nd == 2:
            th = torch.atan2(ks[0].expand_as(kn), ks[1].expand_as(kn))
            ang = torch.ones_like(kn) if q == 0 else (torch.cos(q * th) if q > 0 else torch.sin(-q * th))
        else:
            kz, ky, kx = (k / safe for k in ks)
            ang = [torch.ones_like(kn), kx * ky, ky * kz, kx * kz, kx**2 - ky**2, 3 * kz**2 - 1][q]
        out += [torch.where(ok, ang * torch.cos(r * t) / safe, torch.zeros_like(kn)) for r in range(b["nradial"])]
    alphas = []
    for mode in b["spatial"]:
        al = torch.ones(tuple(shape), device=dev, dtype=torch.float64)
        for a, k in enumerate(mode):
            i = torch.arange(shape[a], device=dev, dtype=torch.float64) * (2 * math.pi * abs(k) / shape[a])
            f = torch.ones_like(i) if k == 0 else (torch.cos(i) if k > 0 else torch.sin(i))
            al = al * f.reshape((-1,) + (1,) * (nd - 1 - a))
        alphas.append(al)
    return out, alphas


def _filtered(x, mult, shape):
    nd = len(shape)
    X = torch.fft.rfftn(torch.nn.functional.pad(x.double(), (16, 16) * nd))
    w = torch.fft.irfftn(X * mult, s=[n + 32 for n in shape])
    return w[tuple(slice(16, 16 + n) for n in shape)]


def exact(case, seed):
    shapes, op = _shapes(case), case["op"]
    shape = shapes[0]
    if op in ("fit", "precond"):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        mult, alphas = _multipliers(case, shape, dev)
        P = len(mult) * len(alphas)
        if op == "precond":
            c, img = _coeffs(case, seed), _trials(shape, case["h"], 1, seed)[0]
            out = 0.0
            for i, al in enumerate(alphas):
                comb = sum(float(c[i * len(mult) + j]) * m for j, m in enumerate(mult))
                out = out + al * _filtered(img, comb, shape)
            return out
        y, x = _pairs(case, shape, seed)
        A = torch.empty((case["p"],) + tuple(shape) + (P,), device=dev, dtype=torch.float64)
        for j in range(case["p"]):
            for k, m in enumerate(mult):
                f = _filtered(x[j], m, shape)
                for i, al in enumerate(alphas):
                    A[j, ..., i * len(mult) + k] = al * f
        A, b = A.reshape(-1, P), y.double().reshape(-1, 1)
        Q, R = torch.linalg.qr(A)
        c = torch.linalg.solve_triangular(R, Q.T @ b, upper=True)
        res = torch.linalg.norm(b - A @ c) / torch.linalg.norm(b)
        return c[:, 0].cpu().numpy(), float(res)
    outs = []
    for k, s in enumerate(shapes):
        w = _Wave(case, s, seed + 17 * k)
        lvl = _dm_level(_background(s, case["h"], seed + 17 * k))
        if op in ("H", "group"):
            outs.append(w.H(_trials(s, case["h"], case["nb"], seed + 17 * k, lvl)))
        elif op == "F":
            dm = _trials(s, case["h"], case["nb"], seed + 17 * k, lvl)
            return torch.cat([w.sweep(sh, dm)[0] for sh in w.groups(case["nb"], False)], 1)
        elif op == "Fadj":
            d, out = _gathers(case, s, case["nb"], seed), 0.0
            for sh in w.groups(case["nb"], True):
                out = out + w.migrate(w.sweep(sh, keep=True)[1], d[:, sh.to(d.device)])
            return out
        elif op == "grad":
            obs = _gathers(case, s, 1, seed)[0] * 1e-3
            m = torch.tensor(_background(s, case["h"], seed), device=obs.device) + 0.2 * _trials(s, case["h"], 1, seed, lvl)[0]
            w, J, g = _Wave(case, s, seed, m), 0.0, 0.0
            for sh in w.groups(1, True):
                d, hist = w.sweep(sh, keep=True, sample_u=True)
                r = d - obs[sh.to(obs.device)].double()
                J, g = J + 0.5 * (r * r).sum(), g + w.migrate(hist, r[None])[0]
                del hist
            return J, g
        else:  # y_1 = rhs / |rhs|, y_{j+1} = H y_j / |H y_j|
            x, ys, xs = _trials(s, case["h"], 1, seed).double(), [], []
            for _ in range(case["iters"]):
                ys.append(x / x.norm())
                x = w.H(ys[-1])
                xs.append(x)
            return torch.cat(ys), torch.cat(xs)
    return outs if op == "group" else outs[0]
