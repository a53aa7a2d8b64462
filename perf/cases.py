"""Timed workloads of the library: what a program that uses it has it do.

Twelve cases over the public entry points of the package: whole level chains
(FP32, FP64, uneven patch sizes, learned surrogate), single levels (the largest
patches, a handful of small ones), surrogate features and training gradients,
direct simulations (HBM-sized, small, Dirichlet boundaries) and the macro
solver.  `draw` gives further cases of the same kinds with sizes spread over
the same ranges, odd ones among them.  `exact` restates each computation in
64-bit torch / numpy without the package.

Tensors of an FP32 solve are returned in FP32: the entry points store them as
FP64 (their averages are accumulated so), but the fields behind them are FP32.
"""
import functools
import math

import numpy as np
import torch

import paper_1510_00451_gb300 as mlsd

TWO_PI = 2.0 * math.pi


# ---------------------------------------------------------------------------
# Flows: Hermitian-complete mode lists of a stream function on [0, 2 pi)^2.
class Modes:
    def __init__(self, k1, k2, c):
        self.k1 = np.ascontiguousarray(np.concatenate([k1, -k1]), dtype=np.int32)
        self.k2 = np.ascontiguousarray(np.concatenate([k2, -k2]), dtype=np.int32)
        self.re = np.ascontiguousarray(np.concatenate([c.real, c.real]), dtype=np.float64)
        self.im = np.ascontiguousarray(np.concatenate([c.imag, -c.imag]), dtype=np.float64)

    def as_arrays(self):
        return self.k1, self.k2, self.re, self.im


def cellular(terms):
    """sum of a sin(m x1) sin(m x2): half of the modes of each product."""
    m = np.array([t[1] for t in terms])
    a = np.array([t[0] for t in terms])
    return Modes(np.concatenate([m, m]), np.concatenate([-m, m]),
                 np.concatenate([a, -a]).astype(complex) / 4)


@functools.lru_cache(maxsize=None)
def _half_plane(kmax):
    """Modes 1 <= |k| <= kmax of the upper half plane and their amplitudes
    |k|^(-7/3) (a k^(-5/3) energy spectrum) at unit rms speed."""
    k1, k2 = np.meshgrid(np.arange(-kmax, kmax + 1), np.arange(0, kmax + 1))
    k1, k2 = k1.ravel(), k2.ravel()
    r2 = k1 * k1 + k2 * k2
    keep = (r2 >= 1) & (r2 <= kmax * kmax) & ((k2 > 0) | (k1 > 0))
    k1, k2, k = k1[keep], k2[keep], np.sqrt(r2[keep].astype(float))
    amp = k ** (-7.0 / 3.0)
    return k1, k2, amp / math.sqrt(2.0 * np.sum((k * amp) ** 2))


def continuous(kmax, seed, bands=None):
    """Random-phase flow of |k| <= kmax; with bands [(lo, hi), ...] only the modes
    whose two magnitudes lie in one of them."""
    k1, k2, amp = _half_plane(kmax)
    c = amp * np.exp(2j * math.pi * np.random.default_rng(seed).random(amp.size))
    if bands is not None:
        a, b = np.abs(k1), np.abs(k2)
        keep = np.zeros(a.size, dtype=bool)
        for lo, hi in bands:
            keep |= (a >= lo) & (a < hi) & (b >= lo) & (b < hi)
        k1, k2, c = k1[keep], k2[keep], c[keep]
    return Modes(k1, k2, c)


def bases(P, kappa, seed):
    """Symmetric positive definite base tensors (B11, B12, B22) around kappa, as the
    finer levels of a flow give them."""
    r = np.random.default_rng(seed)
    d = kappa * np.exp(r.uniform(0.0, 1.5, (P, 2)))
    x = r.uniform(-0.3, 0.3, P) * np.sqrt(d[:, 0] * d[:, 1])
    return np.stack([d[:, 0], x, d[:, 1]], 1)


def network(hidden, seed):
    """Parameters of one ensemble member whose outputs are small, like those of a
    trained one on levels where the resummed series is already close."""
    r = np.random.default_rng(seed)
    out = []
    for i, (a, b) in enumerate([(mlsd.SUR_IN, hidden), (hidden, hidden), (hidden, hidden),
                                (hidden, 3)]):
        s = (0.1 if i == 3 else 1.0) / math.sqrt(a)
        out += [r.uniform(-s, s, a * b), r.uniform(-0.05, 0.05, b) * (0.1 if i == 3 else 1.0)]
    return np.concatenate(out).astype(np.float32)


def gaussian(n, seed, dtype):
    """Gaussian blob (sigma 0.5) at a seeded centre, minimum-image distance."""
    g = np.random.default_rng(seed).uniform(0.0, TWO_PI, 2)
    x = torch.arange(n, dtype=torch.float64, device=_dev()) * (TWO_PI / n)
    d = [torch.minimum((x - c).abs(), TWO_PI - (x - c).abs()) for c in g]
    return torch.exp(-(d[0][None, :] ** 2 + d[1][:, None] ** 2) / 0.5).to(dtype).contiguous()


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def grid_field(modes, n):
    """The flow's stream function on the n x n node grid, 64-bit, by one inverse FFT."""
    F = torch.zeros(n * n, dtype=torch.complex128, device=_dev())
    ix = torch.from_numpy(np.mod(modes.k2, n).astype(np.int64) * n + np.mod(modes.k1, n)).to(F.device)
    F.index_put_((ix,), torch.from_numpy(modes.re + 1j * modes.im).to(F.device), accumulate=True)
    return torch.fft.ifft2(F.view(n, n)).real * (n * n)


# ---------------------------------------------------------------------------
# Cases
def listed():
    return [
        # The headline workload's hierarchy (three cellular scales, 64^2 patches, full
        # relaxation window) at a quarter of its macro grid's side.
        {"name": "chain_cellular_fp32", "kind": "chain", "N": 32, "levels": 3, "alpha": 4, "n": 64,
         "kappa": 0.01, "precision": "fp32", "steps": 0},
        # The plain method in FP64 on the two-scale cellular flow, full window, and the
        # macro step to T = 1 with its mass record: the run that the rest is checked by.
        {"name": "chain_two_scale_fp64", "kind": "chain", "N": 16, "levels": 2, "alpha": 8, "n": 32,
         "kappa": 0.05, "precision": "fp64", "steps": 0},
        # One coarse octave of the continuous spectrum on 256^2 patches, the largest share
        # of the eight-level hierarchy, with its 256-step window.
        {"name": "level_256", "kind": "level", "N": 16, "lo": 4, "n": 256, "steps": 256, "dump": False},
        # A handful of small patches, full window: a program that looks at single macro
        # nodes, where the serial steps decide.
        {"name": "level_32_few", "kind": "level", "N": 5, "lo": 32, "n": 32, "steps": 0, "dump": False},
        # The continuous-spectrum hierarchy with sizes by the size rule (32^2 .. 256^2 mixed)
        # and off-diagonal parts, one captured graph.
        {"name": "chain_uneven", "kind": "uneven", "N": 16, "kmax": 32, "steps": 256},
        # The two finest octaves, served by the trained ensemble in one captured graph: the
        # production rate of K tensors.
        {"name": "chain_surrogate", "kind": "surrogate", "N": 96, "lo": 64, "levels": 2, "hidden": 256},
        # Features of the 64^2 octave, as data sets for training are assembled.
        {"name": "features_64", "kind": "features", "N": 64, "lo": 16, "n": 64},
        # Gradients of the four members on the training batch.
        {"name": "train_gradient", "kind": "gradient", "rows": 2048, "members": 4, "hidden": 256},
        # The full-domain reference simulation on its grid (HBM-sized), then its macro field.
        {"name": "dns_8192", "kind": "dns", "nf": 8192, "steps": 24, "N": 256},
        # A small flow from its modes: stream function, time step, short run, macro field.
        {"name": "dns_flow_512", "kind": "flow", "nf": 512, "steps": 200, "N": 64, "kmax": 50},
        # The paper's Sec. 4 reference: Dirichlet in x1, 512^2, FP64.
        {"name": "dns_dirichlet_fp64", "kind": "dirichlet", "nf": 512, "steps": 256,
         "precision": "fp64"},
        # The macro solve of the headline workload: a thousand steps on its 128^2 grid.
        {"name": "macro_128", "kind": "macro", "N": 128, "steps": 1000, "precision": "fp32",
         "dirichlet": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "level", "level", "uneven", "surrogate", "features", "gradient",
                       "dns", "flow", "dirichlet", "macro"])
    if kind == "chain":
        if rng.random() < 0.3:
            return {"kind": kind, "N": _log(rng, 3, 16), "levels": 2, "alpha": 8, "n": 32,
                    "kappa": round(rng.uniform(0.03, 0.1), 4), "precision": "fp64", "steps": 0}
        n = rng.choice([32, 64])
        return {"kind": kind, "N": _log(rng, 3, 32 if n == 64 else 64), "levels": rng.choice([2, 3]),
                "alpha": 4, "n": n, "kappa": round(rng.uniform(0.01, 0.05), 4), "precision": "fp32",
                "steps": rng.choice([0, 0, _log(rng, 20, 2000)])}
    if kind == "level":
        n = rng.choice([32, 64, 128, 256])
        lo = {32: rng.choice([32, 64]), 64: 16, 128: 8, 256: rng.choice([2, 4])}[n]
        # correctors (and their energy form) are looked at after short windows
        dump = n <= 64 and rng.random() < 0.4
        return {"kind": kind, "N": _log(rng, 3, {32: 128, 64: 64, 128: 32, 256: 16}[n]), "lo": lo,
                "n": n, "steps": _log(rng, 16, 1024 if n < 128 and not dump else 256), "dump": dump}
    if kind == "uneven":
        return {"kind": kind, "N": _log(rng, 5, 16), "kmax": rng.choice([16, 32]),
                "steps": _log(rng, 32, 256)}
    if kind == "surrogate":
        return {"kind": kind, "N": _log(rng, 9, 96), "lo": 64, "levels": rng.choice([1, 2]),
                "hidden": rng.choice([128, 256])}
    if kind == "features":
        n = rng.choice([32, 64, 64, 128])
        return {"kind": kind, "N": _log(rng, 5, {32: 128, 64: 64, 128: 48}[n]),
                "lo": {32: 32, 64: 16, 128: 8}[n], "n": n}
    if kind == "gradient":
        return {"kind": kind, "rows": _log(rng, 100, 4096), "members": rng.choice([1, 2, 4]),
                "hidden": rng.choice([128, 256])}
    if kind == "dns":
        nf = 128 * _log(rng, 4, 64)
        r = [d for d in (2, 4, 8, 16, 32) if nf % d == 0]
        return {"kind": kind, "nf": nf, "steps": _log(rng, 5, 24 if nf > 2048 else 100),
                "N": nf // rng.choice(r)}
    if kind == "flow":
        nf = 128 * _log(rng, 1, 8)
        return {"kind": kind, "nf": nf, "steps": _log(rng, 20, 200), "N": nf // rng.choice([8, 16, 32]),
                "kmax": _log(rng, 8, 50)}
    if kind == "dirichlet":
        return {"kind": kind, "nf": _log(rng, 64, 512), "steps": _log(rng, 16, 256),
                "precision": rng.choice(["fp32", "fp64"])}
    return {"kind": kind, "N": _log(rng, 8, 256), "steps": _log(rng, 20, 1000),
            "precision": rng.choice(["fp32", "fp64"]), "dirichlet": rng.random() < 0.3}


class State:
    pass


def _chain_problem(c, seed):
    r = np.random.default_rng(seed)
    a = c["alpha"]
    amp = 0.9 + 0.2 * r.random(c["levels"])
    if c["alpha"] == 8:            # two scales of equal amplitude
        modes = cellular([(amp[0], 1), (amp[1], 8)])
        return modes, [1.0, 8.0, 9.0]
    modes = cellular([(amp[j] * float(a) ** -j, a ** j) for j in range(c["levels"])])
    return modes, [float(a ** j) for j in range(c["levels"] + 1)]


def _octaves(lo, levels):
    return [float(lo << j) for j in range(levels + 1)]


UNEVEN_EDGES = {16: [1.0, 2.0, 4.0, 8.0, 17.0], 32: [1.0, 2.0, 4.0, 8.0, 16.0, 33.0]}
KAPPA = 1e-3                       # of the continuous-spectrum flows


def prepare(case, seed):
    c, s, dev = case, State(), _dev()
    s.case = c
    kind = c["kind"]
    f64 = torch.float64
    if kind == "chain":
        modes, edges = _chain_problem(c, seed)
        s.lv = mlsd.Levels(modes, c["kappa"], c["N"], edges, [c["n"]] * c["levels"],
                           precision=c["precision"], n_avg_fixed=c["steps"])
        s.K = torch.empty(c["N"] ** 2, 3, dtype=f64, device=dev)
        if c["precision"] == "fp64":
            s.u0 = gaussian(c["N"], seed, f64)
            s.U = s.u0.clone()
            s.dt, s.macro_steps = _two_scale_macro(c)
    elif kind == "level":
        lo = c["lo"]
        s.lv = mlsd.Levels(continuous(256, seed, [(lo, 2 * lo)]), KAPPA, c["N"], [lo, 2.0 * lo],
                           [c["n"]], n_avg_fixed=c["steps"])
        P = c["N"] ** 2
        s.B = torch.from_numpy(bases(P, KAPPA, seed + 1)).to(dev)
        s.K = torch.empty_like(s.B)
        s.w = torch.empty(P, 2, c["n"], c["n"], dtype=torch.float32, device=dev) if c["dump"] else None
        s.E = torch.empty_like(s.B) if c["dump"] else None
    elif kind == "uneven":
        edges = UNEVEN_EDGES[c["kmax"]]
        s.lv = mlsd.Levels(continuous(c["kmax"], seed), KAPPA, c["N"], edges, [0] * (len(edges) - 1),
                           n_avg_fixed=c["steps"])
        s.K = torch.empty(c["N"] ** 2, 3, dtype=f64, device=dev)
    elif kind == "surrogate":
        edges = _octaves(c["lo"], c["levels"])
        bands = list(zip(edges[:-1], edges[1:]))
        s.lv = mlsd.Levels(continuous(256, seed, bands), KAPPA, c["N"], edges, [32] * c["levels"])
        s.sur = mlsd.Surrogate(members=4, hidden=c["hidden"], max_batch=2048)
        for m in range(4):
            s.sur.set_params(m, network(c["hidden"], 4 * seed + m))
        for l in range(c["levels"]):
            s.lv.attach_surrogate(l + 1, s.sur, 1e-3)
        s.K = torch.empty(c["N"] ** 2, 3, dtype=f64, device=dev)
    elif kind == "features":
        lo = c["lo"]
        s.lv = mlsd.Levels(continuous(256, seed, [(lo, 2 * lo)]), KAPPA, c["N"], [lo, 2.0 * lo],
                           [c["n"]])
        P = c["N"] ** 2
        s.B = torch.from_numpy(bases(P, KAPPA, seed + 1)).to(dev)
        s.X = torch.empty(P, mlsd.SUR_IN, dtype=torch.bfloat16, device=dev)
    elif kind == "gradient":
        s.X, s.Y = _rows(c, seed)
        s.sur = mlsd.Surrogate(members=c["members"], hidden=c["hidden"], max_batch=c["rows"])
        for m in range(c["members"]):
            s.sur.set_params(m, network(c["hidden"], 4 * seed + m))
        s.g = [torch.empty(s.sur.n_params, dtype=torch.float32, device=dev)
               for _ in range(c["members"])]
    elif kind == "dns":
        psi64 = grid_field(continuous(min(256, c["nf"] // 4), seed), c["nf"])
        s.psi = psi64.to(torch.float32).contiguous()
        del psi64
        s.u = gaussian(c["nf"], seed + 1, torch.float32)
        s.ut = torch.empty_like(s.u)
        s.dt = _dns_step(c)
        s.U = torch.empty(c["N"], c["N"], dtype=torch.float32, device=dev)
    elif kind == "flow":
        s.modes = continuous(c["kmax"], seed)
        s.psi = torch.empty(c["nf"], c["nf"], dtype=torch.float32, device=dev)
        s.u = gaussian(c["nf"], seed + 1, torch.float32)
        s.ut = torch.empty_like(s.u)
        s.U = torch.empty(c["N"], c["N"], dtype=torch.float32, device=dev)
    elif kind == "dirichlet":
        t = f64 if c["precision"] == "fp64" else torch.float32
        s.psi = grid_field(continuous(50, seed), c["nf"]).to(torch.float32).contiguous()
        s.u = _step_profile(c["nf"], seed).to(t)
        s.ut = torch.empty_like(s.u)
        s.dt = 0.2 * (TWO_PI / c["nf"]) ** 2 / 4.0
    else:
        t = f64 if c["precision"] == "fp64" else torch.float32
        s.Km = torch.from_numpy(_macro_tensors(c["N"], seed)).to(dev)
        s.U = gaussian(c["N"], seed + 1, t)
        s.dt = _macro_step_of(c)
    return s


def _two_scale_macro(c):
    """Time step and count of the macro run to T = 1 (K of this flow stays below 1)."""
    dt = 0.2 * (TWO_PI / c["N"]) ** 2 / 2.0
    n = int(math.ceil(1.0 / dt))
    return 1.0 / n, n


def _dns_step(c):
    h = TWO_PI / c["nf"]
    return 0.2 * min(h / 6.0, h * h / (4.0 * KAPPA))     # |v1| + |v2| of unit rms flows


def _macro_tensors(N, seed):
    """Smooth positive definite K field of a level chain with a moderate spread."""
    r = np.random.default_rng(seed)
    x = np.arange(N) * (TWO_PI / N)
    p = r.uniform(0, TWO_PI, 4)
    f = 0.6 + 0.2 * np.sin(x[None, :] + p[0]) * np.cos(2 * x[:, None] + p[1])
    g = 0.7 + 0.2 * np.cos(2 * x[None, :] + p[2]) * np.sin(x[:, None] + p[3])
    k12 = 0.1 * np.sin(x[None, :] - x[:, None] + p[0])
    return np.ascontiguousarray(np.stack([f, k12, g], -1).reshape(N * N, 3))


def _macro_step_of(c):
    return 0.2 * (TWO_PI / c["N"]) ** 2 / 1.8


def _step_profile(n, seed):
    """The Sec. 4 step (1 left of the middle, 0 right of it) with a seeded ripple."""
    p = np.random.default_rng(seed).uniform(0, TWO_PI, 2)
    x = torch.arange(n, dtype=torch.float64, device=_dev()) * (TWO_PI / n)
    ripple = 0.05 * torch.sin(x[None, :] + p[0]) * torch.cos(x[:, None] + p[1])
    return ((x <= math.pi).double()[None, :] + ripple).contiguous()


def _rows(c, seed):
    """Training rows of feature-like scale: a decaying spectrum of Fourier features,
    order-one tensors, zero padding; small targets."""
    g = torch.Generator(device=_dev())
    g.manual_seed(seed)
    X = torch.randn(c["rows"], mlsd.SUR_IN, device=_dev(), generator=g)
    X[:, :578] *= 0.5
    X[:, mlsd.SUR_FEATURES:] = 0
    Y = 0.1 * torch.randn(c["rows"], 3, device=_dev(), generator=g)
    return X.to(torch.bfloat16), Y


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "chain":
        s.lv.effective_diffusivity(s.K)
        if c["precision"] == "fp64":
            s.U.copy_(s.u0)
            mass = mlsd.macro_step(s.U, s.K, s.dt, s.macro_steps)
            return {"K": s.K, "U": s.U, "mass": mass}
        return {"K": s.K.float()}
    if kind == "level":
        s.lv.solve_level(1, s.B, s.K, w_dump=s.w)
        if not c["dump"]:
            return {"K": s.K.float()}
        s.lv.corrector_energy(1, s.B, s.w, s.E)
        return {"K": s.K.float(), "w": s.w, "E": s.E.float()}
    if kind == "uneven":
        s.lv.effective_diffusivity(s.K)
        return {"K": s.K.float()}
    if kind == "surrogate":
        s.lv.effective_diffusivity(s.K, mode=mlsd.MLSD_SURROGATE)
        return {"K": s.K.float()}
    if kind == "features":
        s.lv.features(1, s.B, s.X)
        return {"X": s.X}
    if kind == "gradient":
        loss = [s.sur.grad(m, s.X, s.Y, s.g[m]) for m in range(c["members"])]
        return {"grad": s.g, "loss": np.array(loss, dtype=np.float32)}
    if kind == "dns":
        mlsd.dns_run(s.u, s.ut, s.psi, KAPPA, s.dt, c["steps"])
        mlsd.coarse_grain(s.u, c["N"], s.U, want_mass=False)
        return {"u": s.u, "U": s.U}
    if kind == "flow":
        mlsd.grid_psi(s.modes, c["nf"], s.psi)
        dt = mlsd.dns_dt(s.psi, KAPPA, 0.2)
        mlsd.dns_run(s.u, s.ut, s.psi, KAPPA, dt, c["steps"])
        mlsd.coarse_grain(s.u, c["N"], s.U, want_mass=False)
        return {"psi": s.psi, "u": s.u, "U": s.U}
    if kind == "dirichlet":
        mlsd.dns_run_dirichlet(s.u, s.ut, s.psi, 1.0, s.dt, c["steps"])
        return {"u": s.u}
    if c["dirichlet"]:
        mlsd.macro_step_dirichlet(s.U, s.Km, s.dt, c["steps"])
    else:
        mlsd.macro_step(s.U, s.Km, s.dt, c["steps"], want_mass=False)
    return {"U": s.U}


# ---------------------------------------------------------------------------
# Work that a pass cannot do without.  A cell-update (one cell of one corrector
# field, one Heun step) is 34 floating-point operations, 39 inside the window.
def _full_window(n, cfl=0.2):
    """8 + 4 relaxation times at the diffusive time step."""
    return int(12 * n * n / (math.pi ** 2 * cfl))


def _patch_flops(P, n, steps):
    if steps > 0:
        return 2.0 * P * n * n * steps * 39
    t = _full_window(n)
    return 2.0 * P * n * n * t * (34 + 5 / 3.0)


def _series_flops(P, n):
    """36 complex n x n FFTs and 17 stencil applications per patch, the 17 x 17 window."""
    nf = min(n, 64)
    fft = 36 * 5.0 * nf * nf * math.log2(nf * nf)
    return P * (fft + 17 * 30.0 * nf * nf + 4.0 * 17 * (nf * nf + 17 * nf))


def _mlp_flops(rows, hidden):
    return 2.0 * rows * (mlsd.SUR_IN * hidden + 2 * hidden * hidden + 3 * hidden)


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("chain", "level"):
        P, n = c["N"] ** 2, c["n"]
        levels = c.get("levels", 1)
        b = levels * P * (24 + 24)
        if c.get("dump"):
            b += 2.0 * P * n * n * 4
        return {"bytes": b, "flops": levels * _patch_flops(P, n, c["steps"])}
    if kind == "uneven":
        # 256^2 down to the octave at 8, then smaller: counted as the size rule gives it
        P, L = c["N"] ** 2, len(UNEVEN_EDGES[c["kmax"]]) - 1
        sizes = [256, 256, 256, 128, 64][:L]
        return {"bytes": L * P * 48, "flops": sum(_patch_flops(P, n, c["steps"]) for n in sizes)}
    if kind == "surrogate":
        P = c["N"] ** 2
        return {"bytes": c["levels"] * P * 48,
                "flops": c["levels"] * (_series_flops(P, 32) + 4 * _mlp_flops(P, c["hidden"]))}
    if kind == "features":
        P = c["N"] ** 2
        return {"bytes": P * (24 + 2 * mlsd.SUR_IN),
                "flops": _series_flops(P, c["n"])}
    if kind == "gradient":
        p = mlsd.SUR_IN * c["hidden"] + 2 * c["hidden"] ** 2 + 3 * c["hidden"]
        return {"bytes": c["rows"] * (2 * mlsd.SUR_IN + 12) + c["members"] * 8.0 * p,
                "flops": c["members"] * 3 * _mlp_flops(c["rows"], c["hidden"])}
    if kind in ("dns", "flow"):
        n2 = float(c["nf"]) ** 2
        w = {"bytes": 12.0 * n2 * c["steps"] + 4 * n2, "flops": 48.0 * n2 * c["steps"]}
        if kind == "flow":
            w["flops"] += 5.0 * n2 * math.log2(n2)
        return w
    if kind == "dirichlet":
        n2, b = float(c["nf"]) ** 2, 8 if c["precision"] == "fp64" else 4
        return {"bytes": n2 * (2 * b + 4), "flops": 48.0 * n2 * c["steps"]}
    n2, b = float(c["N"]) ** 2, 8 if c["precision"] == "fp64" else 4
    return {"bytes": n2 * (2 * b + 24), "flops": 100.0 * n2 * c["steps"]}


# ---------------------------------------------------------------------------
# 64-bit restatements
def _r(x, d1, d2):
    """x at node (a + d1, b + d2), periodic; layout [..., b, a]."""
    return torch.roll(x, (-d2, -d1), (-2, -1))


def _origins(N, Nl, n):
    i = np.arange(N, dtype=np.int64)
    return torch.from_numpy((2 * i * Nl + N) // (2 * N) - n // 2).to(_dev())


def _patches(band, N, n):
    """Samples [P][n][n] of a level's band grid on every patch, p = j N + i."""
    Nl = band.shape[0]
    o = _origins(N, Nl, n)
    t = torch.arange(n, device=_dev())
    i = (o[:, None] + t) % Nl                                   # [N][n]
    g = band[i[:, None, :, None], i[None, :, None, :]]          # [j][i][b][a]
    return g.reshape(N * N, n, n)


def _patch_K(psi, B, L, steps, cfl=0.2):
    """Heun time stepping of both correctors of every patch: K and the final w."""
    P, n, _ = psi.shape
    h = L / n
    v1 = -(_r(psi, 0, 1) - _r(psi, 0, -1)) / (2 * h)
    v2 = (_r(psi, 1, 0) - _r(psi, -1, 0)) / (2 * h)
    vm = (v1.abs() + v2.abs()).amax((1, 2))
    b11, b12, b22 = B[:, 0], B[:, 1], B[:, 2]
    lmin = 0.5 * ((b11 + b22) - torch.sqrt((b11 - b22) ** 2 + 4 * b12 ** 2))
    dt = cfl * torch.minimum(h * h / (2 * (b11 + b22) + 4 * b12.abs()), h / vm)
    dt = torch.minimum(dt, (8 * lmin * h * h / vm ** 4) ** (1.0 / 3.0))
    tau = L * L / (4 * math.pi ** 2 * lmin)
    nb = torch.ceil(8 * tau / dt) if steps == 0 else torch.zeros_like(dt)
    na = torch.ceil(4 * tau / dt) if steps == 0 else torch.full_like(dt, float(steps))
    e = lambda t: t.view(P, 1, 1, 1)                            # noqa: E731
    cx, cy = (e(dt) * v1[:, None] / (2 * h)), (e(dt) * v2[:, None] / (2 * h))
    src = torch.stack([dt.view(P, 1, 1) * v1, dt.view(P, 1, 1) * v2], 1)
    d11, d22, d12 = e(dt * b11 / h ** 2), e(dt * b22 / h ** 2), e(dt * b12 / (2 * h ** 2))

    def f(x):
        E, W, Nn, S = _r(x, 1, 0), _r(x, -1, 0), _r(x, 0, 1), _r(x, 0, -1)
        g = cx * (E - W) + cy * (Nn - S) + d11 * (E + W - 2 * x) + d22 * (Nn + S - 2 * x) + src
        D = E - W
        return g + d12 * (_r(D, 0, 1) - _r(D, 0, -1))

    w = torch.zeros(P, 2, n, n, dtype=torch.float64, device=psi.device)
    S = torch.zeros(P, 2, 2, dtype=torch.float64, device=psi.device)
    total = int((nb + na).max().item())
    last = nb + na
    same = bool((nb == nb[0]).all() and (na == na[0]).all())
    for k in range(total):
        k1 = f(w)
        nw = w + 0.5 * (k1 + f(w + k1))
        w = nw if same else torch.where(e(last > k), nw, w)
        if k >= int(nb.min().item()) if same else True:
            m = torch.stack([(v1[:, None] * w).mean((2, 3)), (v2[:, None] * w).mean((2, 3))], 1)
            S += m * ((nb <= k) & (last > k)).view(P, 1, 1)
    S = S / na.view(P, 1, 1)
    K = torch.stack([b11 + S[:, 0, 0], b12 + 0.5 * (S[:, 0, 1] + S[:, 1, 0]), b22 + S[:, 1, 1]], 1)
    return K, w


def _energy(w, B, h):
    fx, fy = (_r(w, 1, 0) - w) / h, (_r(w, 0, 1) - w) / h
    cx, cy = (_r(w, 1, 0) - _r(w, -1, 0)) / (2 * h), (_r(w, 0, 1) - _r(w, 0, -1)) / (2 * h)
    out = []
    for j, k in ((0, 0), (0, 1), (1, 1)):
        out.append(B[:, 0] * (fx[:, j] * fx[:, k]).mean((1, 2)) + B[:, 2] * (fy[:, j] * fy[:, k]).mean((1, 2))
                   + B[:, 1] * (cx[:, j] * cy[:, k] + cy[:, j] * cx[:, k]).mean((1, 2)))
    return torch.stack(out, 1)


def _wynn(p, K):
    """[K/K] at 1 of sum p_k x^k from the partial sums' epsilon table (p [..., 9]); where
    a difference vanishes, the last even column reached."""
    cur = torch.cumsum(p[..., :2 * K + 1], -1)
    prev = torch.zeros(*cur.shape[:-1], cur.shape[-1] + 1, dtype=cur.dtype, device=cur.device)
    best, live = cur[..., -1], torch.ones(cur.shape[:-1], dtype=torch.bool, device=cur.device)
    for k in range(1, 2 * K + 1):
        d = cur[..., 1:] - cur[..., :-1]
        live = live & (d.abs() >= 1e-300).all(-1)
        prev, cur = cur, prev[..., 1:-1] + 1.0 / d
        if k % 2 == 0:
            best = torch.where(live, cur[..., 0], best)
    return best


def _features(psi, B, kappa):
    """The 606 features of every patch and the series estimate E [P][3]."""
    P, n, _ = psi.shape
    nf = min(n, 64)
    psi = psi[:, ::n // nf, ::n // nf]
    n = nf
    psi = psi - psi.mean((1, 2), keepdim=True)
    F = torch.fft.fft2(psi)
    k = torch.arange(-8, 9, device=psi.device) % n
    win = F[:, k[:, None], k[None, :]] / (n * n)
    tr = (B[:, 0] + B[:, 2])
    win = win * (mlsd.SUR_PSI_SCALE / (0.5 * tr)).view(P, 1, 1)
    t = TWO_PI * torch.arange(n, device=psi.device, dtype=torch.float64) / n
    t1, t2 = t[None, :], t[:, None]
    e = lambda x: x.view(P, 1, 1)                               # noqa: E731
    D = (e(B[:, 0]) * (2 - 2 * torch.cos(t1)) + e(B[:, 2]) * (2 - 2 * torch.cos(t2))
         + 2 * e(B[:, 1]) * torch.sin(t1) * torch.sin(t2))
    D[:, 0, 0] = 1
    g = 1 / D
    g[:, 0, 0] = 0
    v1 = -(_r(psi, 0, 1) - _r(psi, 0, -1)) / 2
    v2 = (_r(psi, 1, 0) - _r(psi, -1, 0)) / 2
    c = torch.fft.ifft2(torch.fft.fft2(torch.complex(v1, v2)) * g)
    T = []
    for m in range(2, 20):
        c1, c2 = c.real, c.imag
        T.append(torch.stack([(v1 * c1).mean((1, 2)), 0.5 * ((v1 * c2).mean((1, 2)) + (v2 * c1).mean((1, 2))),
                              (v2 * c2).mean((1, 2))], 1))
        if m == 19:
            break
        a = v1 * (_r(c, 1, 0) - _r(c, -1, 0)) / 2 + v2 * (_r(c, 0, 1) - _r(c, 0, -1)) / 2
        c = torch.fft.ifft2(torch.fft.fft2(a) * g)
    T = torch.stack(T, 2)                                       # [P][3][18]
    p = T[..., 0::2] + T[..., 1::2]
    pade = [_wynn(p, q) for q in (2, 3, 4)]
    sc = (mlsd.SUR_T_SCALE / tr)[:, None]
    out = torch.zeros(P, mlsd.SUR_FEATURES, dtype=torch.float64, device=psi.device)
    out[:, 0:578] = torch.view_as_real(win).reshape(P, 578)
    out[:, 578:581] = B / kappa
    out[:, 581] = math.log(kappa)
    out[:, 582:597] = torch.asinh(sc[:, :, None] * T[..., :5].transpose(1, 2)).reshape(P, 15)
    for q in range(3):
        out[:, 597 + 3 * q:600 + 3 * q] = torch.asinh(sc * pade[q])
    return out, pade[2]


def _layers(params, hidden):
    p, o, out = torch.from_numpy(params).double().to(_dev()), 0, []
    for a, b in [(mlsd.SUR_IN, hidden), (hidden, hidden), (hidden, hidden), (hidden, 3)]:
        out.append((p[o:o + a * b].view(b, a), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _mlp(layers, x):
    for i, (W, b) in enumerate(layers):
        x = x @ W.T + b
        if i < 3:
            x = torch.nn.functional.gelu(x)
    return x


def _macro_rhs(U, K, H, dirichlet):
    """div(K grad U) in flux form; face tensors are node means."""
    k11, k12, k22 = K
    if dirichlet:                  # the column past the last is the boundary value 0
        U = torch.cat([U, torch.zeros_like(U[:, :1])], 1)
        k11, k12, k22 = (torch.cat([k, k[:, :1]], 1) for k in K)
    else:
        U = torch.cat([U, U[:, :1]], 1)
        k11, k12, k22 = (torch.cat([k, k[:, :1]], 1) for k in K)
    up, dn = torch.roll(U, -1, 0), torch.roll(U, 1, 0)
    dy = up - dn                                                # 2H d/dy at nodes
    a, b = slice(None, -1), slice(1, None)
    fx = (0.5 * (k11[:, a] + k11[:, b]) * (U[:, b] - U[:, a]) / H
          + 0.5 * (k12[:, a] + k12[:, b]) * (dy[:, a] + dy[:, b]) / (4 * H))   # faces i + 1/2
    if dirichlet:
        dx = torch.zeros_like(fx)
        dx[:, 1:] = U[:, 2:] - U[:, :-2]
    else:
        dx = U[:, b] - torch.roll(U[:, a], 1, 1)
    k12c, k22c, Uc = k12[:, a], k22[:, a], U[:, a]
    fy = (0.5 * (k22c + torch.roll(k22c, -1, 0)) * (torch.roll(Uc, -1, 0) - Uc) / H
          + 0.5 * (k12c + torch.roll(k12c, -1, 0)) * (dx + torch.roll(dx, -1, 0)) / (4 * H))
    r = (fx - torch.roll(fx, 1, 1)) / H + (fy - torch.roll(fy, 1, 0)) / H
    if dirichlet:
        r[:, 0] = 0
    return r


def _macro(U, Kn, dt, steps, dirichlet, mass=False):
    N = U.shape[0]
    H = TWO_PI / N
    K = [Kn[:, q].reshape(N, N).contiguous() for q in range(3)]
    if dirichlet:
        U = U.clone()
        U[:, 0] = 1.0
    m = [U.sum() * H * H]
    for _ in range(steps):
        k1 = dt * _macro_rhs(U, K, H, dirichlet)
        U = U + 0.5 * (k1 + dt * _macro_rhs(U + k1, K, H, dirichlet))
        if mass:
            m.append(U.sum() * H * H)
    return U, torch.stack(m)


def _dns(u, psi, kappa, dt, steps, dirichlet=False):
    n = u.shape[0]
    h = TWO_PI / n
    psi = psi.double()
    cx = dt / (4 * h * h) * (_r(psi, 0, -1) - _r(psi, 0, 1))
    cy = dt / (4 * h * h) * (_r(psi, 1, 0) - _r(psi, -1, 0))
    cd = dt * kappa / (h * h)
    if dirichlet:
        u[:, 0] = 1.0

    def f(x):
        E, W, Nn, S = _r(x, 1, 0), _r(x, -1, 0), _r(x, 0, 1), _r(x, 0, -1)
        if dirichlet:
            E[:, -1] = 0.0
        g = cd * (E + W + Nn + S - 4 * x)
        E -= W
        g += cx * E
        Nn -= S
        g += cy * Nn
        if dirichlet:
            g[:, 0] = 0
        return g

    for _ in range(steps):
        k1 = f(u)
        s = u + k1
        k1 += f(s)
        u = u + 0.5 * k1
    return u


def _coarse(u, N):
    n = u.shape[0]
    r = n // N
    return torch.roll(u, (r // 2, r // 2), (0, 1)).reshape(N, r, N, r).mean((1, 3))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "chain":
        # full windows of 64^2 patches are tens of thousands of 64-bit steps a level
        if c["n"] > 32 and (c["steps"] == 0 or c["steps"] * c["N"] ** 2 > 200_000):
            return None
        if c["N"] ** 2 * c["levels"] > 1100:
            return None
        modes, edges = _chain_problem(c, seed)
        P, K = c["N"] ** 2, None
        B = torch.zeros(P, 3, dtype=torch.float64, device=_dev())
        B[:, 0] = B[:, 2] = c["kappa"]
        for l in reversed(range(c["levels"])):
            m = int(edges[l])
            top = np.maximum(np.abs(modes.k1), np.abs(modes.k2))
            keep = (top >= (0 if l == 0 else edges[l])) & (top < edges[l + 1])
            part = State()
            part.k1, part.k2, part.re, part.im = (x[keep] for x in modes.as_arrays())
            psi = _patches(grid_field(part, c["n"] * m), c["N"], c["n"])
            K, _ = _patch_K(psi, B, TWO_PI / m, c["steps"])
            B = K
        if c["precision"] != "fp64":
            return {"K": K}
        dt, n = _two_scale_macro(c)
        U, mass = _macro(gaussian(c["N"], seed, torch.float64), K, dt, n, False, True)
        return {"K": K, "U": U, "mass": mass}
    if kind == "level":
        lo, n, P = c["lo"], c["n"], c["N"] ** 2
        steps = c["steps"] or 4 * _full_window(n)
        if P * n * n * steps > 6e9 or steps > 40_000:
            return None
        band = grid_field(continuous(256, seed, [(lo, 2 * lo)]), n * lo)
        B = torch.from_numpy(bases(P, KAPPA, seed + 1)).to(_dev())
        K, w = _patch_K(_patches(band, c["N"], n), B, TWO_PI / lo, c["steps"])
        if not c["dump"]:
            return {"K": K}
        return {"K": K, "w": w, "E": _energy(w, B, TWO_PI / lo / n)}
    if kind == "uneven":
        return None                # every algorithm of the chain at four patch sizes
    if kind == "surrogate":
        P = c["N"] ** 2
        edges = _octaves(c["lo"], c["levels"])
        flow = continuous(256, seed, list(zip(edges[:-1], edges[1:])))
        nets = [_layers(network(c["hidden"], 4 * seed + m), c["hidden"]) for m in range(4)]
        B = torch.zeros(P, 3, dtype=torch.float64, device=_dev())
        B[:, 0] = B[:, 2] = KAPPA
        for l in reversed(range(c["levels"])):
            m = int(edges[l])
            keep = (np.abs(flow.k1) >= edges[l]) & (np.abs(flow.k1) < edges[l + 1])
            part = State()
            part.k1, part.k2, part.re, part.im = (x[keep] for x in flow.as_arrays())
            F, E = _features(_patches(grid_field(part, 32 * m), c["N"], 32), B, KAPPA)
            X = torch.zeros(P, mlsd.SUR_IN, dtype=torch.float64, device=_dev())
            X[:, :mlsd.SUR_FEATURES] = F
            o = sum(torch.sinh(_mlp(net, X)) for net in nets) / 4
            B = B + E + (B[:, 0] + B[:, 2])[:, None] / mlsd.SUR_Y_SCALE * o
        return {"K": B}
    if kind == "features":
        lo, n, P = c["lo"], c["n"], c["N"] ** 2
        band = grid_field(continuous(256, seed, [(lo, 2 * lo)]), n * lo)
        B = torch.from_numpy(bases(P, KAPPA, seed + 1)).to(_dev())
        F, _ = _features(_patches(band, c["N"], n), B, KAPPA)
        X = torch.zeros(P, mlsd.SUR_IN, dtype=torch.float64, device=_dev())
        X[:, :mlsd.SUR_FEATURES] = F
        return {"X": X}
    if kind == "gradient":
        X, Y = _rows(c, seed)
        grads, losses = [], []
        for m in range(c["members"]):
            layers = _layers(network(c["hidden"], 4 * seed + m), c["hidden"])
            leaves = [t.clone().requires_grad_() for pair in layers for t in pair]
            loss = ((_mlp(list(zip(leaves[::2], leaves[1::2])), X.double()) - Y.double()) ** 2).mean()
            grads.append(torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, leaves)]))
            losses.append(loss.detach())
        return {"grad": grads, "loss": torch.stack(losses)}
    if kind == "dns":
        psi = grid_field(continuous(min(256, c["nf"] // 4), seed), c["nf"]).to(torch.float32)
        u = _dns(gaussian(c["nf"], seed + 1, torch.float32).double(), psi, KAPPA, _dns_step(c),
                 c["steps"])
        return {"u": u, "U": _coarse(u, c["N"])}
    if kind == "flow":
        psi = grid_field(continuous(c["kmax"], seed), c["nf"])
        h = TWO_PI / c["nf"]
        v = ((_r(psi, 0, 1) - _r(psi, 0, -1)).abs() + (_r(psi, 1, 0) - _r(psi, -1, 0)).abs()).max()
        dt = 0.2 * min(h / (v.item() / (2 * h)), h * h / (4 * KAPPA))
        u = _dns(gaussian(c["nf"], seed + 1, torch.float32).double(), psi, KAPPA, dt, c["steps"])
        return {"psi": psi, "u": u, "U": _coarse(u, c["N"])}
    if kind == "dirichlet":
        t = torch.float64 if c["precision"] == "fp64" else torch.float32
        psi = grid_field(continuous(50, seed), c["nf"]).to(torch.float32)
        dt = 0.2 * (TWO_PI / c["nf"]) ** 2 / 4.0
        return {"u": _dns(_step_profile(c["nf"], seed).to(t).double(), psi, 1.0, dt, c["steps"], True)}
    t = torch.float64 if c["precision"] == "fp64" else torch.float32
    U = gaussian(c["N"], seed + 1, t).double()
    Km = torch.from_numpy(_macro_tensors(c["N"], seed)).to(_dev())
    return {"U": _macro(U, Km, _macro_step_of(c), c["steps"], c["dirichlet"])[0]}
