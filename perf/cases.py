"""Performance cases: the evaluations that a user of this library runs.

Each case is a plan that a program keeps (aperture, wavelength, tolerance,
precision) and one call, or one design step, through the public entry points:
fields on uniform grids and at scattered targets, wavelength and instance
batches, and the gradients of aperture designs.  Sizes are those of the
repository's workloads (the disc at Fresnel number 10, the five-armed star at
100, the 24-petal starshade sweep and its spline design, the random smooth
aperture at 1000 and its uneven batch, the Koch snowflake, the kite), and the
drawn cases spread over the same ranges.

Shapes and targets are drawn from the seed; `exact` is the same sum written
out in FP64 torch (dense matrix products over the grid's axes, or over a
Chebyshev product grid that resolves the field for scattered targets).
"""
import math

import numpy as np
import torch

from paper_2010_05978_gb300 import BatchPlan, Plan
from paper_2010_05978_gb300.fresnel import profile_field

TWO_PI = 2.0 * math.pi
EXACT_FLOPS = 1.1e13          # FP64 operations above which `exact` is left out


# ---------------------------------------------------------------- the cases
def _grid(name, **kw):
    c = {"kind": "grid", "shape": "star", "n_panels": 128, "p": 16, "m": 256, "fresnel": 100.0,
         "n1": 1000, "n2": 1000, "span": 3.0, "x0": 0.0, "y0": 0.0, "precision": "fp32",
         "tol": 1e-6, "output": "aperture", "recompute": True, "sync": False, "screen": 0}
    c.update(kw)
    c["name"] = name
    return c


def _scattered(name, **kw):
    c = {"kind": "scattered", "shape": "star", "n_panels": 128, "p": 16, "m": 256,
         "fresnel": 100.0, "targets": 1000000, "half": 1.5, "region": "disc",
         "precision": "fp32", "tol": 1e-6, "output": "aperture", "recompute": True}
    c.update(kw)
    c["name"] = name
    return c


def listed():
    return [
        # the first call anyone makes, and the one a live display repeats: a
        # small disc on a 100 x 100 grid with the default options (quadrature
        # kept in the plan, status read back on every call)
        _grid("disc_grid_small", shape="disc", n_panels=64, m=16, fresnel=10.0, n1=100, n2=100,
              recompute=False, sync=True),
        # the ordinary call: half a million nodes onto a 1000 x 1000 grid,
        # quadrature regenerated (an aperture that moves between calls)
        _grid("star_grid"),
        # the same aperture seen at a million scattered detector positions
        _scattered("star_scattered"),
        # reference-quality fields: FP64 at the tightest tolerance in use
        _grid("star_grid_fp64", precision="fp64", tol=1e-12),
        # FP64 at an ordinary tolerance, scattered targets
        _scattered("star_scattered_fp64", precision="fp64"),
        # odd and ragged: a kite given by its boundary rule, seen off axis on a
        # 701 x 533 grid through a source screen (amplitude and path difference)
        _grid("kite_screen_odd", shape="kite", n_panels=900, p=1, m=130, fresnel=60.0, n1=701,
              n2=533, span=2.4, x0=0.21, y0=-0.13, screen=65, recompute=False),
        # a starshade's shadow at 64 wavelengths on the 512 x 512 pupil grid
        {"name": "starshade_sweep64", "kind": "sweep", "n_lambda": 64, "n": 512, "tol": 1e-6,
         "precision": "fp32"},
        # one step of a starshade design loop: the field at 8 wavelengths as a
        # differentiable function of 200 spline coefficients, loss and gradient
        {"name": "starshade_design_step", "kind": "design", "n_lambda": 8, "n": 256,
         "n_coef": 200, "tol": 1e-6, "precision": "fp32"},
        # one step of fitting an aperture's outline in FP64: field and the
        # gradient of mean |u|^2 in its Fourier coefficients, plan kept
        {"name": "star_shape_gradient_fp64", "kind": "shape_grad", "n_panels": 64, "p": 16,
         "m": 128, "fresnel": 50.0, "n": 256, "tol": 1e-10, "precision": "fp64"},
        # a fractal aperture: four million one-point triangles
        {"name": "koch_grid", "kind": "koch", "level": 11, "lz": 0.01, "n": 1000, "tol": 1e-6,
         "precision": "fp32"},
        # many apertures of uneven size, each with its own targets, in one call
        {"name": "random_batch32", "kind": "batch", "n": 32, "nodes_lo": 1e5, "nodes_hi": 2e6,
         "targets_lo": 1e5, "targets_hi": 1e7, "tol": 1e-6, "precision": "fp32"},
        # the largest: ten million nodes, a hundred million targets, F = 1000
        _scattered("random_aperture_F1000", shape="random", n_panels=640, m=1024, fresnel=1000.0,
                   targets=100000000, half=1.2, region="square"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid64", "scattered", "scattered", "scattered64", "sweep",
                       "design", "shape_grad", "koch", "batch", "screen"])
    c = None
    if kind in ("grid", "grid64", "screen"):
        F = _log(rng, 5.0, 200.0)
        n1 = int(_log(rng, 64, 1400))
        n2 = max(33, int(n1 * rng.uniform(0.6, 1.4)))
        m = max(16, int(2.2 * F * rng.uniform(0.8, 1.6)))
        panels = max(24, int(m * rng.uniform(0.4, 0.8)))
        tol = 1e-6
        if kind == "grid64":
            tol = 10.0 ** -rng.choice([6, 8, 9, 10, 12])
        c = _grid("", shape=rng.choice(["star", "disc", "random"]), n_panels=panels, m=m, fresnel=F,
                  n1=n1, n2=n2, span=rng.uniform(2.0, 3.0), tol=tol,
                  precision="fp64" if kind == "grid64" else "fp32",
                  output=rng.choice(["aperture", "occulter"]), recompute=rng.random() < 0.6,
                  sync=rng.random() < 0.3)
        if kind == "screen":
            c.update(shape="kite", n_panels=16 * panels, p=1, x0=rng.uniform(-0.4, 0.4),
                     y0=rng.uniform(-0.4, 0.4), screen=rng.choice([33, 64, 97]))
    elif kind in ("scattered", "scattered64"):
        F = _log(rng, 5.0, 150.0 if kind == "scattered64" else 700.0)
        m = max(16, int(1.2 * F * rng.uniform(0.8, 1.6)) + 12)
        c = _scattered("", shape=rng.choice(["star", "disc", "random"]),
                       n_panels=max(24, int(m * rng.uniform(0.5, 0.7))), m=m, fresnel=F,
                       targets=int(_log(rng, 1e3, 2e6 if kind == "scattered64" else 2e7)),
                       half=rng.uniform(1.0, 1.6), region=rng.choice(["disc", "square"]),
                       precision="fp64" if kind == "scattered64" else "fp32",
                       tol=10.0 ** -rng.choice([6, 8, 10, 12]) if kind == "scattered64" else 1e-6,
                       output=rng.choice(["aperture", "occulter"]), recompute=rng.random() < 0.6)
    elif kind == "sweep":
        c = {"kind": "sweep", "n_lambda": rng.randint(2, 48), "n": int(_log(rng, 96, 640)),
             "tol": 1e-6, "precision": rng.choice(["fp32", "fp32", "fp64"])}
    elif kind == "design":
        c = {"kind": "design", "n_lambda": rng.randint(1, 8), "n": int(_log(rng, 48, 300)),
             "n_coef": rng.randint(20, 200), "tol": 1e-6, "precision": "fp32"}
    elif kind == "shape_grad":
        m = rng.randint(40, 160)
        c = {"kind": "shape_grad", "n_panels": max(24, m // 2), "p": 16, "m": m,
             "fresnel": _log(rng, 5.0, 60.0), "n": int(_log(rng, 48, 320)),
             "tol": 10.0 ** -rng.choice([8, 10, 12]), "precision": "fp64"}
    elif kind == "koch":
        c = {"kind": "koch", "level": rng.randint(7, 10), "lz": _log(rng, 0.01, 0.04),
             "n": int(_log(rng, 200, 1200)), "tol": 1e-6, "precision": "fp32"}
    else:
        c = {"kind": "batch", "n": rng.randint(2, 12), "nodes_lo": 5e4, "nodes_hi": 1e6,
             "targets_lo": 1e4, "targets_hi": 3e6, "tol": 1e-6, "precision": "fp32"}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _npr(seed, stream=0):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, int(stream)])


def _fourier_params(shape, g):
    if shape == "disc":            # the unit disc, out of round by a part in a thousand
        par = np.zeros(9)
        par[0] = 1.0
        par[1:] = 1e-3 * g.standard_normal(8)
        return par, 1.0
    if shape == "star":            # r = 1 + 0.3 cos 5t and small imperfections
        par = np.zeros(15)
        par[0], par[9] = 1.0, 0.3
        par[1:] += 1e-3 * g.standard_normal(14)
        return par, 1.3
    a, ph = g.uniform(0.0, 0.02, 20), g.uniform(0.0, TWO_PI, 20)
    par = np.empty(41)             # random smooth aperture, 20 modes
    par[0], par[1::2], par[2::2] = 1.0, a * np.cos(ph), -a * np.sin(ph)
    th = TWO_PI * np.arange(4096) / 4096
    k = np.arange(1, 21)[:, None]
    r = 1.0 + (par[1::2, None] * np.cos(k * th) + par[2::2, None] * np.sin(k * th)).sum(0)
    return par, float(r.max())


def _aperture(c, seed, stream=0):
    """(families, lambda z) of a Fourier-boundary or kite case."""
    g = _npr(seed, stream)
    if c["shape"] == "kite":       # periodic trapezoid boundary rule, dilated radii
        n = c["n_panels"]
        t = TWO_PI * np.arange(1, n + 1) / n
        e = 1.0 + 0.02 * g.standard_normal(2)
        X, Y = e[0] * (0.5 * np.cos(t) + 0.5 * np.cos(2 * t)), e[1] * np.sin(t)
        W, V = e[0] * (-0.5 * np.sin(t) - np.sin(2 * t)) * TWO_PI / n, e[1] * np.cos(t) * TWO_PI / n
        fam = {"kind": "line_rule", "X": X, "Y": Y, "W": W, "V": V, "m": c["m"]}
        return [fam], 1.13 ** 2 / c["fresnel"]
    par, R = _fourier_params(c["shape"], g)
    fam = {"kind": "fourier", "params": par, "n_panels": c["n_panels"], "p": c["p"], "m": c["m"]}
    return [fam], R * R / c["fresnel"]


def _screen(c, seed):
    """Smooth amplitude and path difference over [-1.5, 1.5]^2, or None."""
    n = c["screen"]
    if not n:
        return None
    g = _npr(seed, 7)
    s = np.linspace(-1.5, 1.5, n)
    X, Y = np.meshgrid(s, s, indexing="xy")
    k, q = g.uniform(1.0, 3.0, 6), g.uniform(0.0, TWO_PI, 6)
    amp = 1.0 + 0.1 * np.cos(k[0] * X + q[0]) * np.cos(k[1] * Y + q[1])
    lam = 1.13 ** 2 / c["fresnel"]     # the kite's wavelength at z = 1: a third of it, peak to valley
    opd = lam * (0.12 * np.sin(k[2] * X + q[2]) * np.sin(k[3] * Y + q[3])
                 + 0.05 * np.cos(k[4] * (X + Y)))
    return {"amp": amp, "opd": opd, "box": (-1.5, 1.5, -1.5, 1.5)}


def _targets(n, half, region, seed, stream=1):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFF)
    t = torch.rand((n, 2), generator=g, device="cuda", dtype=torch.float64)
    if region == "disc":           # uniform in |xi| <= half
        rho, th = half * torch.sqrt(t[:, 0]), TWO_PI * t[:, 1]
        return torch.stack([rho * torch.cos(th), rho * torch.sin(th)], 1).contiguous()
    return t.mul_(2.0 * half).sub_(half)


STARSHADE = {"n_petals": 24, "a": 6.0, "R": 14.0, "b": 3.9, "q": 6.0, "z": 3.7e7, "pupil": 2.4}


def _starshade_resolution(lam):
    F = STARSHADE["R"] ** 2 / (lam * STARSHADE["z"])
    m, n_p = max(30, math.ceil(3 * F)), max(15, math.ceil(1.5 * F))
    return m, n_p, math.ceil(0.3 * STARSHADE["n_petals"] * n_p), m


def _starshade(lam, profile):
    s = STARSHADE
    m, n_p, n_d, m_d = _starshade_resolution(lam)
    return {"kind": "petals", "n_petals": s["n_petals"], "a": s["a"], "R": s["R"], "m": m,
            "n_p": n_p, "n_d": n_d, "m_d": m_d, "profile": profile}


def _lambdas(n):
    return [float(x) for x in np.linspace(400e-9, 1000e-9, n)] if n > 1 else [600e-9]


def _sweep_profile(seed):
    g = _npr(seed)
    return {"kind": "hg", "b": STARSHADE["b"] * (1 + 0.01 * g.standard_normal()),
            "q": STARSHADE["q"] * (1 + 0.01 * g.standard_normal())}


def _pupil_grid(n):
    return {"n1": n, "n2": n, "h": STARSHADE["pupil"] / n}


def _design_theta(c, seed):
    """Spline coefficients: the hyper-Gaussian at the Greville abscissae plus noise."""
    s, n = STARSHADE, c["n_coef"]
    t = np.concatenate([[s["a"]] * 4, np.linspace(s["a"], s["R"], n - 2)[1:-1], [s["R"]] * 4])
    grev = (t[1:n + 1] + t[2:n + 2] + t[3:n + 3]) / 3.0
    return np.exp(-((grev - s["a"]) / s["b"]) ** s["q"]) + 1e-3 * _npr(seed).standard_normal(n)


def _koch(c, seed):
    """Triangles of the level-L Koch snowflake, slightly turned, per level with its p."""
    turn = 0.05 * _npr(seed).standard_normal()
    ang = math.pi / 2 + TWO_PI / 3 * np.arange(3) + turn
    P = np.stack([np.cos(ang), np.sin(ang)], 1)
    tris = [P.reshape(1, 6)]
    A, B = P, np.roll(P, -1, axis=0)
    for _ in range(c["level"]):
        d0 = (B - A) / 3.0
        p1, p2 = A + d0, A + 2.0 * d0
        apex = p1 + np.stack([0.5 * d0[:, 0] + math.sqrt(0.75) * d0[:, 1],
                              -math.sqrt(0.75) * d0[:, 0] + 0.5 * d0[:, 1]], 1)
        tris.append(np.concatenate([p1, apex, p2], 1))
        A, B = (np.stack([A, p1, apex, p2], 1).reshape(-1, 2),
                np.stack([p1, apex, p2, B], 1).reshape(-1, 2))
    side = math.sqrt(3.0)
    return [{"kind": "triangles", "tri": t,
             "p": max(1, math.ceil(side / 3.0 ** k / (0.8 * c["lz"])))} for k, t in enumerate(tris)]


def _batch(c, seed):
    """Uneven random apertures: sizes fixed by the case, shapes and targets by the seed."""
    size = _npr(20105978, 5)
    N = np.exp(size.uniform(math.log(c["nodes_lo"]), math.log(c["nodes_hi"]), c["n"]))
    M = np.exp(size.uniform(math.log(c["targets_lo"]), math.log(c["targets_hi"]), c["n"]))
    problems = []
    for i in range(c["n"]):
        m = math.ceil(math.sqrt(N[i] / 10.0))
        par, R = _fourier_params("random", _npr(seed, 100 + i))
        fam = {"kind": "fourier", "params": par, "n_panels": math.ceil(N[i] / (16.0 * m)), "p": 16,
               "m": m}
        problems.append({"families": [fam], "lam": R * R / (1000.0 * math.sqrt(N[i] / 1e7)),
                         "z": 1.0})
    return problems, [int(x) for x in M]


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "grid":
        fams, lz = _aperture(c, seed)
        h = c["span"] / max(c["n1"], c["n2"])
        plan = Plan(fams, lz, 1.0, c["tol"], precision=c["precision"], output=c["output"],
                    grid={"n1": c["n1"], "n2": c["n2"], "h": h, "x0": c["x0"], "y0": c["y0"]},
                    recompute_nodes=c["recompute"], sync_status=c["sync"],
                    screen=_screen(c, seed))
        return {"kind": kind, "plan": plan}
    if kind == "scattered":
        fams, lz = _aperture(c, seed)
        b = c["half"]
        plan = Plan(fams, lz, 1.0, c["tol"], precision=c["precision"], output=c["output"],
                    box=(-b, b, -b, b), recompute_nodes=c["recompute"], sync_status=False)
        return {"kind": kind, "plan": plan, "targets": _targets(c["targets"], b, c["region"], seed)}
    if kind == "sweep":
        prof = _sweep_profile(seed)
        probs = [{"families": [_starshade(lam, prof)], "lam": lam, "z": STARSHADE["z"]}
                 for lam in _lambdas(c["n_lambda"])]
        plan = BatchPlan(probs, c["tol"], precision=c["precision"], output="occulter",
                         grid=_pupil_grid(c["n"]), recompute_nodes=True, sync_status=False)
        return {"kind": kind, "plan": plan}
    if kind == "design":
        theta = torch.tensor(_design_theta(c, seed), device="cuda", requires_grad=True)
        grid = _pupil_grid(c["n"])

        def make_plan(th):
            probs = [{"families": [_starshade(lam, {"kind": "bspline", "coefs": th})], "lam": lam,
                      "z": STARSHADE["z"]} for lam in _lambdas(c["n_lambda"])]
            return BatchPlan(probs, c["tol"], precision=c["precision"], output="occulter", grid=grid)

        return {"kind": kind, "theta": theta, "make_plan": make_plan}
    if kind == "shape_grad":
        fams, lz = _aperture(dict(c, shape="star"), seed)
        plan = Plan(fams, lz, 1.0, c["tol"], precision=c["precision"],
                    grid={"n1": c["n"], "n2": c["n"], "h": 3.0 / c["n"]}, sync_status=False)
        return {"kind": kind, "plan": plan}
    if kind == "koch":
        n = c["n"]
        plan = Plan(_koch(c, seed), c["lz"], 1.0, c["tol"], precision=c["precision"],
                    output="occulter", grid={"n1": n, "n2": n, "h": 3.0 / n}, recompute_nodes=True,
                    sync_status=False)
        return {"kind": kind, "plan": plan}
    problems, counts = _batch(c, seed)
    plan = BatchPlan(problems, c["tol"], precision=c["precision"], box=(-1.2, 1.2, -1.2, 1.2),
                     recompute_nodes=True, sync_status=False)
    return {"kind": kind, "plan": plan, "counts": counts,
            "targets": _targets(sum(counts), 1.2, "square", seed)}


def run(state):
    kind = state["kind"]
    if kind == "scattered":
        return state["plan"].eval(state["targets"])
    if kind == "batch":
        return state["plan"].eval(state["targets"], state["counts"])
    if kind == "design":
        u = profile_field(state["theta"], state["make_plan"])
        loss = (u.real ** 2 + u.imag ** 2).mean()
        return u.detach(), torch.autograd.grad(loss, state["theta"])[0]
    if kind == "shape_grad":
        u = state["plan"].eval()
        return u, state["plan"].grad_shape(u * (2.0 / u.numel()))
    return state["plan"].eval()


# ---------------------------------------------------------------- work
def _n_nodes(c):
    """Nodes of each problem."""
    if c["kind"] in ("sweep", "design"):
        out = []
        for lam in _lambdas(c["n_lambda"]):
            m, n_p, n_d, m_d = _starshade_resolution(lam)
            out.append(n_d * m_d + STARSHADE["n_petals"] * n_p * m)
        return out
    if c["kind"] == "koch":
        return [sum((1 if k == 0 else 3 * 4 ** (k - 1)) *
                    max(1, math.ceil(math.sqrt(3.0) / 3.0 ** k / (0.8 * c["lz"]))) ** 2
                    for k in range(c["level"] + 1))]
    if c["kind"] == "batch":
        return [f["families"][0]["n_panels"] * 16 * f["families"][0]["m"]
                for f in _batch(c, 0)[0]]
    return [c["n_panels"] * c.get("p", 16) * c["m"]]


def work(case):
    """Bytes: the targets read and the fields (and gradients) written.  Flops:
    per node and target the kernel's w^2 complex-by-real multiply-adds (w one
    digit each and one more), and per problem one FFT of the 2x oversampled
    product grid (of the field's bandwidth for scattered targets)."""
    c = case
    nodes = _n_nodes(c)
    real = 8 if c["precision"] == "fp64" else 4
    w2 = (math.ceil(-math.log10(c["tol"])) + 1) ** 2
    fft = lambda g: 5.0 * g * math.log2(max(g, 2.0))
    flops = sum(nodes) * w2 * 4.0
    if c["kind"] in ("scattered", "batch"):
        M = [c["targets"]] if c["kind"] == "scattered" else _batch(c, 0)[1]
        half = c.get("half", 1.2)
        for b, n in enumerate(nodes):
            F = c["fresnel"] if c["kind"] == "scattered" else 1000.0 * math.sqrt(n / 1e7)
            band = 4.0 * half * F          # cycles over the box, both directions
            flops += M[b] * w2 * 4.0 + fft((2.0 * band) ** 2)
        return {"bytes": sum(M) * (16 + 2 * real), "flops": flops}
    n1, n2 = c.get("n1", c.get("n")), c.get("n2", c.get("n"))
    points = n1 * n2 * len(nodes)
    flops += len(nodes) * fft(4.0 * n1 * n2)
    nbytes = points * 2 * real
    if c["kind"] in ("design", "shape_grad"):   # the gradient: read the field, a type-2 transform
        flops *= 2.0
        nbytes = 2 * nbytes + 8 * c.get("n_coef", 15)
    if c["kind"] == "koch":
        nbytes += 48 * sum(1 if k == 0 else 3 * 4 ** (k - 1) for k in range(c["level"] + 1))
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- exact values
def _leggauss(n, a, b):
    x, w = np.polynomial.legendre.leggauss(int(n))
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    return (torch.tensor(0.5 * (b - a) * (x + 1.0) + a, dtype=torch.float64, device=dev),
            torch.tensor(0.5 * (b - a) * w, dtype=torch.float64, device=dev))


def _t(x):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    return torch.as_tensor(np.asarray(x), dtype=torch.float64, device=dev)


def _dilate(X, Y, cross, m):
    a, wa = _leggauss(m, 0.0, 1.0)
    return ((X[:, None] * a).reshape(-1), (Y[:, None] * a).reshape(-1),
            (cross[:, None] * (a * wa)).reshape(-1))


def _fourier_nodes(par, n_panels, p, m):
    """Areal nodes of a Fourier boundary (par a FP64 tensor, differentiable)."""
    tq, wq = _leggauss(p, 0.0, TWO_PI / n_panels)
    t = (torch.arange(n_panels, dtype=torch.float64, device=tq.device)[:, None]
         * (TWO_PI / n_panels) + tq).reshape(-1)
    wt = wq.repeat(n_panels)
    k = torch.arange(1, (len(par) - 1) // 2 + 1, dtype=torch.float64, device=tq.device)
    r = par[0] + torch.cos(t[:, None] * k) @ par[1::2] + torch.sin(t[:, None] * k) @ par[2::2]
    return _dilate(r * torch.cos(t), r * torch.sin(t), wt * r * r, m)   # x V - y W = r^2 what


def _bspline(a, R, coefs, r):
    """Clamped uniform cubic B-spline at r (differentiable in coefs): Cox-de Boor."""
    n = len(coefs)
    knots = np.concatenate([[a] * 4, np.linspace(a, R, n - 2)[1:-1], [R] * 4])
    rr = r.cpu().numpy()
    B = ((rr[:, None] >= knots[None, :-1]) & (rr[:, None] < knots[None, 1:])).astype(float)
    for d in range(1, 4):
        nb = len(knots) - 1 - d
        N = np.zeros((len(rr), nb))
        for i in range(nb):
            u, v = knots[i + d] - knots[i], knots[i + d + 1] - knots[i + 1]
            if u > 0:
                N[:, i] += (rr - knots[i]) / u * B[:, i]
            if v > 0:
                N[:, i] += (knots[i + d + 1] - rr) / v * B[:, i + 1]
        B = N
    return _t(B) @ coefs


def _starshade_nodes(lam, A_of_r):
    s = STARSHADE
    m, n_p, n_d, m_d = _starshade_resolution(lam)
    t = TWO_PI * _t(np.arange(1, n_d + 1)) / n_d
    xd, yd, wd = _dilate(s["a"] * torch.cos(t), s["a"] * torch.sin(t),
                         torch.full_like(t, s["a"] ** 2 * TWO_PI / n_d), m_d)
    r, wr = _leggauss(m, s["a"], s["R"])
    q, wq = _leggauss(n_p, -math.pi / s["n_petals"], math.pi / s["n_petals"])
    A = A_of_r(r)
    th = (A[None, :] * q[:, None])[None] + (TWO_PI / s["n_petals"]) * _t(
        np.arange(s["n_petals"]))[:, None, None]
    x, y = (r * torch.cos(th)).reshape(-1), (r * torch.sin(th)).reshape(-1)
    w = ((r * wr * A)[None, :] * wq[:, None]).reshape(-1).repeat(s["n_petals"])
    return torch.cat([xd, x]), torch.cat([yd, y]), torch.cat([wd, w])


def _keys(s):
    s = s.abs()
    return torch.where(s <= 1, 1.5 * s ** 3 - 2.5 * s ** 2 + 1,
                       torch.where(s < 2, -0.5 * s ** 3 + 2.5 * s ** 2 - 4 * s + 2,
                                   torch.zeros_like(s)))


def _screen_at(scr, lam, x, y):
    """A exp(2 pi i OPD / lam) by cubic convolution of the samples."""
    x0, x1, y0, y1 = scr["box"]
    n2, n1 = scr["amp"].shape
    u = ((x - x0) * (n1 - 1) / (x1 - x0)).clamp(1.0, n1 - 2.0)
    v = ((y - y0) * (n2 - 1) / (y1 - y0)).clamp(1.0, n2 - 2.0)
    i, k = u.floor().long().clamp(max=n1 - 3), v.floor().long().clamp(max=n2 - 3)
    out = []
    for name in ("amp", "opd"):
        a, tot = _t(scr[name]), torch.zeros_like(x)
        for dk in (-1, 0, 1, 2):
            for di in (-1, 0, 1, 2):
                tot = tot + _keys(v - (k + dk)) * _keys(u - (i + di)) * a[k + dk, i + di]
        out.append(tot)
    return torch.polar(out[0], TWO_PI * out[1] / lam)


def _cis(ph):
    return torch.polar(torch.ones_like(ph), ph)


def _axis(n, h, x0):
    return _t(x0 + h * (np.arange(n) - n // 2))


def _product_sum(x, y, c, xi, eta, lz, chunk=32768):
    """sum_j c_j exp(-2 pi i (xi_a x_j + eta_b y_j) / lz) as (b, a), by matrix products."""
    out = torch.zeros((len(eta), len(xi)), dtype=torch.complex128, device=x.device)
    for i in range(0, len(x), chunk):
        s = slice(i, i + chunk)
        ex = _cis((-TWO_PI / lz) * x[s, None] * xi[None, :])
        ey = _cis((-TWO_PI / lz) * eta[:, None] * y[None, s])
        out = out + (ey * c[s]) @ ex
    return out


def _chirped(x, y, w, lz):
    return w * _cis((math.pi / lz) * (x * x + y * y))


def _field_on_grid(x, y, w, lz, xi, eta, output):
    v = _product_sum(x, y, _chirped(x, y, w, lz), xi, eta, lz)
    u = v * _cis((math.pi / lz) * (xi[None, :] ** 2 + eta[:, None] ** 2)) / (1j * lz)
    return 1.0 - u if output == "occulter" else u


def _cheb_rows(t, n):
    """Barycentric interpolation rows from the n Chebyshev points of [-1, 1] to t."""
    k = torch.arange(n, dtype=torch.float64, device=t.device)
    th = (2 * k + 1) * (math.pi / (2 * n))
    d = t[:, None] - torch.cos(th)[None, :]
    d = torch.where(d == 0, torch.full_like(d, 1e-300), d)
    q = torch.sin(th) * (1 - 2 * (k % 2)) / d
    return q / q.sum(1, keepdim=True)


def _field_at_targets(x, y, w, lz, targets, half, output):
    """The band-limited sum on a Chebyshev product grid over [-half, half]^2, interpolated."""
    cx, cy = 0.5 * (x.max() + x.min()), 0.5 * (y.max() + y.min())
    X = float(max((x - cx).abs().max(), (y - cy).abs().max()))
    kap = TWO_PI * X * half / lz
    p = int(kap + 13.0 * kap ** (1.0 / 3.0) + 40)
    if 8.0 * len(x) * p * p + 4.0 * len(targets) * p * p > EXACT_FLOPS:
        return None
    nodes = half * torch.cos((2 * _t(np.arange(p)) + 1) * (math.pi / (2 * p)))
    G = _product_sum(x - cx, y - cy, _chirped(x, y, w, lz), nodes, nodes, lz)
    out = []
    for i in range(0, len(targets), 65536):
        t = targets[i:i + 65536]
        L1, L2 = _cheb_rows(t[:, 0] / half, p), _cheb_rows(t[:, 1] / half, p)
        v = torch.complex(((L2 @ G.real) * L1).sum(1), ((L2 @ G.imag) * L1).sum(1))
        ph = (math.pi / lz) * (t[:, 0] ** 2 + t[:, 1] ** 2)
        ph = ph - (TWO_PI / lz) * (t[:, 0] * cx + t[:, 1] * cy)
        out.append(v * _cis(ph) / (1j * lz))
    u = torch.cat(out)
    return 1.0 - u if output == "occulter" else u


def exact(case, seed):
    c, kind = case, case["kind"]
    nodes = _n_nodes(c)
    if kind in ("grid", "sweep", "koch", "design", "shape_grad"):
        n1, n2 = c.get("n1", c.get("n")), c.get("n2", c.get("n"))
        if 8.0 * sum(nodes) * n1 * n2 > EXACT_FLOPS:
            return None
    if kind in ("grid", "scattered", "shape_grad"):
        fams, lz = _aperture(dict(c, shape=c.get("shape", "star")), seed)
        f = fams[0]
        if f["kind"] == "line_rule":
            x, y, w = _dilate(_t(f["X"]), _t(f["Y"]), _t(f["X"] * f["V"] - f["Y"] * f["W"]), f["m"])
        elif kind != "shape_grad":
            x, y, w = _fourier_nodes(_t(f["params"]), f["n_panels"], f["p"], f["m"])
    if kind == "scattered":
        if 32.0 * sum(nodes) * c["fresnel"] ** 2 > EXACT_FLOPS or c["targets"] > 4000000:
            return None
        return _field_at_targets(x, y, w, lz, _targets(c["targets"], c["half"], c["region"], seed),
                                 c["half"], c["output"])
    if kind == "grid":
        h = c["span"] / max(c["n1"], c["n2"])
        scr = _screen(c, seed)
        if scr is not None:
            w = w * _screen_at(scr, lz, x, y)
        return _field_on_grid(x, y, w, lz, _axis(c["n1"], h, c["x0"]), _axis(c["n2"], h, c["y0"]),
                              c["output"])
    if kind == "koch":
        xs, ys, ws = [], [], []
        for f in _koch(c, seed):
            T = _t(f["tri"])
            s, sw = _leggauss(f["p"], 0.0, 1.0)
            v0, d1, e = T[:, 0:2], T[:, 2:4] - T[:, 0:2], T[:, 4:6] - T[:, 2:4]
            rel = d1[:, None, :] + s[None, :, None] * e[:, None, :]
            pt = v0[:, None, None, :] + s[None, None, :, None] * rel[:, :, None, :]
            cr = (d1[:, 0] * e[:, 1] - d1[:, 1] * e[:, 0])[:, None, None]
            xs.append(pt[..., 0].reshape(-1))
            ys.append(pt[..., 1].reshape(-1))
            ws.append((cr * sw[None, :, None] * (s * sw)[None, None, :]).reshape(-1))
        ax = _axis(c["n"], 3.0 / c["n"], 0.0)
        return _field_on_grid(torch.cat(xs), torch.cat(ys), torch.cat(ws), c["lz"], ax, ax,
                              "occulter")
    if kind == "sweep":
        prof, ax = _sweep_profile(seed), _axis(c["n"], STARSHADE["pupil"] / c["n"], 0.0)
        A = lambda r: torch.exp(-((r - STARSHADE["a"]) / prof["b"]) ** prof["q"])
        return torch.stack([_field_on_grid(*_starshade_nodes(lam, A), lam * STARSHADE["z"], ax, ax,
                                           "occulter") for lam in _lambdas(c["n_lambda"])])
    if kind == "design":
        th = _t(_design_theta(c, seed)).requires_grad_(True)
        ax = _axis(c["n"], STARSHADE["pupil"] / c["n"], 0.0)
        A = lambda r: _bspline(STARSHADE["a"], STARSHADE["R"], th, r)
        us, g = [], torch.zeros_like(th)
        for lam in _lambdas(c["n_lambda"]):
            u = _field_on_grid(*_starshade_nodes(lam, A), lam * STARSHADE["z"], ax, ax, "occulter")
            loss = (u.real ** 2 + u.imag ** 2).sum() / (c["n_lambda"] * c["n"] ** 2)
            g = g + torch.autograd.grad(loss, th)[0]
            us.append(u.detach())
        return torch.stack(us), g
    if kind == "shape_grad":
        par = _t(f["params"]).requires_grad_(True)
        ax = _axis(c["n"], 3.0 / c["n"], 0.0)
        u = _field_on_grid(*_fourier_nodes(par, f["n_panels"], f["p"], f["m"]), lz, ax, ax,
                           "aperture")
        g = torch.autograd.grad((u.real ** 2 + u.imag ** 2).mean(), par)[0]
        return u.detach(), g
    return None
