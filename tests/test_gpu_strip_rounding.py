"""Rounding of the strip-sorted spreading against the tile kernel's.

Every addition to the grid rounds a cell's whole sum, so plans whose records
share a few cells show how often a kernel adds: distances from the
deterministic mode (exact fixed-point sums of the same records) over repeats
of the default plan and of the tile kernel (max_spin set).  What is compared is
their quotient's geometric mean over the plans of a group.  A distance is that of a
field or gradient to which some ten (gradients: two) cells or modes contribute
independently, so the logarithm of its root mean square over 8 repeats
scatters by 1 / sqrt(2 * 8 * 10) = 0.08 (gradients 0.18) and a group of n
quotients by sqrt(2 / n) times that; the bars lie four such deviations above 1
(and 1.15 at least: a strip's rows close with one addition more than a tile).
20 repeats are taken, as a gradient's error may lie in one mode alone."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

REPEATS = 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _quotients(make):
    """make(**options) -> outputs; per output rms(default) / rms(tiles)."""
    exact = make(deterministic=True)
    rms = lambda kw: np.sqrt(np.mean([[float((u - e).norm() / e.norm()) ** 2
                                       for u, e in zip(make(**kw), exact)]
                                      for _ in range(REPEATS)], axis=0))
    return rms({}) / rms({"max_spin": 1 << 22})


def _held(q, deviation):
    """The quotients' geometric mean against four deviations of it above 1."""
    assert np.exp(np.mean(np.log(q))) <= max(1.15, np.exp(4 * deviation * np.sqrt(2.0 / len(q))))


def _design(n_lambda, n, prec, **opts):
    from paper_2010_05978_gb300 import BatchPlan
    lams = tuple(np.linspace(400e-9, 1000e-9, n_lambda)) if n_lambda > 1 else (600e-9,)
    _, probs, grid, _ = W.spline_starshade("c4", n_coef=60, lams=lams, ngrid=n)
    probs = [{"families": [p["family"]], "lam": p["lam"], "z": p["z"]} for p in probs]

    def make(**kw):
        p = BatchPlan(probs, 1e-6, precision=prec, output="occulter", grid=grid, **opts, **kw)
        u = p.eval()
        return u, p.grad_profile(u * (2.0 / u.numel()))

    return make


DESIGNS = [(nl, n) for nl in (1, 2, 4, 8) for n in (48, 49, 64, 128, 256)]


def test_starshade_designs_fp32():
    q = np.array([_quotients(_design(nl, n, "fp32")) for nl, n in DESIGNS])
    _held(q[:, 0], 0.08)
    _held(q[:, 1], 0.18)


@pytest.mark.parametrize("prec,opts,designs", [
    ("fp32", {"sigma": 1.25}, [(1, 64), (4, 128), (8, 128)]),
    ("fp32", {"kernel_w": 9}, [(2, 64), (4, 128), (8, 128)]),
    ("fp32", {"kernel_w": 10}, [(2, 64), (4, 128), (8, 128)]),
    ("fp32", {"kernel_w": 16}, [(2, 64), (4, 128), (8, 128)]),
    ("fp64", {}, [(1, 64), (2, 128), (6, 128), (8, 64)]),
])
def test_wide_kernels_and_fp64(prec, opts, designs):
    q = np.array([_quotients(_design(nl, n, prec, **opts)) for nl, n in designs])
    _held(q[:, 0], 0.08)
    _held(q[:, 1], 0.18)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_starshade_beside_a_disc_that_covers_the_grid(prec):
    from paper_2010_05978_gb300 import BatchPlan

    def mixed(n, n_coef):
        _, probs, grid, _ = W.spline_starshade("c4", n_coef=n_coef, lams=(600e-9,), ngrid=n)
        s = probs[0]
        disc = W.fourier_family([0.45 * s["lam"] * s["z"] / grid["h"], 0.0, 0.0], 200, 16, 100)
        both = [{"families": [f], "lam": s["lam"], "z": s["z"]} for f in (disc, s["family"])]

        def make(**kw):
            p = BatchPlan(both, 1e-6, precision=prec, output="occulter", grid=grid, **kw)
            u = p.eval()
            return u[0], u[1], p.grad_profile(u * (2.0 / u.numel()))

        return _quotients(make)

    q = np.array([mixed(n, n_coef) for n, n_coef in ((128, 60), (128, 30), (100, 60), (112, 90))])
    _held(q[:, :2].ravel(), 0.08)
    _held(q[:, 2], 0.18)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_nodes_with_a_third_on_one_point(prec):
    from paper_2010_05978_gb300 import Plan

    def case(n):
        g = W.rng(9, n)
        x, y = g.uniform(-1, 1, n), g.uniform(-1, 1, n)
        x[: n // 3], y[: n // 3] = 0.25, -0.125
        fam = {"kind": "nodes", "x": x, "y": y, "w": g.uniform(0.5, 1.5, n)}
        t = torch.tensor(g.uniform(-1, 1, (500, 2)), device="cuda")
        return lambda **kw: [Plan([fam], 0.07, 1.0, 1e-6, precision=prec, box=(-1, 1, -1, 1),
                                  recompute_nodes=True, **kw).eval(t)]

    q = np.concatenate([_quotients(case(n)) for n in (10000, 20000, 40000, 80000, 155647, 155649)])
    _held(q, 0.18)   # one point: its cells' errors come together


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("w", [2, 4, 5, 8, 9, 10, 13, 16])
def test_blocks_that_merge_their_rows(prec, w):
    # every kernel width, nodes that wrap round both edges of the grid, half of
    # them on 40 points (runs of warps on one strip), record counts at the
    # edges of a batch, of a block and of the widest blocks
    from paper_2010_05978_gb300 import Plan
    for n in (1, 33, 511, 513, 1025, 4096, 4607, 4609, 4641, 30000, 117000):
        g = W.rng(12, 100 * n + w)
        x, y = g.uniform(-1, 1, n), g.uniform(-1, 1, n)
        k = g.integers(0, min(40, n), n // 2)
        x[: n // 2], y[: n // 2] = x[k], y[k]
        fam = {"kind": "nodes", "x": x, "y": y, "w": g.uniform(0.5, 1.5, n)}
        make = lambda **kw: Plan([fam], 0.05, 1.0, 1e-6, precision=prec, kernel_w=w,
                                 grid=W.grid_spec(101, 77, 0.03), **kw).eval()
        u, v, t = make(), make(deterministic=True), make(max_spin=1 << 22)
        rel = lambda a: float((a - v).norm() / v.norm())
        # repeats' bound, or twice the tile kernel's own distance where the
        # deconvolution amplifies rounding beyond it (as in test_gpu_strips)
        assert rel(u) <= max({"fp32": 2e-6, "fp64": 1e-13}[prec], 2.0 * rel(t))
