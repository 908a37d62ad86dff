"""Strip-sorted spreading (csrc/strips.cuh) against the tile kernel.

The deterministic option sorts by tiles and sums in fixed point, so the same
plan with it on is an independent grid of the same records, free of rounding
in its sums.  Outputs agree with it to the rounding of the floating-point
sums: as a repeat of one plan does (2e-6 relative L2 in FP32, 1e-13 in FP64),
or, where the deconvolution amplifies that rounding beyond it (sigma = 5/4 and
long runs on one point or forced widths), within twice the distance of the
floating-point tile kernel, which a set max_spin selects.  Every kernel width, nodes that
wrap round the periodic grid in both directions, record counts at the edges
of a batch and of a warp's range, dense single cells, stacked problems, and
evaluations after a gradient has used the grid."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BAR = {"fp32": 2e-6, "fp64": 1e-13}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _rel(a, b):
    return float((a - b).norm() / b.norm())


def _agree(make, prec, parts=lambda o: [o]):
    """make(**options) -> outputs: default against deterministic and tiles."""
    for u, v, t in zip(*(parts(make(**kw)) for kw in ({}, {"deterministic": True},
                                                      {"max_spin": 1 << 22}))):
        assert _rel(u, v) <= max(BAR[prec], 2.0 * _rel(t, v))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("w", [2, 3, 5, 7, 8, 9, 10, 12, 13, 16])
def test_widths_and_wrap(prec, w):
    # the disc of radius 1 at h / lz = 0.6 covers 1.2 periods of the grid:
    # supports wrap round both edges and the corners
    from paper_2010_05978_gb300 import Plan
    fam = W.fourier_family([1.0], 40, 16, 37)
    make = lambda **kw: Plan([fam], 0.05, 1.0, 1e-6, precision=prec, kernel_w=w,
                             grid=W.grid_spec(101, 77, 0.03), **kw).eval()
    _agree(make, prec)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 4096, 155649, 311297])
def test_record_counts_scattered(prec, n):
    # explicit nodes, a third of them on one point; type 3, regenerated twice
    from paper_2010_05978_gb300 import Plan
    g = W.rng(9, n)
    x, y = g.uniform(-1, 1, n), g.uniform(-1, 1, n)
    x[: n // 3], y[: n // 3] = 0.25, -0.125
    fam = {"kind": "nodes", "x": x, "y": y, "w": g.uniform(0.5, 1.5, n)}
    t = torch.tensor(g.uniform(-1, 1, (500, 2)), device="cuda")

    def make(**kw):
        p = Plan([fam], 0.07, 1.0, 1e-6, precision=prec, box=(-1, 1, -1, 1),
                 recompute_nodes=True, **kw)
        p.eval(t)
        return p.eval(t)

    _agree(make, prec)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_stacked_problems_and_grid_restored_after_a_gradient(prec):
    # three problems' grids stacked by rows: a folded disc that wraps at the
    # top and bottom, a small one in a few cells, another far off centre
    from paper_2010_05978_gb300 import BatchPlan
    fams = [W.fourier_family([1.0, 0.0, 0.0], 24, 16, 30),
            W.fourier_family([0.02, 0.0, 0.0], 24, 16, 30),
            W.fourier_family([0.3, 0.05, 0.0], 24, 16, 30, cx=0.6, cy=-0.7)]
    probs = [{"families": [f], "lam": lam, "z": 1.0} for f, lam in zip(fams, (0.05, 0.05, 0.08))]

    def make(**kw):
        p = BatchPlan(probs, 1e-6, precision=prec, grid=W.grid_spec(90, 100, 0.03), **kw)
        u = p.eval().clone()
        p.grad_shape(u)
        again = p.eval().clone()
        p.nodes()
        return u, again, p.eval()

    _agree(make, prec, parts=lambda outs: [u[b] for u in outs for b in range(3)])


def test_memory_cap_keeps_what_fitted():
    # a cap exactly at the tile sort's size is still accepted
    from paper_2010_05978_gb300 import Plan
    fam = {"kind": "nodes", "x": [-0.9, 0.9], "y": [-0.9, 0.9], "w": [1.0, 1.0]}
    kw = dict(precision="fp32", grid=W.grid_spec(100, 100, 0.03))
    by_tiles = Plan([fam], 0.1, 1.0, 1e-6, max_spin=1 << 22, **kw)   # the ready-flag form
    cap = by_tiles.info()["device_bytes"]
    u = Plan([fam], 0.1, 1.0, 1e-6, max_device_bytes=cap, **kw).eval()
    assert _rel(u, by_tiles.eval()) <= BAR["fp32"]
