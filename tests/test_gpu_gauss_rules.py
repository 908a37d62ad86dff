"""Gauss-Legendre rules of the node kernels at the sizes where they change:
the recurrence with and without its table, and orders at which the first
Newton step is already small (n >= 30,400), against Newton's iteration in
extended precision on the host.

Read through a circle's dilation rule of one panel and one boundary node (at
angle pi): node l lies at -alpha_l with weight 2 pi alpha_l what_l.  Bars: the
root is exact to rounding, and x = 1 - 2 alpha enters the end weights as 1 /
(1 - x^2), so a relative error of eps n^2 is one ulp of x; a root is off by an
ulp of x (2.2e-16 in alpha at most, twice that with the mapping and the node's
own products)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _rule(n, i):
    """Roots i (from the upper end) on (-1, 1), as 1 - x, and their weights."""
    N = np.longdouble(n)
    th = np.pi * (i + np.longdouble(0.75)) / (N + np.longdouble(0.5))
    x = (1 - (N - 1) / (8 * N ** 3)) * np.cos(th)
    for _ in range(5):
        p0, p1 = np.ones_like(x), x.copy()
        for j in range(1, n):
            J = np.longdouble(j)
            p0, p1 = p1, ((2 * J + 1) * x * p1 - J * p0) / (J + 1)
        dp = N * (x * p1 - p0) / (x * x - 1)
        w = 2 / ((1 - x * x) * dp * dp)
        x = x - p1 / dp
    return x, w


@pytest.mark.parametrize("n", [16, 3072, 3073, 6143, 6144, 31000, 65536])
def test_rules(n):
    from paper_2010_05978_gb300 import Plan
    p = Plan([W.fourier_family([1.0], 1, 1, n)], 0.05, 1.0, 1e-6, precision="fp64",
             grid=W.grid_spec(32, 32, 0.03))
    x, _, w = (t.cpu().numpy() for t in p.nodes())
    order = np.argsort(-x)               # alpha ascending
    alpha, what = -x[order], w[order] / (2 * np.pi * -x[order])
    assert len(alpha) == n and np.all(np.diff(alpha) > 0)
    i = np.unique(np.r_[0:min(12, n // 2), np.linspace(0, n // 2 - 1, 12).astype(int)])
    rx, rw = _rule(n, i)                 # upper roots; the lower ones mirror them
    assert np.max(np.abs(alpha[i] - (1 - rx) / 2)) <= 5e-16
    assert np.max(np.abs(alpha[n - 1 - i] - (1 + rx) / 2)) <= 5e-16
    bar = 2.2e-16 * (n * n + 50.0 * np.sqrt(n))
    assert np.max(np.abs(what[n - 1 - i] / (rw / 2) - 1)) <= bar
    assert abs(what.sum() - 1) <= 1e-13 * np.sqrt(n)
