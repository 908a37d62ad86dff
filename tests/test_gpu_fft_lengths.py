"""FFT passes over the radices and line shapes that their plans can take.

Type-1 plans with sigma = 2 transform lengths nf = 2 n: the pairs below cover
every radix (16 .. 2, and 15, 12, 10, 9 in FP32), two to five stages, several
short rows per block, odd numbers of columns, and the longest single passes;
with fft_split_above the same lengths run as four steps.  The reference is the
direct sum by matrix products; the bars are the modes' own contracts (relative
L2 at most tol = 1e-6 in FP32, 1e-10 at tol = 1e-12 in FP64)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (n1, n2): row length 2 n1, column length 2 n2 (multiples of 32)
PAIRS = [(32, 48), (80, 144), (160, 240), (432, 720), (600, 200), (1000, 64), (1728, 33),
         (33, 1875), (37, 3000), (3240, 50)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("split", [0, 64])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n1,n2", PAIRS)
def test_lengths(n1, n2, prec, split):
    from paper_2010_05978_gb300 import Plan
    g = W.rng(10, n1 * 10000 + n2)
    N, lz, h = 300, 0.02, 2.0 / max(n1, n2)
    x, y, w = g.uniform(-1, 1, N), g.uniform(-1, 1, N), g.uniform(0.5, 1.5, N) / N
    p = Plan([{"kind": "nodes", "x": x, "y": y, "w": w}], lz, 1.0, 1e-6 if prec == "fp32" else 1e-12,
             precision=prec, sigma=2.0, grid=W.grid_spec(n1, n2, h), fft_split_above=split)
    u = p.eval().cpu().numpy()
    xi, eta = (h * (np.arange(n) - n // 2) for n in (n1, n2))
    cis = lambda a: np.exp(1j * a)
    v = (cis(-2 * np.pi / lz * np.outer(eta, y)) * (w * cis(np.pi / lz * (x * x + y * y)))) @ \
        cis(-2 * np.pi / lz * np.outer(x, xi))
    ref = v * cis(np.pi / lz * (xi[None, :] ** 2 + eta[:, None] ** 2)) / (1j * lz)
    assert np.linalg.norm(u - ref) / np.linalg.norm(ref) <= (1e-6 if prec == "fp32" else 1e-10)


@pytest.mark.parametrize("cap", [0, 1 << 34])
def test_long_columns_of_scattered_plans(cap):
    # FP32 scattered plans split columns beyond 2,400 points into four steps;
    # a memory cap keeps the single pass (no scratch grid)
    from paper_2010_05978_gb300 import Plan
    g = W.rng(11, 1)
    N, lz, M = 300, 0.0085, 400
    x, y, w = g.uniform(-1, 1, N), g.uniform(-1, 1, N), g.uniform(0.5, 1.5, N) / N
    t = g.uniform(-1.5, 1.5, (M, 2))
    p = Plan([{"kind": "nodes", "x": x, "y": y, "w": w}], lz, 1.0, 1e-6, box=(-1.5, 1.5, -1.5, 1.5),
             max_device_bytes=cap)
    assert p.info()["nfft2"] > 2400
    u = p.eval(torch.tensor(t, device="cuda")).cpu().numpy()
    r2 = (t[:, 0, None] - x) ** 2 + (t[:, 1, None] - y) ** 2
    ref = (w * np.exp(1j * np.pi / lz * r2)).sum(1) / (1j * lz)
    assert np.linalg.norm(u - ref) / np.linalg.norm(ref) <= 1e-6
