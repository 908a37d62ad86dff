"""The ends of the FFT passes' range: the longest lengths that one pass takes
(12,960 points in rows, 13,122 and more in columns in FP32; 6,400 in FP64), and
a forced split of a length that has none.  References: the direct sum; bars as
in test_gpu_fft_lengths."""
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


def _nodes(stream, N=300):
    g = W.rng(15, stream)
    return g.uniform(-1, 1, N), g.uniform(-1, 1, N), g.uniform(0.5, 1.5, N) / N


cis = lambda a: np.exp(1j * a)


@pytest.mark.parametrize("prec,n1,n2", [("fp32", 6480, 33), ("fp32", 33, 4096), ("fp64", 3200, 33),
                                        ("fp64", 33, 3200)])
def test_longest_single_passes_on_grids(prec, n1, n2):
    from paper_2010_05978_gb300 import Plan
    x, y, w = _nodes(n1)
    lz, h = 0.02, 2.0 / max(n1, n2)
    p = Plan([{"kind": "nodes", "x": x, "y": y, "w": w}], lz, 1.0, 1e-6 if prec == "fp32" else 1e-12,
             precision=prec, sigma=2.0, grid=W.grid_spec(n1, n2, h))
    assert max(p.info()["nfft1"], p.info()["nfft2"]) == 2 * max(n1, n2)
    u = p.eval().cpu().numpy()
    xi, eta = (h * (np.arange(n) - n // 2) for n in (n1, n2))
    v = (cis(-2 * np.pi / lz * np.outer(eta, y)) * (w * cis(np.pi / lz * (x * x + y * y)))) @ \
        cis(-2 * np.pi / lz * np.outer(x, xi))
    ref = v * cis(np.pi / lz * (xi[None, :] ** 2 + eta[:, None] ** 2)) / (1j * lz)
    assert np.linalg.norm(u - ref) / np.linalg.norm(ref) <= (1e-6 if prec == "fp32" else 1e-10)


def test_longest_single_pass_columns_of_scattered_plans():
    # under a memory cap FP32 columns stay one pass up to 13,671 points
    from paper_2010_05978_gb300 import Plan
    x, y, w = _nodes(1)
    lz, M = 0.0019, 300
    t = W.rng(15, 2).uniform(-1, 1, (M, 2)) * [0.02, 1.5]
    p = Plan([{"kind": "nodes", "x": x, "y": y, "w": w}], lz, 1.0, 1e-6, box=(-0.02, 0.02, -1.5, 1.5),
             max_device_bytes=1 << 34)
    assert 12500 < p.info()["nfft2"] <= 13671
    u = p.eval(torch.tensor(t, device="cuda")).cpu().numpy()
    d2 = (t[:, :1] - x) ** 2 + (t[:, 1:] - y) ** 2
    ref = (w * cis(np.pi / lz * d2)).sum(1) / (1j * lz)
    assert np.linalg.norm(u - ref) / np.linalg.norm(ref) <= 1e-6


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_forced_split_of_a_length_that_has_none_runs_in_one_pass(prec):
    # 50 points: 2 x 25 and 5 x 10 each leave a factor of one stage
    from paper_2010_05978_gb300 import Plan
    x, y, w = _nodes(3)
    t = torch.tensor(W.rng(15, 4).uniform(-1, 1, (200, 2)), device="cuda")
    make = lambda split: Plan([{"kind": "nodes", "x": x, "y": y, "w": w}], 1.0, 1.0, 1e-6,
                              precision=prec, sigma=1.55, box=(-1, 1, -1, 1), fft_split_above=split)
    p = make(16)
    assert p.info()["nfft1"] == 50
    u, v = p.eval(t), make(0).eval(t)
    # the same transform twice: repeats' bounds
    assert float((u - v).norm() / v.norm()) <= (2e-6 if prec == "fp32" else 1e-13)
