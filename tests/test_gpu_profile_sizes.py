"""Profile gradients over the sizes of the profile data: values against the
gradient of fewer parameters by the chain rule, and a time that does not grow
with parameters that no radius touches."""
import time

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


def _plan(profile, m):
    from paper_2010_05978_gb300 import Plan
    fam = W.petal_family(6, 0.4, 1.0, profile, m, 12, 40, 20)
    return Plan([fam], 0.05, 1.0, 1e-12, precision="fp64", grid=W.grid_spec(40, 36, 0.05))


def _basis(a, R, n, r):
    """Clamped uniform cubic B-splines at r by the Cox-de Boor recursion, (len(r), n)."""
    t = np.concatenate([[a] * 4, np.linspace(a, R, n - 2)[1:-1], [R] * 4])
    B = ((r[:, None] >= t[None, :-1]) & (r[:, None] < t[None, 1:])).astype(float)
    for d in range(1, 4):
        u, v = t[d:-1] - t[:-1 - d], t[1 + d:] - t[1:-d]
        left = np.where(u > 0, (r[:, None] - t[None, :-1 - d]) / np.where(u > 0, u, 1), 0) * B[:, :-1]
        right = np.where(v > 0, (t[None, 1 + d:] - r[:, None]) / np.where(v > 0, v, 1), 0) * B[:, 1:]
        B = left + right
    return B


@pytest.mark.parametrize("m", [1, 2, 255, 256, 257, 600])
@pytest.mark.parametrize("n", [4, 5, 20, 700, 5000])
def test_spline_gradient_is_the_tables_gradient_times_the_basis(m, n):
    # A(r_l) = sum_j c_j B_j(r_l): the same values as a table have the same
    # field, and dL/dc = B^T dL/dA.  FP64 sums of at most 256 terms at a time
    # and of m in all, each product rounded a few times: 1e-13 (m) of the norm;
    # the two plans' fields repeat to 1e-13
    a, R = 0.4, 1.0
    x, _ = np.polynomial.legendre.leggauss(m)
    B = _basis(a, R, n, 0.5 * (R - a) * (x + 1) + a)
    c = 0.5 + 0.3 * W.rng(13, n).random(n)
    spline, table = _plan({"kind": "bspline", "coefs": c}, m), _plan({"kind": "table", "A": B @ c}, m)
    g = W.rng(13, 1)
    gamma = torch.tensor(g.standard_normal((36, 40)) + 1j * g.standard_normal((36, 40)), device="cuda")
    got = spline.grad_profile(gamma).cpu().numpy()
    ref = B.T @ table.grad_profile(gamma).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-11 * np.linalg.norm(ref)


def test_time_does_not_grow_with_untouched_parameters():
    # 200 radii touch at most 800 of 200,000 coefficients, whose gradient is
    # otherwise the clearing of 1.6 MB: a few microseconds
    def seconds(n):
        p = _plan({"kind": "bspline", "coefs": np.full(n, 0.6)}, 200)
        gamma = torch.ones((36, 40), dtype=torch.complex128, device="cuda")
        best = 1e9
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            p.grad_profile(gamma)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    assert seconds(200000) <= 3.0 * seconds(200)
