"""The FP32 gradient of starshade designs against FP64, in the deterministic
mode (so that the transforms' rounding is all that differs from one radix
order to another).

Lengths 160, 288 and 480, whose radices may be ordered in several ways.  With
the order 16, 8, 4, 2, 3, 5 the errors are (2.5 .. 4.9)e-7, 3.62e-7 in root
mean square; with the fewest stages instead (16, 10; 12, 12, 2; 16, 15, 2)
each is larger, by up to 1.7 times, 4.64e-7 together.  The bar is a tenth
above the former."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_profile_gradient_of_designs_with_lengths_of_several_orders():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import BatchPlan, build
    build.build()
    torch.cuda.set_device(0)
    err = []
    for n, n_lambda, n_coef in ((71, 6, 60), (74, 8, 120), (133, 7, 60), (136, 4, 60),
                                (140, 5, 150), (129, 3, 40), (205, 4, 60), (230, 2, 90)):
        lams = tuple(np.linspace(400e-9, 1000e-9, n_lambda))
        _, probs, grid, _ = W.spline_starshade("c4", n_coef=n_coef, lams=lams, ngrid=n)
        probs = [{"families": [p["family"]], "lam": p["lam"], "z": p["z"]} for p in probs]
        g = []
        for tol, kw in ((1e-6, {"deterministic": True}), (1e-12, {"precision": "fp64"})):
            p = BatchPlan(probs, tol, output="occulter", grid=grid, **kw)
            u = p.eval()
            g.append(p.grad_profile(u * (2.0 / u.numel())).view(n_lambda, n_coef).sum(0))
        assert p.info()["nfft1"] in (160, 288, 480)
        err.append(float((g[0] - g[1]).norm() / g[1].norm()))
    assert np.sqrt(np.mean(np.square(err))) <= 1.1 * 3.62e-7
