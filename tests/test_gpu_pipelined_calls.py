"""A call's kernels in a row take no longer than one by one.

Stage times are recorded with an event between the kernels, which serialises
them; without events a kernel may start while the one before it ends.  Its
blocks must not take places that make the pass itself slower."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,n", [("fp64", 400), ("fp64", 512), ("fp64", 700), ("fp32", 512),
                                    ("fp32", 1000)])
def test_calls_in_a_row(prec, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import Plan, build
    build.build()
    torch.cuda.set_device(0)
    fam = W.fourier_family(W.STAR_PARAMS, 48, 16, 60)
    p = Plan([fam], 1.69 / 40, 1.0, 1e-6 if prec == "fp32" else 1e-10, precision=prec,
             grid=W.grid_spec(n, n, 3.0 / n), sync_status=False)
    u = p.eval()
    p.set_timing(True)
    stages = []
    for _ in range(30):
        p.eval(out=u)
        torch.cuda.synchronize()
        stages.append(sum(p.stage_times().values()))
    p.set_timing(False)
    calls = []
    for _ in range(10):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(20):
            p.eval(out=u)
        b.record()
        torch.cuda.synchronize()
        calls.append(a.elapsed_time(b) / 20)
    assert np.median(calls) <= np.median(stages)
