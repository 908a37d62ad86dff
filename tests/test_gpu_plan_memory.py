"""Device memory of plans: what info() reports is what is held, small plans hold
little, and plans that fit in the memory that is left are not refused."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("kind", ["grid", "scattered"])
def test_held_memory_is_reported_and_small_plans_hold_little(kind):
    from paper_2010_05978_gb300 import Plan
    fam = W.fourier_family([1.0, 0.02, 0.01], 12, 8, 12)
    where = {"grid": {"grid": W.grid_spec(24, 24, 0.05)}, "scattered": {"box": (-1, 1, -1, 1)}}[kind]
    # FP64: FP32 scattered plans have a stream of their own, which takes device
    # memory (0.6 MB) that is no allocation of the plan's
    make = lambda **kw: Plan([fam], 0.5, 1.0, 1e-6, precision="fp64", **where, **kw)
    make().close()
    exact = make(max_device_bytes=1 << 40).info()["device_bytes"]   # every allocation its own
    before = _free()
    plans = [make() for _ in range(200)]
    held, reported = before - _free(), sum(p.info()["device_bytes"] for p in plans)
    # cudaMalloc takes memory from the device 2 MB at a time
    assert held <= 1.05 * reported + 4 * MB
    # at most as much again in the slabs as the tables in them, and one slab more
    assert plans[0].info()["device_bytes"] <= 2 * exact + (64 << 10)


def test_a_plan_that_fits_without_its_scratch_grid_is_not_refused():
    # FP32 scattered plans put columns above 2,400 points through a scratch grid
    # of the FFT grid's size; with room for the plan but not for it, they take
    # single passes.  The rest of the memory is taken by one tensor
    from paper_2010_05978_gb300 import BatchPlan, Plan
    g = W.rng(14, 0)
    n, M = 300, 400
    x, y, w = g.uniform(-1, 1, n), g.uniform(-1, 1, n), g.uniform(0.5, 1.5, n) / n
    fam = {"kind": "nodes", "x": x, "y": y, "w": w}
    t = torch.tensor(g.uniform(-1.5, 1.5, (M, 2)), device="cuda")
    box = (-1.5, 1.5, -1.5, 1.5)
    one = lambda **kw: Plan([fam], 0.0035, 1.0, 1e-6, box=box, **kw)
    two = lambda **kw: BatchPlan([{"families": [fam], "lam": 0.0035, "z": 1.0}] * 2, 1e-6, box=box, **kw)
    run = {one: lambda p: p.eval(t), two: lambda p: p.eval(torch.cat([t, t]), [M, M])}
    for make in (one, two):
        p = make(fft_split_above=1 << 30)
        single, ref = p.info()["device_bytes"], run[make](p)
        p.close()
        p = make()
        split = p.info()["device_bytes"]
        assert float((run[make](p) - ref).norm() / ref.norm()) <= 2e-6
        p.close()
        assert split > single + 100 * MB
        torch.cuda.empty_cache()
        hog = torch.empty(_free() - (single + split) // 2, dtype=torch.uint8, device="cuda")
        try:
            p = make()
            assert p.info()["device_bytes"] < single + 8 * MB
            out = run[make](p)
            p.close()
        finally:
            del hog
            torch.cuda.empty_cache()
        assert float((out - ref).norm() / ref.norm()) <= 2e-6


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_a_capped_gradient_takes_only_its_own_arrays(prec):
    # a starshade on a few cells (direct column DFT, which has no stage
    # twiddles); a cap with room for the adjoint's two grids and the nodes'
    # contributions is enough
    from paper_2010_05978_gb300 import Plan
    _, probs, grid, _ = W.spline_starshade("c4", n_coef=20, lams=(600e-9,), ngrid=64)
    q = probs[0]
    make = lambda cap: Plan([q["family"]], q["lam"], q["z"], 1e-6, precision=prec, output="occulter",
                            grid=grid, max_device_bytes=cap)
    p = make(1 << 40)
    u = p.eval()
    info, cs = p.info(), 8 if prec == "fp32" else 16
    own = cs * 64 * 64 + cs * 64 * info["nf1"] + 8 * info["n_nodes"]
    rest = 8 * 8   # where the family's gradient lies, and its number
    g = p.grad_profile(u)
    assert p.info()["device_bytes"] - info["device_bytes"] <= own + rest
    p = make(info["device_bytes"] + own + rest)
    got = p.grad_profile(p.eval())
    again = p.grad_profile(p.eval())
    ref = make(0)
    ref = ref.grad_profile(ref.eval())
    for v in (g, got, again):   # gradients repeat as their fields do
        assert float((v - ref).norm() / ref.norm()) <= (2e-5 if prec == "fp32" else 1e-11)


def test_split_tiles_are_those_that_the_plan_splits():
    from paper_2010_05978_gb300 import Plan
    fam = W.fourier_family([1.0, 0.0, 0.0], 64, 16, 64)
    make = lambda **kw: Plan([fam], 0.1, 1.0, 1e-6, grid=W.grid_spec(100, 100, 0.03), **kw)
    assert make().info()["split_tiles"] == 0                    # by column strips
    assert make(max_spin=1 << 22).info()["split_tiles"] > 0     # by tiles
    assert make(deterministic=True).info()["split_tiles"] > 0
