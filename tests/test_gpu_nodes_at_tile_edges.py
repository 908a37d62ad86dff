"""fresnel_get_nodes where a node lies at a tile's edge to within rounding.

The evaluation places FP32 nodes by double-float arithmetic; the FP64 nodes
that are handed out may round to the cell before, in a tile that holds no
records of the plan.  Handing them out changes nothing: no error, and the same
field bit for bit (one node: no sum whose order could vary)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("recompute", [False, True])
def test_one_node_on_either_side_of_a_tile_edge(recompute):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_05978_gb300 import Plan, build
    build.build()
    torch.cuda.set_device(0)
    # nf = 128, U = nf h / lz = 12.8 cells per unit, w = 8: the first support
    # cell is floor(U x - w / 2 + 80) + 1, which passes from 95 to 96 at x =
    # 19 / 12.8.  The node lies half a radius left of the centre
    x0 = 19 / 12.8
    ulp = np.spacing(x0 + 0.5)
    for k in range(-160, 161):
        fam = W.fourier_family([1.0], 1, 1, 1, cx=x0 + 0.5 + k * ulp)
        p = Plan([fam], 0.5, 1.0, 1e-6, kernel_w=8, sigma=2.0, grid=W.grid_spec(64, 64, 0.05),
                 recompute_nodes=recompute)
        assert p.info()["nf1"] == 128
        u = p.eval().clone()
        x, _, _ = p.nodes()
        assert abs(float(x[0]) - (x0 + k * ulp)) <= 4 * ulp
        assert torch.equal(p.eval(), u)
        p.close()
