"""The register-tiled FP32 rollout (variant 0) against the per-box kernel (variant 2): the same bits at every tile edge,
with tiles that hold samples of several boxes, layer widths around each warp block, and images beyond shared memory."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NETS = {"one": (1, 1, [1], 3, 0.0), "tiny": (4, 2, [32, 32], 5, 0.0), "odd": (5, 3, [100, 33, 9], 4, 0.05),
        "pushing": (8, 2, [128, 128, 128], 6, 0.01), "wide": (16, 4, [160, 32, 64], 4, 0.01),
        "outputs17": (17, 2, [132, 68], 3, 0.0), "streamed": (32, 4, [256] * 4, 4, 0.01)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("net", sorted(NETS))
@pytest.mark.parametrize("n,M", [(1, 1), (5, 63), (3, 64), (7, 65), (70, 3), (40, 200)])
def test_rows_equal_per_box_tiles(gp, net, n, M):
    from paper_2412_09584_gb300 import binding as B
    s, k, hidden, H, rho = NETS[net]
    p = W.make_problem(s, k, hidden, H, rho, seed=n + M, weight_scale=0.5)
    lo, hi, ids = W.random_boxes(k * H, n, seed=M, min_width=0.0, max_width=1.0)
    g = gp(p)
    out = []
    for v in (0, 2):
        B.bab_set_variant(g.ctx, B.KERNEL_ROLLOUT_FP32, v)
        out.append(g.rollout(lo, hi, ids, M=M, seed=9, incumbent=True))
    for key in ("ub", "best_u", "inc_val", "inc_u"):
        assert np.array_equal(out[0][key], out[1][key])
