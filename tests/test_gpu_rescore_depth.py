"""The top-k re-score of networks whose columns fill a cluster's shared memory, or exceed it (the layers beyond it are
staged at every step): the listed boxes carry the bits of the every-box re-score, the others their BF16 value."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# bytes of a CTA's columns; 191488 fit beside the kernel's own arrays (199680 with the obstacle cost)
NETS = {"five": (4, 2, [256] * 5),                 # 133508
        "seven4": (4, 2, [256] * 7),               # 199300
        "seven8": (8, 2, [256] * 7),               # 199812
        "seven16": (16, 2, [256] * 7),             # 201864
        "mixed32": (32, 2, [256] * 6 + [192]),     # 196720
        "seven32": (32, 2, [256] * 7)}             # 205968


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


# (tensor-core rollouts carry the obstacle cost up to 8 states)
@pytest.mark.parametrize("net,cost", [(v, "squared") for v in NETS] + [(v, "obstacles") for v in NETS if NETS[v][0] <= 8])
def test_exactly_the_listed_boxes_are_rescored(gp, net, cost):
    s, k, hidden = NETS[net]
    H, n = 8, 150  # 2.1 M multiply-adds a box at least: the cluster kernel's range; one wave of clusters holds 120 boxes
    p = W.make_problem(s, k, hidden, H, 0.01, seed=len(net), weight_scale=0.1)
    lo, hi, ids = W.random_boxes(k * H, n, seed=n, min_width=0.1, max_width=1.0)
    g = gp(p)
    if cost == "obstacles":
        B.bab_set_cost(g.ctx, B.COST_PUSHING_OBSTACLES, **W.obstacle_cost(H, 3))

    def ub(topk):
        B.bab_set_rescore_topk(g.ctx, topk)
        return g.rollout(lo, hi, ids, M=8, seed=3, precision=B.PREC_BF16)["ub"]

    full, first = ub(0), ub(1)
    for topk in (2, 15, 130):
        some = ub(topk)

        def expected(best):
            # `best` took the first run's single re-score; the rest of the list is chosen on the others' BF16 values
            out = first.copy()
            rest = np.delete(np.arange(n), best)
            more = rest[np.lexsort((ids[rest], first[rest]))][:topk - 1]
            out[more] = full[more]
            return out

        assert any(np.array_equal(some, expected(b)) for b in np.nonzero(first == full)[0])
    assert np.array_equal(ub(n + 1), full)
