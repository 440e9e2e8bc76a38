"""The FP64 incumbent (one CTA, and clusters that share every layer) and the top-k re-score on clusters at the edges of
their splits: outputs that do not divide by the CTAs, layers narrower than the cluster, more listed boxes than a wave."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NETS = {"one": (1, 1, [1], 3), "tiny": (4, 2, [32, 32], 5), "just_one_cta": (8, 2, [62, 50], 3), "ragged": (5, 3, [67, 250, 3, 129], 4),
        "pushing": (8, 2, [128, 128, 128], 20), "large": (32, 4, [256] * 7, 3), "long": (4, 2, [40], 600)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("net", sorted(NETS))
def test_incumbent_value(oracle, gp, net):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=len(net), weight_scale=0.3)
    lo, hi, ids = W.random_boxes(k * H, 19, seed=4, min_width=0.0, max_width=0.5)
    r = gp(p).rollout(lo, hi, ids, M=70, seed=2, incumbent=True)
    assert np.array_equal(r["inc_u"], r["best_u"][int(np.argmin(r["ub"]))])
    assert r["inc_val"] == pytest.approx(oracle.objective(p, r["inc_u"].astype(np.float64)), rel=1e-10)


@pytest.mark.parametrize("net", ["wide", "odd"])
@pytest.mark.parametrize("topk", [1, 7, 64, 130])
def test_topk_rescore_on_clusters(gp, net, topk):
    """The boxes of smallest BF16 ub get the bits of the every-box re-score, the others keep their BF16 ub."""
    from paper_2412_09584_gb300 import binding as B
    s, k, hidden, H = {"wide": (32, 4, [256, 256, 256], 20), "odd": (9, 3, [224, 160, 256], 24)}[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=topk, weight_scale=0.1)
    n = 300
    lo, hi, ids = W.random_boxes(k * H, n, seed=topk, min_width=0.1, max_width=1.0)
    g = gp(p)
    full = g.rollout(lo, hi, ids, M=8, seed=3, precision=B.PREC_BF16)
    B.bab_set_rescore_topk(g.ctx, n + 1)  # every box through the list
    listed = g.rollout(lo, hi, ids, M=8, seed=3, precision=B.PREC_BF16)
    B.bab_set_rescore_topk(g.ctx, topk)
    some = g.rollout(lo, hi, ids, M=8, seed=3, precision=B.PREC_BF16)
    assert np.array_equal(full["ub"], listed["ub"])
    assert np.array_equal(full["best_u"], some["best_u"])
    same = some["ub"] == full["ub"]
    assert same.sum() >= topk and np.allclose(some["ub"], full["ub"], rtol=2e-2)
