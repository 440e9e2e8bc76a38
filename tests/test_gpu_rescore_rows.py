"""The FP32 re-score of every box over its tile sizes: box counts on both sides of each size's last wave, with the
network image in shared memory (2, 4 and 8 boxes per group) and read through the cache (4, 8, 16 and 28 per CTA).  Each
output is one chain of multiply-adds over the inputs in order and each sum is in index order, as in the re-score of
listed boxes, so that the two give equal bits."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NETS = {"pushing": (8, 2, [128, 128, 128], 3), "odd": (5, 3, [96, 32], 4), "wide": (20, 3, [256, 224, 256], 2)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("net", sorted(NETS))
@pytest.mark.parametrize("rows", [0, 4, 8, 16, 28, 40])
def test_every_box_gets_the_bits_of_the_listed_rescore(gp, net, rows):
    s, k, hidden, H = NETS[net]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = W.make_problem(s, k, hidden, H, 0.01, seed=rows + 1, weight_scale=0.2)
    g = gp(p)
    for n in ((1, 5) if rows == 0 else (rows * sms - 1, rows * sms + 1)):
        lo, hi, ids = W.random_boxes(k * H, n, seed=n, min_width=0.1, max_width=1.0)
        B.bab_set_rescore_topk(g.ctx, 0)
        every = g.rollout(lo, hi, ids, M=3, seed=3, precision=B.PREC_BF16)
        B.bab_set_rescore_topk(g.ctx, n + 1)
        listed = g.rollout(lo, hi, ids, M=3, seed=3, precision=B.PREC_BF16)
        assert np.array_equal(every["ub"], listed["ub"])
        assert np.array_equal(every["best_u"], listed["best_u"])
