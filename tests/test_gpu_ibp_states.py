"""Bounds of networks with many states and streamed weights: the tiles have as many rows as fit in shared memory beside
the ring (32 up to 112 states of a 256-wide network, 28, then 24)."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W
from test_gpu_shapes import REL, ibp_error_bound

pytestmark = pytest.mark.gpu

NETS = {"112": (112, 8, [256, 256], 2), "113": (113, 7, [256, 255], 2), "128": (128, 8, [256, 256], 3),
        "200": (200, 8, [256, 256, 256], 2), "255": (255, 1, [256], 2)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("net", sorted(NETS))
def test_bounds_against_the_oracle(oracle, gp, net):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=s)
    lo, hi, _ = W.random_boxes(k * H, 37, seed=s + 1, min_width=0.0, max_width=1.0)
    g = gp(p)
    lb, pl, pu, xl, xu = g.ibp(lo, hi)
    lb_o, pl_o, pu_o, xl_o, xu_o = oracle.ibp(p, lo, hi)
    e_pre, e_x = ibp_error_bound(p, lo, hi, pl_o, pu_o, xl_o, xu_o)
    for gv, ov, e in ((pl, pl_o, e_pre), (pu, pu_o, e_pre), (xl, xl_o, e_x), (xu, xu_o, e_x)):
        assert np.all(np.abs(gv - ov) <= e + 1e-30)
    assert np.all(pl <= pl_o + 1e-12 * np.abs(pl_o)) and np.all(pu >= pu_o - 1e-12 * np.abs(pu_o))
    assert np.all(lb <= lb_o + 1e-12 * np.abs(lb_o))
    o = oracle.crown(p, lo, hi)
    scale = np.maximum(o["scale"], 1.0)
    r = g.crown(lo, hi)
    assert np.all(np.abs(r["lb"].astype(np.float64) + r["margin"] - o["lb"]) <= REL * scale)
    assert np.all(r["lb"] <= o["lb"] + 1e-12 * np.abs(o["lb"]))
    _, _, hist = g.alpha_steps(lo, hi, steps=1, lr=0.1)
    _, grad_o, _ = oracle.alpha_grad(p, lo, hi, oracle.adaptive_alpha(p, lo, hi))
    gs = np.maximum(np.abs(grad_o).max(axis=(1, 2), keepdims=True), 1e-30)
    # a neuron whose end lies within the intervals' rounding of 0 has a slope on one side only: no gradient to compare
    decided = (np.abs(pl_o) > e_pre) & (np.abs(pu_o) > e_pre)
    assert decided.mean() > 0.99 and np.all((np.abs(hist[0]["grad"] - grad_o) <= 1e-4 * gs)[decided])


@pytest.mark.parametrize("net,rows", [("112", 32), ("128", 28), ("255", 24)])
def test_full_tiles_and_the_rest_give_the_same_bits(gp, net, rows):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=4, weight_scale=0.5)
    n = (rows + 5) * torch.cuda.get_device_properties(0).multi_processor_count - 3  # one wave of tiles and a part of one
    lo, hi, _ = W.random_boxes(k * H, n, seed=5, min_width=0.0, max_width=0.8)
    g = gp(p)
    full = g.ibp(lo, hi)
    for part in (slice(0, 40), slice(n - 40, n)):
        for a, b in zip(full, g.ibp(lo[part], hi[part])):
            assert np.array_equal(a[part], b)
