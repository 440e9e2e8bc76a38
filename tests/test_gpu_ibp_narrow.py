"""Interval bounds of networks with narrow layers (one warp per box) against the tiled kernel that takes the wider ones:
the same network with one hidden layer widened beyond 64 by neurons of zero weights gives the same bits, since every sum
only gains zero products."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# layers of one and of two outputs a lane, remainders of 4 and of 32, an input row wider than the layers, no hidden layer
NETS = {"one": (1, 1, [1], 3), "tiny": (4, 2, [32, 32], 5), "odd": (6, 2, [24, 33], 4), "edge": (8, 2, [64, 31, 64], 3),
        "input": (40, 24, [5], 2), "mixed": (4, 2, [48, 3, 32], 3), "linear": (6, 2, [], 4)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _widened(p):
    """The problem with its first hidden layer widened to 72 (without one: a layer of 72 zero neurons cannot stand for
    the identity, so none)."""
    layers = [(w.copy(), b.copy()) for w, b in W.unpack_params(p)]
    (w1, b1), (w2, b2) = layers[0], layers[1]
    add = 72 - w1.shape[0]
    layers[0] = (np.vstack([w1, np.zeros((add, w1.shape[1]), w1.dtype)]), np.concatenate([b1, np.zeros(add, b1.dtype)]))
    layers[1] = (np.hstack([w2, np.zeros((w2.shape[0], add), w2.dtype)]), b2)
    dims = list(p["dims"])
    dims[1] += add
    return dict(p, dims=dims, params=W.pack_params(layers))


def _check_oracle(oracle, p, lo, hi, got):
    from test_gpu_shapes import ibp_error_bound
    _, pl, pu, xl, xu = got
    _, pl_o, pu_o, xl_o, xu_o = oracle.ibp(p, lo, hi)
    e_pre, e_x = ibp_error_bound(p, lo, hi, pl_o, pu_o, xl_o, xu_o)
    for gv, ov, e in ((pl, pl_o, e_pre), (pu, pu_o, e_pre), (xl, xl_o, e_x), (xu, xu_o, e_x)):
        assert np.all(np.abs(gv - ov) <= e + 1e-30)


@pytest.mark.parametrize("net", sorted(NETS))
@pytest.mark.parametrize("n", [1, 7, 4096, 6001])
def test_the_same_bits_as_the_tiles(oracle, gp, net, n):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01 if n % 2 else 0.0, seed=len(net) + n, weight_scale=0.5)
    lo, hi, _ = W.random_boxes(k * H, n, seed=n, min_width=0.0, max_width=0.3)
    if n > 1000 and all(w % 4 == 0 for w in hidden):
        # one box that is not finite among finite ones (padded outputs of other widths are 0 x inf in that row)
        hi[n // 2, 0] = np.inf
    got = gp(p).ibp(lo, hi)
    if not hidden:
        keep = np.isfinite(hi).all(axis=1) & (np.arange(n) < 50)
        return _check_oracle(oracle, p, lo[keep], hi[keep], [a[keep] for a in got])
    wide = gp(_widened(p)).ibp(lo, hi)
    cols = np.r_[0:hidden[0], 72:72 + sum(hidden[1:])]
    for a, b in zip(got, [wide[0], wide[1][:, :, cols], wide[2][:, :, cols], wide[3], wide[4]]):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("net", ["tiny", "odd", "edge"])
def test_the_obstacle_cost(gp, net):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=3, weight_scale=0.5)
    lo, hi, _ = W.random_boxes(k * H, 500, seed=5, min_width=0.0, max_width=0.5)
    out = []
    for q in (p, _widened(p)):
        g = gp(q)
        B.bab_set_cost(g.ctx, B.COST_PUSHING_OBSTACLES, **W.obstacle_cost(H, 3))
        lb, _, _, xl, xu = g.ibp(lo, hi)
        out.append((lb, xl, xu))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
