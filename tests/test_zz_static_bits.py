"""bab_bound_crown_static gives the bits of the context's call on every route of the interval bounds, and no finite bound
where a parameter of the network on the device is not finite."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W
from test_zz_no_alloc import _context_bound, _static_bound, built  # noqa: F401

pytestmark = pytest.mark.gpu

# one warp per box; tiles with the weights in shared memory; streamed weights
NETS = {"narrow": (4, 2, [33, 64], 4, 300), "tiles": (8, 2, [128, 96, 128], 5, 70), "streamed": (32, 4, [256] * 3, 3, 50)}


@pytest.mark.parametrize("net", sorted(NETS))
def test_the_context_bits(net):
    s, k, hidden, H, n = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=4, weight_scale=0.3)
    lo, hi, _ = W.random_boxes(k * H, n, seed=6, min_width=0.0, max_width=0.6)
    for m in (n, 1):
        for a, b in zip(_static_bound(p, lo[:m], hi[:m]), _context_bound(p, lo[:m], hi[:m])):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("net", ["tiles", "streamed"])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_a_parameter_that_is_not_finite(net, value):
    s, k, hidden, H, n = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=4, weight_scale=0.3)
    lo, hi, _ = W.random_boxes(k * H, n, seed=6, min_width=0.0, max_width=0.6)
    good = _static_bound(p, lo, hi)[0]
    for at in (0, p["params"].size - s - 1):  # the first weight, and the last one before the output's biases
        q = p["params"].copy()
        q[at] = value
        assert not np.isfinite(_static_bound(dict(p, params=q), lo, hi)[0]).any()
    assert np.array_equal(_static_bound(p, lo, hi)[0], good)
