"""The interval-bound kernel's row groups and tiles: box counts and widths around each tile's edge (weights in shared
memory and streamed), boxes whose lower activations are mostly positive (the products of the lower end), rows that do
not depend on their neighbours, and boxes that are not finite."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W
from test_gpu_shapes import ibp_error_bound

pytestmark = pytest.mark.gpu

NETS = {"narrow": (3, 1, [1, 5], 3), "tiny": (4, 2, [32, 32], 4), "odd": (5, 3, [100, 33, 64], 3),
        "pushing": (8, 2, [128, 128, 128], 4), "wide_input": (40, 8, [128, 132], 2), "streamed": (32, 4, [256] * 3, 3),
        "streamed_odd": (33, 3, [256, 130, 250, 20], 2)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _check(oracle, p, lo, hi, got):
    _, pl, pu, xl, xu = got
    lb_o, pl_o, pu_o, xl_o, xu_o = oracle.ibp(p, lo, hi)
    e_pre, e_x = ibp_error_bound(p, lo, hi, pl_o, pu_o, xl_o, xu_o)
    for gv, ov, e in ((pl, pl_o, e_pre), (pu, pu_o, e_pre), (xl, xl_o, e_x), (xu, xu_o, e_x)):
        assert np.all(np.abs(gv - ov) <= e + 1e-30)
    assert np.all(pl <= pl_o + 1e-12 * np.abs(pl_o)) and np.all(pu >= pu_o - 1e-12 * np.abs(pu_o))
    assert np.all(got[0] <= lb_o + 1e-12 * np.abs(lb_o))


@pytest.mark.parametrize("net", sorted(NETS))
@pytest.mark.parametrize("n", [1, 5, 33, 700])
def test_tiles_against_the_oracle(oracle, gp, net, n):
    s, k, hidden, H = NETS[net]
    if n == 700 and net.startswith("streamed"):
        n = 40  # the oracle's time; rows past one tile of 32
    p = W.make_problem(s, k, hidden, H, 0.01, seed=len(net) + n, weight_scale=0.5)
    # widths from points to wide boxes: lower activations positive in the first, 0 in the last
    lo, hi, _ = W.random_boxes(k * H, n, seed=n, min_width=0.0, max_width=0.02 if n % 2 else 1.0)
    g = gp(p)
    _check(oracle, p, lo, hi, g.ibp(lo, hi))


@pytest.mark.parametrize("net", ["tiny", "pushing", "streamed"])
def test_rows_do_not_depend_on_their_tile(oracle, gp, net):
    """The same box gives the same bits in any batch: alone, among few and among many, whatever its neighbours."""
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=3, weight_scale=0.5)
    lo, hi, _ = W.random_boxes(k * H, 4000, seed=8, min_width=0.0, max_width=0.6)
    g = gp(p)
    full, full_c = g.ibp(lo, hi), g.crown(lo, hi)
    for rows in ([0], [3999, 1], list(range(100, 137)), list(range(0, 4000, 4))):
        part, part_c = g.ibp(lo[rows], hi[rows]), g.crown(lo[rows], hi[rows])
        for a, b in zip(full, part):
            assert np.array_equal(a[rows], b)
        for key in ("lb", "margin", "lin_coef", "lin_const"):
            assert np.array_equal(full_c[key][rows], part_c[key])


@pytest.mark.parametrize("net", ["tiny", "pushing", "streamed"])
def test_boxes_that_are_not_finite(gp, net):
    """An infinite box bounds its own row by infinities, without NaN, and leaves the others' bits alone."""
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.0, seed=5, weight_scale=0.5)
    lo, hi, _ = W.random_boxes(k * H, 30, seed=2, min_width=0.1, max_width=0.5)
    g = gp(p)
    ref = g.ibp(lo, hi)
    hi2 = hi.copy()
    hi2[7, k] = np.inf  # an action of step 1
    got = g.ibp(lo, hi2)
    keep = np.arange(30) != 7
    for a, b in zip(ref, got):
        assert np.array_equal(a[keep], b[keep])
    pl, pu, xl, xu = got[1][7], got[2][7], got[3][7], got[4][7]
    assert np.array_equal(pl[0], ref[1][7, 0]) and np.array_equal(xu[1], ref[4][7, 1])  # before that step
    assert not np.isnan(pl[1]).any() and not np.isnan(pu[1]).any() and np.isinf(pu[1]).any()
    assert not np.isnan(xl[2]).any() and np.all(np.isneginf(xl[2])) and np.all(np.isposinf(xu[2]))
