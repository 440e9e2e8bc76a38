"""The pool planner where identifiers decide: few distinct bounds, and only one, at the row counts of the counting planner
and of a lone CTA's radix passes; identifiers that differ in their last or in their first byte."""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("n", [2, 31, 129, 200, 255, 256, 257, 600, 1500, 2100])
@pytest.mark.parametrize("levels", [1, 5])
@pytest.mark.parametrize("shift", [0, 52])
def test_identifiers_decide(oracle, gp, n, levels, shift):
    d = 6
    rng = np.random.default_rng(n + levels)
    lo, hi, _ = W.random_boxes(d, n, seed=n, min_width=0.1, max_width=1.0)
    ids = (rng.permutation(n).astype(np.uint64) + np.uint64(1)) << np.uint64(shift)
    lb, ub = rng.integers(0, levels, n).astype(np.float32), rng.integers(0, levels, n).astype(np.float32) + 9
    g = gp(W.config_problem("tiny"))
    for n_pick, eta in ((max(1, n // 3), 0.75), (n - 1, 0.4), (1, 1.0), (max(1, n // 2), 0.0)):
        r = g.prune_branch(lo, hi, lb, ub, ids, 100.0, n_pick, eta)
        o = oracle.prune_branch(lo, hi, lb, ub, ids, 100.0, n_pick, eta)
        assert (r["n_children"], r["n_rest"]) == (o["n_children"], o["n_rest"])
        for key in ("lo", "hi", "lb", "ub", "id"):
            assert np.array_equal(r[key], np.asarray(o[key]))
