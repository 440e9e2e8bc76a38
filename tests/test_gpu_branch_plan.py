"""The pool planner (counting for at most 256 rows, clusters of 1 to 8 CTAs beyond) and the row writer (16-byte words with
8, 16 or 32 lanes a row, single coordinates otherwise): bit-exact against the oracle at the edges of each."""
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


def _pool(n, d, seed, ties, nan):
    lo, hi, ids = W.dyadic_boxes(d, n, seed=seed)
    lb, ub = W.pool_values(n, seed, nan_frac=nan, tie_frac=ties)
    return lo, hi, ids[np.random.default_rng(seed).permutation(n)], lb, ub


@pytest.mark.parametrize("n", [1, 33, 256, 257, 2048, 2049, 5000, 17000, 66000])
@pytest.mark.parametrize("d", [1, 10, 32, 40, 68, 132])
def test_plan_and_write(oracle, gp, n, d):
    if n > 60000 and d != 10:
        pytest.skip("the share that is read again in every pass: once")
    g = gp(W.config_problem("tiny"))
    ties, nan = (0.6, 0.02) if n % 2 else (0.0, 0.0)
    lo, hi, ids, lb, ub = _pool(n, d, n + d, ties, nan)
    inc = float(np.nanquantile(lb, 0.8))
    for n_pick, eta in ((max(1, n // 3), 0.75), (n, 0.5), (0, 0.5), (max(1, n // 50), 0.0)):
        r = g.prune_branch(lo, hi, lb, ub, ids, inc, n_pick, eta)
        o = oracle.prune_branch(lo, hi, lb, ub, ids, inc, n_pick, eta)
        assert np.array_equal(r["keep"].astype(bool), np.asarray(o["keep"]).astype(bool))
        assert (r["n_children"], r["n_rest"]) == (o["n_children"], o["n_rest"])
        for key in ("lo", "hi", "lb", "ub", "id"):
            assert np.array_equal(r[key], np.asarray(o[key]), equal_nan=key in ("lb", "ub"))


@pytest.mark.parametrize("n", [100, 3000, 9000, 70000])
def test_softmax_pick(oracle, gp, n):
    from paper_2412_09584_gb300 import binding as B
    from gpu_util import DEV, T, ids_t
    d = 12
    g = gp(W.config_problem("tiny"))
    lo, hi, ids, lb, ub = _pool(n, d, n, 0.1, 0.01)
    inc, n_pick = float(np.nanquantile(lb, 0.9)), n // 4
    cap = n + n_pick
    out = [torch.zeros(cap, d, device=DEV), torch.zeros(cap, d, device=DEV), torch.zeros(cap, device=DEV),
           torch.zeros(cap, device=DEV), torch.zeros(cap, dtype=torch.int64, device=DEV)]
    keep, counts = torch.zeros(n, dtype=torch.uint8, device=DEV), torch.zeros(3, dtype=torch.int32, device=DEV)
    B.bab_prune_branch_heuristic(g.ctx, d, T(lo), T(hi), T(lb), T(ub), ids_t(ids), n,
                                 torch.tensor([inc], dtype=torch.float64, device=DEV), n_pick, 0.5, 1, 0.05, 77, cap, *out,
                                 keep, counts)
    o = oracle.prune_branch_heuristic(lo, hi, lb, ub, ids, inc, n_pick, 0.5, pick_rule=1, temperature=0.05, pick_seed=77)
    m = o["n_children"] + o["n_rest"]
    assert counts.cpu().tolist() == [o["n_children"], o["n_rest"], m]
    for t, key in zip(out, ("lo", "hi", "lb", "ub", "id")):
        got = t.cpu().numpy()[:m]
        assert np.array_equal(got.astype(np.uint64) if key == "id" else got, np.asarray(o[key]), equal_nan=key in ("lb", "ub"))
