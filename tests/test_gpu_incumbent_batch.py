"""The FP64 incumbents of batched problems on both sides of the rules that pick one CTA or a cluster a problem and weights
in shared memory or read through L2."""
import numpy as np
import pytest
import torch

from gpu_util import DEV, T, ids_t
from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


# one CTA: few multiply-adds a step (1408), many problems, more than 64; a cluster: 10 problems of 5248 (512 P = 5120)
# but not 11, 64 of 76032 but not 65; one CTA whose weights (287 KB as doubles) exceed shared memory; one or two steps,
# whose weights are not copied
@pytest.mark.parametrize("P,s,k,hidden,H_hi", [
    (3, 4, 2, [32, 32], 5), (10, 8, 2, [64, 64], 4), (11, 8, 2, [64, 64], 4), (11, 8, 2, [64, 64], 2),
    (64, 16, 4, [256, 256], 2), (65, 16, 4, [256, 256], 3), (100, 8, 2, [128, 128, 128], 3), (5, 3, 1, [67, 250, 3], 1)])
def test_values_of_all_problems(oracle, P, s, k, hidden, H_hi):
    probs, _ = W.batch_problems(P, P, s, k, hidden, 1, H_hi, float(np.float32(0.01)))
    probs[0]["H"] = H_hi
    params, x0, goal, H, rho = W.pack_batch(probs)
    d, n = k * H_hi, 2 * P
    rng = np.random.default_rng(P)
    lo = rng.uniform(-1, 0, (n, d)).astype(np.float32)
    hi = (lo + rng.uniform(0, 1, (n, d))).astype(np.float32)
    prob = np.repeat(np.arange(P), 2).astype(np.int32)
    ctx = B.bab_load_dynamics_batch(probs[0]["dims"], params, s, k)
    try:
        ub, u = torch.empty(n, device=DEV), torch.empty(n, d, device=DEV)
        val = torch.full((P,), np.inf, dtype=torch.float64, device=DEV)
        best = torch.zeros(P, d, device=DEV)
        B.bab_rollout_batch(ctx, T(x0), T(goal), T(H, torch.int32), T(rho), H_hi, d, T(lo), T(hi),
                            ids_t(np.arange(n) + 1), T(prob, torch.int32), n, 16, 3, ub, u, val, best)
        torch.cuda.synchronize()
    finally:
        B.bab_destroy(ctx)
    ub, u, val, best = ub.cpu().numpy(), u.cpu().numpy(), val.cpu().numpy(), best.cpu().numpy()
    for p in range(P):
        row = 2 * p + int(ub[2 * p + 1] < ub[2 * p])
        dp = k * int(H[p])
        assert np.array_equal(best[p, :dp], u[row, :dp])
        assert val[p] == pytest.approx(oracle.objective(probs[p], best[p, :dp].astype(np.float64)), rel=1e-10)
