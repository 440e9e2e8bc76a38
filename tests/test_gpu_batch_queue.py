"""The queue of batched alpha-CROWN: any mix of problems, horizons and row counts gives each row the bits it has alone (few
rows for many problems, problems without rows, a device row count, more problems than the queue serves)."""
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


def _bound(probs, lo, hi, prob, n=None, steps=3):
    from gpu_util import DEV, T
    from paper_2412_09584_gb300 import binding as B
    params, x0, goal, H, rho = W.pack_batch(probs)
    ctx = B.bab_load_dynamics_batch(probs[0]["dims"], params, probs[0]["s"], probs[0]["k"])
    try:
        rows = lo.shape[0]
        lb = torch.full((rows,), 7.0, device=DEV)
        d_n = None if n is None else torch.tensor([n], dtype=torch.int32, device=DEV)
        B.bab_bound_batch(ctx, T(x0), T(goal), T(H, torch.int32), T(rho), int(H.max()), lo.shape[1], T(lo), T(hi),
                          T(prob, torch.int32), rows, lb, alpha_steps=steps, lr=0.1, d_n=d_n)
        torch.cuda.synchronize()
        return lb.cpu().numpy()
    finally:
        B.bab_destroy(ctx)


@pytest.mark.parametrize("P,rows", [(2, 1), (3, 17), (64, 40), (70, 300), (1100, 30)])
def test_rows_alone_and_in_the_batch(P, rows):
    probs, H = W.batch_problems(P, seed=P, H_lo=1, H_hi=9, rho=0.01)
    rng = np.random.default_rng(P)
    prob = rng.integers(0, P, rows).astype(np.int32)
    d = 2 * int(H.max())
    lo = rng.uniform(-1, 0, (rows, d)).astype(np.float32)
    hi = (lo + rng.uniform(0, 1, (rows, d))).astype(np.float32)
    full = _bound(probs, lo, hi, prob)
    order = rng.permutation(rows)
    assert np.array_equal(_bound(probs, lo[order], hi[order], prob[order]), full[order])
    live = rows // 2
    part = _bound(probs, lo, hi, prob, n=live)
    assert np.array_equal(part[:live], full[:live]) and np.all(part[live:] == 7.0)
    i = rows // 3  # the same row as a batch of its own, in a context of two problems
    two = [dict(probs[prob[i]]), dict(probs[prob[i]])]
    dp = 2 * int(H[prob[i]])
    assert _bound(two, lo[i:i + 1, :dp], hi[i:i + 1, :dp], np.array([1], np.int32))[0] == full[i]


def test_more_problems_than_the_queue_serves():
    probs, H = W.batch_problems(40, seed=5, H_lo=2, H_hi=6)
    rng = np.random.default_rng(1)
    rows, d = 90, 2 * int(H.max())
    lo = rng.uniform(-1, 0, (rows, d)).astype(np.float32)
    hi = (lo + 0.5).astype(np.float32)
    prob = rng.integers(0, 40, rows).astype(np.int32)
    many = [probs[i % 40] for i in range(2080)]
    shift = (rng.integers(0, 52, rows) * 40).astype(np.int32)
    assert np.array_equal(_bound(probs, lo, hi, prob), _bound(many, lo, hi, prob + shift))
