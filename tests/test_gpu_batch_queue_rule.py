"""Batched bounds on both sides of the rule that sends a call to the queue (work done, rows a problem): the rows' bits do
not depend on the route."""
import numpy as np
import pytest

from paper_2412_09584_gb300 import workloads as W
from test_gpu_batch_queue import _bound, built  # noqa: F401

pytestmark = pytest.mark.gpu


# horizons up to 15 and 16 without alpha steps, 7 and 8 with one; rows up to 4 a problem less one, and 4
@pytest.mark.parametrize("steps,H_hi", [(0, 15), (0, 16), (1, 7), (1, 8), (2, 3)])
@pytest.mark.parametrize("P,rows", [(12, 47), (12, 48), (300, 1300)])
def test_the_route_does_not_change_a_row(steps, H_hi, P, rows):
    probs, _ = W.batch_problems(P, seed=P, H_lo=1, H_hi=H_hi, rho=0.01)
    probs[0]["H"] = H_hi  # the call's longest horizon
    H = np.array([p["H"] for p in probs])
    rng = np.random.default_rng(rows)
    prob = rng.integers(0, P, rows).astype(np.int32)
    d = 2 * H_hi
    lo = rng.uniform(-1, 0, (rows, d)).astype(np.float32)
    hi = (lo + rng.uniform(0, 1, (rows, d))).astype(np.float32)
    full = _bound(probs, lo, hi, prob, steps=steps)
    few = slice(5, 25)  # fewer rows than 4 a problem: the queue
    assert np.array_equal(_bound(probs, lo[few], hi[few], prob[few], steps=steps), full[few])
    for i in (0, rows - 1):  # alone
        two = [dict(probs[prob[i]]), dict(probs[prob[i]])]
        dp = 2 * int(H[prob[i]])
        assert _bound(two, lo[i:i + 1, :dp], hi[i:i + 1, :dp], np.array([1], np.int32), steps=steps)[0] == full[i]
