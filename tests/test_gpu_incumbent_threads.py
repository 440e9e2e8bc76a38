"""FP64 incumbents of networks of different sizes from several threads at once: a launch's shared-memory limit does not
depend on what another thread has launched."""
import threading

import numpy as np
import pytest
import torch

from gpu_util import DEV, GpuProblem, T
from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NETS = [(4, 2, [32, 32], 5), (8, 2, [128, 128, 128], 4), (32, 4, [256] * 6, 3), (8, 2, [64, 64], 3)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def test_threads_with_different_networks(oracle):
    errors, ready = [], threading.Barrier(len(NETS))

    def work(i):
        s, k, hidden, H = NETS[i]
        p = W.make_problem(s, k, hidden, H, 0.0, seed=i, weight_scale=0.1)
        g = GpuProblem(p)
        try:
            u = np.random.default_rng(i).uniform(-1, 1, (6, k * H)).astype(np.float32)
            ub = np.arange(6, 0, -1).astype(np.float32)  # the last row is the smallest
            with torch.cuda.stream(torch.cuda.Stream()):
                tu, tb, best = T(u), T(ub), torch.zeros(k * H, device=DEV)
                ready.wait(60)
                for _ in range(200):
                    val = torch.full((1,), np.inf, dtype=torch.float64, device=DEV)
                    B.bab_update_incumbent(g.ctx, g.x0, g.goal, H, 0.0, tb, tu, 6, val, best)
                torch.cuda.current_stream().synchronize()
            value = oracle.objective(p, u[-1].astype(np.float64))
            if not (abs(float(val.item()) - value) <= 1e-10 * abs(value) and np.array_equal(best.cpu().numpy(), u[-1])):
                errors.append((i, float(val.item()), value))
        except Exception as e:  # reported by the test's own thread
            errors.append((i, repr(e)))
        finally:
            g.close()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(NETS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
