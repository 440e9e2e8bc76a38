"""FP32 CROWN and its adjoint over more boxes than one wave of CTAs holds: whole waves and the rest are separate launches,
and every row has the bits it has in a small batch, also with a device row count and under a scratch limit; widths beyond
128, whose tiles differ by the rows of a group."""
import numpy as np
import pytest
import torch

from gpu_util import DEV, T
from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NETS = {"tiny": (4, 2, [32, 32], 3), "odd": (5, 3, [132, 40], 2), "wide": (16, 4, [256, 250], 2)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available()


def _grad(g, lo, hi, alpha, d_n=None):
    n = lo.shape[0]
    lb, grad = torch.full((n,), 7.0, device=DEV), torch.full((n, g.H, g.sumh), 7.0, device=DEV)
    B.bab_alpha_grad(g.ctx, g.x0, g.goal, g.H, g.rho, T(lo), T(hi), n, T(alpha), lb, grad,
                     d_n=None if d_n is None else torch.tensor([d_n], dtype=torch.int32, device=DEV))
    torch.cuda.synchronize()
    return lb.cpu().numpy(), grad.cpu().numpy()


@pytest.mark.parametrize("net", sorted(NETS))
@pytest.mark.parametrize("rest", [0, 1, 700, 2500])
def test_rows_beyond_one_wave(gp, net, rest):
    s, k, hidden, H = NETS[net]
    p = W.make_problem(s, k, hidden, H, 0.01, seed=7, weight_scale=0.4)
    wave = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    n = wave + rest
    lo, hi, _ = W.random_boxes(k * H, n, seed=rest, min_width=0.0, max_width=0.6)
    alpha = np.random.default_rng(rest).uniform(0, 1, (n, H, sum(hidden))).astype(np.float32)
    g = gp(p)
    crown, grad = g.crown(lo, hi, alpha), _grad(g, lo, hi, alpha)
    for part in (slice(0, 30), slice(wave - 20, min(n, wave + 20)), slice(n - 25, n)):
        small = g.crown(lo[part], hi[part], alpha[part])
        for key in small:
            assert np.array_equal(crown[key][part], small[key])
        for a, b in zip(grad, _grad(g, lo[part], hi[part], alpha[part])):
            assert np.array_equal(a[part], b)
    for live in (wave - 3, wave + rest // 2):
        part = _grad(g, lo, hi, alpha, d_n=live)
        for a, b in zip(part, grad):
            assert np.array_equal(a[:live], b[:live]) and np.all(a[live:] == 7.0)
    B.bab_set_scratch_limit(g.ctx, 2000 * 4 * (H * (4 * sum(hidden) + s) + 2 * (H + 1) * s + 2 * k * H) + (1 << 16))
    for key, v in g.crown(lo, hi, alpha).items():
        assert np.array_equal(v, crown[key])
