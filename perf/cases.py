"""The work a user of this library has it do, as measurable cases.

Each case is one call, or one short sequence of calls, of the public binding on device tensors: the sampled search
(`rollout`), the interval bounds (`ibp`), the CROWN bounds (`crown`), the slope optimisation (`alpha`), the bound
with its gradient through torch.autograd (`grad`), many problems in one launch (`batch`), the pruner and splitter
(`prune`), and a whole branch-and-bound iteration (`iteration`).  The networks and sizes are those of
paper_2412_09584_gb300.workloads and of the benchmark; `draw` spreads them over the ranges in between.
"""
import math

import numpy as np
import torch

from paper_2412_09584_gb300 import binding as B
from paper_2412_09584_gb300 import workloads as W
from paper_2412_09584_gb300.autograd import CrownProblem, crown_bound

PRECISION = {"fp32": B.PREC_FP32, "bf16x3": B.PREC_BF16X3, "bf16": B.PREC_BF16, "tf32x3": B.PREC_TF32X3}
ETA = 0.75       # share of the pick-out quota taken by upper bound
LR = 0.1         # Adam step of the slopes
F64 = torch.float64


def _net(s, k, hidden, H, rho):
    return {"s": s, "k": k, "hidden": hidden, "H": H, "rho": rho}


TINY = _net(4, 2, "32-32", 5, 0.0)
PUSHING = _net(8, 2, "128-128-128", 20, 0.01)
MANIP = _net(32, 4, "256-256-256-256", 40, 0.01)


def listed():
    return [
        # One whole branch-and-bound iteration of the smallest planning problem (64 children, 256 samples each): a
        # replanning loop on a small model runs these one after another, so launches and latencies count.
        {"name": "iteration_tiny", "kind": "iteration", **TINY, "n": 64, "samples": 256, "precision": "fp32"},
        # The search in full precision at the pushing scale: 512 children of an iteration, 1024 samples each.
        {"name": "rollout_pushing_fp32", "kind": "rollout", **PUSHING, "n": 512, "samples": 1024,
         "precision": "fp32", "topk": 0},
        # The benchmark's search: BF16 samples of 4096 children, each box's pick re-scored in FP32.
        {"name": "rollout_pushing_bf16", "kind": "rollout", **PUSHING, "n": 4096, "samples": 1024,
         "precision": "bf16", "topk": 0},
        # The object-manipulation search: 65536 BF16 rollouts, the best 64 boxes re-scored in FP32.
        {"name": "rollout_manip_bf16", "kind": "rollout", **MANIP, "n": 16384, "samples": 4, "precision": "bf16",
         "topk": 64},
        # Interval bounds alone with every intermediate bound returned (a user's own relaxation on top of them),
        # a ragged number of boxes.
        {"name": "ibp_pushing", "kind": "ibp", **PUSHING, "n": 3001, "intervals": "fp32"},
        # The lower bounds of an iteration's children in full precision.
        {"name": "crown_pushing_fp32", "kind": "crown", **PUSHING, "n": 4096, "precision": "fp32",
         "intervals": "fp32"},
        # The same in the benchmark's precision: interval bounds in FP32, backward products as BF16 splits.
        {"name": "crown_pushing_bf16x3", "kind": "crown", **PUSHING, "n": 4096, "precision": "bf16x3",
         "intervals": "fp32"},
        # The largest bound call: the object-manipulation network, 16384 boxes, horizon 40.
        {"name": "crown_manip_bf16x3", "kind": "crown", **MANIP, "n": 16384, "precision": "bf16x3",
         "intervals": "fp32"},
        # alpha-CROWN on the small network: 4096 children, 20 Adam steps on the slopes.
        {"name": "alpha_tiny", "kind": "alpha", **TINY, "n": 4096, "steps": 20, "precision": "fp32"},
        # The bound as a torch.autograd function, forward and backward, at the pushing scale: the step of a user's
        # own optimiser over the slopes.
        {"name": "grad_pushing_fp32", "kind": "grad", **PUSHING, "n": 512, "precision": "fp32"},
        # Many independent problems of one architecture in one call, horizons 10 to 80, 20 slope steps each.
        {"name": "bound_batch", "kind": "batch", "s": 4, "k": 2, "hidden": "32-32", "H": 80, "H_lo": 10, "rho": 0.0,
         "problems": 64, "n": 8889, "steps": 20},
        # The pool late in a search: prune, pick out, split, and compact the survivors.
        {"name": "prune_pool", "kind": "prune", "d": 40, "n": 60000, "n_pick": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds and ranges."""
    kind = rng.choice(["iteration", "rollout", "rollout", "ibp", "crown", "crown", "alpha", "grad", "batch", "prune"])
    if kind == "prune":
        n = _log_int(rng, 100, 60000)
        return {"kind": kind, "d": rng.randint(5, 160), "n": n, "n_pick": max(1, int(n * rng.uniform(0.02, 0.6)))}
    if kind == "batch":
        H = rng.randint(12, 80)
        return {"kind": kind, "s": 4, "k": 2, "hidden": rng.choice(["32-32", "32-32", "48-32", "64"]), "H": H,
                "H_lo": rng.randint(2, H), "rho": rng.choice([0.0, 0.01]), "problems": rng.randint(2, 64),
                "n": _log_int(rng, 64, 8000), "steps": rng.randint(1, 20)}
    if kind == "rollout":
        precision = rng.choice(["fp32", "bf16", "bf16x3"])
    elif kind == "crown":
        precision = rng.choice(["fp32", "bf16x3", "bf16x3", "tf32x3"])
    elif kind == "grad":
        precision = rng.choice(["fp32", "bf16x3"])
    else:
        precision = "fp32"
    size = rng.choice(["tiny", "pushing", "pushing", "odd"] if kind in ("iteration", "grad", "alpha") else
                      ["tiny", "pushing", "odd", "manip"])
    if size == "tiny":
        c = dict(TINY, H=rng.randint(3, 12))
    elif size == "pushing":
        c = dict(PUSHING, H=rng.randint(5, 20))
    elif size == "manip":
        c = dict(MANIP, H=rng.randint(5, 40))
    else:
        widths = [32, 64, 96, 128] if precision != "fp32" else [24, 33, 50, 64, 96, 100, 128, 160]
        c = _net(rng.randint(2, 16), rng.randint(1, 8), "-".join(str(rng.choice(widths)) for _ in range(rng.randint(1, 3))),
                 rng.randint(3, 24), rng.choice([0.0, 0.01, 0.1]))
    c["kind"] = kind
    c["precision"] = precision
    macs = _macs(c) * c["H"]
    if kind == "rollout":
        c["topk"] = rng.choice([0, 0, 64]) if precision == "bf16" else 0
        c["samples"] = rng.choice([_log_int(rng, 3, 100), _log_int(rng, 100, 1024), 256, 1024])
        most = (0.35e12 if precision == "fp32" else 2.5e12) / (macs * c["samples"])
        c["n"] = _log_int(rng, 16, max(17, min(16384, most)))
    elif kind == "iteration":
        c["samples"] = rng.randint(64, 512)
        c["n"] = 2 * _log_int(rng, 8, max(9, min(512, 0.05e12 / (macs * c["samples"]))))
    elif kind == "alpha":
        c["steps"] = rng.randint(2, 20)
        c["n"] = _log_int(rng, 16, max(17, min(4096, 0.01e12 / (macs * c["steps"]))))
    elif kind == "grad":
        c["n"] = _log_int(rng, 16, 512)
    else:
        c["n"] = _log_int(rng, 16, max(17, min(16384, 0.09e12 / macs)))
        c["intervals"] = "fp32"
        if kind == "crown" and precision != "fp32":
            c["intervals"] = rng.choice(["fp32", "bf16x3", "tf32x3"])
    return c


def _dims(c):
    return [c["s"] + c["k"]] + [int(w) for w in c["hidden"].split("-")] + [c["s"]]


def _macs(c):
    d = _dims(c)
    return sum(a * b for a, b in zip(d, d[1:]))


def work(c):
    kind, n = c["kind"], c["n"]
    if kind == "prune":
        d, p = c["d"], c["n_pick"]
        rest = max(0, n - p)
        row = 8 * d + 16
        return {"bytes": n * row + (2 * p + rest) * row + n, "flops": n + p * d}
    H = c["H"] if kind != "batch" else (c["H"] + c["H_lo"]) / 2
    sumh = sum(_dims(c)[1:-1])
    mac, box = _macs(c) * H * n, n * 8 * c["k"] * H
    if kind == "rollout":
        return {"bytes": box + n * (12 + 4 * c["k"] * H), "flops": 2 * mac * c["samples"]}
    if kind == "ibp":
        return {"bytes": box + n * 4 * (1 + 2 * H * sumh + 2 * (H + 1) * c["s"]), "flops": 4 * mac}
    if kind == "crown":
        return {"bytes": box + n * 4 * (3 + c["k"] * H), "flops": 6 * mac}
    if kind == "alpha":
        return {"bytes": box + n * 4 * (1 + H * sumh), "flops": (4 + 4 * c["steps"]) * mac}
    if kind == "grad":
        return {"bytes": box + n * 4 * (1 + 3 * H * sumh), "flops": 8 * mac}
    if kind == "batch":
        return {"bytes": box + 12 * n, "flops": (4 + 4 * c["steps"]) * mac}
    return {"bytes": 5 * box + 64 * n, "flops": (2 * c["samples"] + 6) * mac}  # iteration


def _split_boxes(d, n, rng):
    """n distinct boxes of [-1, 1]^d after widest-dimension bisection (the pool a search holds), as float32 arrays
    and their path identifiers: a random choice of the 2^levels cells of the grid."""
    levels = max(1, math.ceil(math.log2(n)))
    cell = rng.permutation(1 << levels)[:n].astype(np.int64)
    lo, hi = np.full((n, d), -1.0, np.float32), np.full((n, d), 1.0, np.float32)
    for j in range(levels):
        upper = ((cell >> (levels - 1 - j)) & 1) == 1
        a, b = lo[:, j % d], hi[:, j % d]
        mid = np.float32(0.5) * (a + b)
        lo[:, j % d], hi[:, j % d] = np.where(upper, mid, a), np.where(upper, b, mid)
    return lo, hi, (np.int64(1) << levels) + cell


def _problem(c, seed):
    return W.make_problem(c["s"], c["k"], _dims(c)[1:-1], c["H"], c["rho"], seed)


def _inputs(c, seed):
    """Host inputs of a case."""
    rng = np.random.Generator(np.random.PCG64(seed + 104729))
    n = c["n"]
    if c["kind"] == "prune":
        lo, hi, ids = _split_boxes(c["d"], n, rng)
        lb, ub = W.pool_values(n, seed)
        return {"lo": lo, "hi": hi, "ids": ids, "lb": lb, "ub": ub, "inc": float(np.quantile(lb, 0.9))}
    if c["kind"] == "batch":
        P = c["problems"]
        probs, _ = W.batch_problems(P, seed, c["s"], c["k"], _dims(c)[1:-1], c["H_lo"], c["H"], c["rho"])
        probs[0]["H"] = c["H"]
        params, x0, goal, H, rho = W.pack_batch(probs)
        # rows grouped by problem, as the batched splitter writes them; every problem has its own share of the rows
        share = rng.uniform(0.2, 1.0, P)
        prob = np.sort(rng.choice(P, n, p=share / share.sum())).astype(np.int32)
        d = c["k"] * c["H"]
        lo, hi = np.zeros((n, d), np.float32), np.zeros((n, d), np.float32)
        for p in range(P):
            rows = np.nonzero(prob == p)[0]
            if len(rows):
                dp = c["k"] * int(H[p])
                lo[rows, :dp], hi[rows, :dp], _ = _split_boxes(dp, len(rows), rng)
        return {"dims": probs[0]["dims"], "params": params, "x0": x0, "goal": goal, "H": H, "rho": rho, "lo": lo,
                "hi": hi, "prob": prob}
    p = _problem(c, seed)
    rows = n if c["kind"] != "iteration" else max(n // 2 + n // 4, 1)  # the pool an iteration's children come from
    lo, hi, ids = _split_boxes(c["k"] * c["H"], rows, rng)
    p.update(lo=lo, hi=hi, ids=ids, seed=seed & 0x7FFFFFFF)
    if c["kind"] == "iteration":
        p["lb"], p["ub"] = W.pool_values(rows, seed)
        p["inc"] = float(np.quantile(p["lb"], 0.95))
    if c["kind"] == "grad":
        p["alpha"] = rng.uniform(0.0, 1.0, (n, c["H"], sum(_dims(c)[1:-1]))).astype(np.float32)
    return p


class _State:
    """A case's device inputs, outputs and context (destroyed with it)."""

    def __init__(self):
        self.ctx = None

    def __del__(self):
        if self.ctx is not None:
            B.bab_destroy(self.ctx)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _pool_out(st, cap, d):
    st.out = [torch.zeros(cap, d, device="cuda"), torch.zeros(cap, d, device="cuda"), torch.zeros(cap, device="cuda"),
              torch.zeros(cap, device="cuda"), torch.zeros(cap, dtype=torch.int64, device="cuda")]
    st.keep = torch.zeros(st.lo.shape[0], dtype=torch.uint8, device="cuda")
    st.counts = torch.zeros(3, dtype=torch.int32, device="cuda")
    st.cap = cap


def prepare(c, seed):
    st, h, kind, n = _State(), _inputs(c, seed), c["kind"], c["n"]
    st.case, st.n = c, n
    empty = lambda *shape: torch.zeros(*shape, device="cuda")
    st.lo, st.hi = _dev(h["lo"]), _dev(h["hi"])
    if kind == "prune":
        st.ctx = B.bab_context_create()
        st.lb, st.ub, st.ids = _dev(h["lb"]), _dev(h["ub"]), _dev(h["ids"])
        st.inc = torch.tensor([h["inc"]], dtype=F64, device="cuda")
        _pool_out(st, n + c["n_pick"], c["d"])
        return st
    H, d = c["H"], c["k"] * c["H"]
    if kind == "batch":
        st.ctx = B.bab_load_dynamics_batch(h["dims"], h["params"], c["s"], c["k"])
        st.x0, st.goal, st.H, st.rho, st.prob = (_dev(h[v]) for v in ("x0", "goal", "H", "rho", "prob"))
        st.lb, st.lb_ibp = empty(n), empty(n)
        return st
    st.ctx = B.bab_load_dynamics(h["dims"], h["params"], c["s"], c["k"])
    st.x0, st.goal, st.ids, st.seed = _dev(h["x0"]), _dev(h["goal"]), _dev(h["ids"]), h["seed"]
    if c.get("intervals", "fp32") != "fp32":
        B.bab_set_interval_precision(st.ctx, PRECISION[c["intervals"]])
    st.precision = PRECISION[c["precision"]] if "precision" in c else None
    sumh = sum(_dims(c)[1:-1])
    if kind in ("rollout", "iteration"):
        st.inc_val, st.inc_u = torch.full((1,), math.inf, dtype=F64, device="cuda"), empty(d)
        st.ubs, st.best_u = empty(n), empty(n, d)
        if c.get("topk"):
            B.bab_set_rescore_topk(st.ctx, c["topk"])
    if kind == "iteration":
        st.lb, st.ub = _dev(h["lb"]), _dev(h["ub"])
        st.inc = torch.tensor([h["inc"]], dtype=F64, device="cuda")
        _pool_out(st, st.lo.shape[0] + n // 2, d)
        st.lbs = empty(n)
    elif kind == "ibp":
        st.outs = [empty(n), empty(n, H, sumh), empty(n, H, sumh), empty(n, H + 1, c["s"]), empty(n, H + 1, c["s"])]
    elif kind == "crown":
        st.outs = [empty(n), empty(n), empty(n, d), empty(n)]
    elif kind == "alpha":
        st.lb_best, st.alpha = empty(n), empty(n, H, sumh)
    elif kind == "grad":
        st.prob = CrownProblem(st.ctx, st.x0, st.goal, H, c["rho"], st.lo, st.hi, st.precision)
        st.alpha = _dev(h["alpha"]).requires_grad_(True)
        st.ones = torch.ones(n, device="cuda")
    return st


def run(st):
    c, n = st.case, st.n
    kind = c["kind"]
    if kind == "prune":
        B.bab_prune_branch(st.ctx, c["d"], st.lo, st.hi, st.lb, st.ub, st.ids, n, st.inc, c["n_pick"], ETA, st.cap,
                           *st.out, st.keep, st.counts)
        return [*st.out, st.keep, st.counts]
    H, rho = c["H"], c["rho"]
    if kind == "batch":
        B.bab_bound_batch(st.ctx, st.x0, st.goal, st.H, st.rho, H, c["k"] * H, st.lo, st.hi, st.prob, n, st.lb,
                          alpha_steps=c["steps"], lr=LR, lb_ibp=st.lb_ibp)
        return [st.lb, st.lb_ibp]
    if kind == "rollout":
        B.bab_rollout(st.ctx, st.x0, st.goal, H, rho, st.lo, st.hi, st.ids, n, c["samples"], st.seed, st.precision,
                      st.ubs, st.best_u, st.inc_val, st.inc_u)
        return [st.ubs, st.best_u, st.inc_val, st.inc_u]
    if kind == "ibp":
        B.bab_bound_ibp(st.ctx, st.x0, st.goal, H, rho, st.lo, st.hi, n, *st.outs)
        return list(st.outs)
    if kind == "crown":
        lb, margin, coef, const = st.outs
        B.bab_bound_crown(st.ctx, st.x0, st.goal, H, rho, st.lo, st.hi, n, lb, precision=st.precision, margin=margin,
                          lin_coef=coef, lin_const=const)
        return [lb, margin, coef, const]
    if kind == "alpha":
        B.bab_alpha_optimize(st.ctx, st.x0, st.goal, H, rho, st.lo, st.hi, n, c["steps"], LR, st.lb_best,
                             alpha=st.alpha, precision=st.precision)
        return [st.lb_best, st.alpha]
    if kind == "grad":
        lb = crown_bound(st.alpha, st.prob)
        (g,) = torch.autograd.grad(lb, st.alpha, st.ones)
        return [lb.detach(), g]
    # iteration: split the pool, search the children, bound them
    rows = st.lo.shape[0]
    B.bab_prune_branch(st.ctx, c["k"] * H, st.lo, st.hi, st.lb, st.ub, st.ids, rows, st.inc, n // 2, ETA, st.cap,
                       *st.out, st.keep, st.counts)
    lo, hi, ids = st.out[0], st.out[1], st.out[4]
    B.bab_rollout(st.ctx, st.x0, st.goal, H, rho, lo, hi, ids, n, c["samples"], st.seed, st.precision, st.ubs,
                  st.best_u, st.inc_val, st.inc_u, d_n=st.counts)
    B.bab_bound_crown(st.ctx, st.x0, st.goal, H, rho, lo, hi, n, st.lbs, precision=st.precision, d_n=st.counts)
    return [*st.out, st.keep, st.counts, st.ubs, st.best_u, st.inc_val, st.inc_u, st.lbs]


# ---------------------------------------------------------------------------
# the same quantities in 64 bits, from the formulas
# ---------------------------------------------------------------------------
def _c64(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda().to(F64)


def _layers(dims, params):
    """[(W, b)] in 64 bits from packed parameters: [n_params] or one row per problem [P][n_params]."""
    p, out, off = _c64(params), [], 0
    for i, o in zip(dims, dims[1:]):
        w = p[..., off:off + o * i].reshape(*p.shape[:-1], o, i)
        off += o * i
        out.append((w, p[..., off:off + o]))
        off += o
    return out


def _mul(a, w):
    """a [n, i] times w^T: w [o, i], or one matrix per row [n, o, i]."""
    return a @ w.T if w.dim() == 2 else torch.bmm(w, a.unsqueeze(2)).squeeze(2)


def _mul_t(a, w):
    return a @ w if w.dim() == 2 else torch.bmm(a.unsqueeze(1), w).squeeze(1)


def _intervals(c, layers, x0, lo, hi, H):
    """Interval bounds: per layer and step the pre-activation intervals, and the state intervals."""
    n, k = lo.shape[0], c["k"]
    xl = xu = x0.expand(n, -1)
    pre, xs = [], [(xl, xu)]
    for t in range(H):
        al, au = torch.cat([xl, lo[:, t * k:(t + 1) * k]], 1), torch.cat([xu, hi[:, t * k:(t + 1) * k]], 1)
        step = []
        for i, (w, b) in enumerate(layers):
            ctr, rad = _mul((al + au) / 2, w) + b, _mul((au - al) / 2, w.abs())
            al, au = ctr - rad, ctr + rad
            if i + 1 < len(layers):
                step.append((al, au))
                al, au = al.clamp(min=0), au.clamp(min=0)
        pre.append(step)
        xl, xu = xl + al, xu + au
        xs.append((xl, xu))
    return pre, xs


def _sq_min(lo, hi):
    return torch.where(lo > 0, lo * lo, torch.where(hi < 0, hi * hi, torch.zeros_like(lo)))


def _lb_intervals(c, xs, goal, rho, lo, hi, H, Hrow):
    n, k = lo.shape[0], c["k"]
    out = torch.zeros(n, dtype=F64, device=lo.device)
    for t in range(H):
        v = _sq_min(xs[t + 1][0] - goal, xs[t + 1][1] - goal).sum(1) + \
            (rho * _sq_min(lo[:, t * k:(t + 1) * k], hi[:, t * k:(t + 1) * k])).sum(1)
        out = out + torch.where(Hrow > t, v, torch.zeros_like(v))
    return out


def _crown(c, layers, pre, xs, x0, goal, rho, lo, hi, H, Hrow, alpha=None):
    """Lower bound by backward substitution: (lb, coefficient of u, constant).  alpha: per layer and step the lower
    slopes of the unstable neurons (None: adaptive)."""
    n, s, k = lo.shape[0], c["s"], c["k"]
    lam = torch.zeros(n, s, dtype=F64, device=lo.device)
    cst = torch.zeros(n, dtype=F64, device=lo.device)
    mu = [None] * H
    for t in range(H - 1, -1, -1):
        on = (Hrow > t).to(F64)
        xl, xu = xs[t + 1]
        m = (xl + xu) / 2 - goal
        lam = lam + on[:, None] * 2 * m
        cst = cst - on * (2 * m * goal + m * m).sum(1)
        w, b = layers[-1]
        cst = cst + (lam * b).sum(1)
        A = _mul_t(lam, w)
        for i in range(len(layers) - 2, -1, -1):
            zl, zu = pre[t][i]
            unstable = (zl < 0) & (zu > 0)
            low = alpha[t][i] if alpha is not None else (zu >= -zl).to(F64)
            chord = zu / torch.where(unstable, zu - zl, torch.ones_like(zu))
            up = unstable & (A < 0)
            D = torch.where(zl >= 0, torch.ones_like(zl), torch.where(up, chord, torch.where(unstable, low, torch.zeros_like(zl))))
            w, b = layers[i]
            cst = cst + torch.where(up, -A * chord * zl, torch.zeros_like(A)).sum(1)
            A = A * D
            cst = cst + (A * b).sum(1)
            A = _mul_t(A, w)
        mu[t] = A[:, s:s + k]
        lam = lam + A[:, :s]
    mu = torch.cat(mu, 1)
    cst = cst + (lam * x0).sum(1)
    r = rho if torch.is_tensor(rho) else torch.full((n, 1), float(rho), dtype=F64, device=lo.device)
    inner = torch.minimum(torch.maximum(-mu / (2 * torch.where(r > 0, r, torch.ones_like(r))), lo), hi)
    u = torch.where(r > 0, inner, torch.where(mu >= 0, lo, hi)).detach()
    return cst + (mu * u + r * u * u).sum(1), mu, cst


def _mix(x):
    """The SplitMix64 output function on int64 tensors (64-bit wrap-around)."""
    sh = lambda v, s: (v >> s) & ((1 << (64 - s)) - 1)
    x = x + (0x9E3779B97F4A7C15 - (1 << 64))
    x = (x ^ sh(x, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    x = (x ^ sh(x, 27)) * (0x94D049BB133111EB - (1 << 64))
    return x ^ sh(x, 31)


def _samples(ids, seed, lo, hi, M):
    """The counter-based uniform samples of boxes [lo, hi] (float32): [n, M, d]."""
    d = lo.shape[1]
    hb = _mix(seed ^ _mix(ids))
    mj = (torch.arange(M, device=lo.device)[:, None] << 32) | torch.arange(d, device=lo.device)[None, :]
    h = _mix(hb[:, None, None] ^ mj[None])
    r = ((h >> 40) & 0xFFFFFF).to(torch.float32) * 2.0 ** -24
    return lo[:, None, :] + (hi - lo)[:, None, :] * r


def _objective(c, layers, x0, goal, u):
    """sum_t |x_t - goal|^2 + rho |u_t|^2 of action rows u [rows, d] (64 bits)."""
    x, f = x0.expand(u.shape[0], -1), torch.zeros(u.shape[0], dtype=F64, device=u.device)
    k = c["k"]
    for t in range(c["H"]):
        ut = u[:, t * k:(t + 1) * k]
        a = torch.cat([x, ut], 1)
        for i, (w, b) in enumerate(layers):
            a = torch.addmm(b, a, w.T)
            if i + 1 < len(layers):
                a.clamp_(min=0)
        x = x + a
        f = f + ((x - goal) ** 2).sum(1) + c["rho"] * (ut * ut).sum(1)
    return f


def _search(c, layers, x0, goal, lo, hi, ids, seed):
    """(ub, incumbent value) of the sampled search."""
    n, M, d = lo.shape[0], c["samples"], lo.shape[1]
    ub = torch.empty(n, dtype=F64, device=lo.device)
    step = max(1, (1 << 19) // M)
    for i in range(0, n, step):
        u = _samples(ids[i:i + step], seed, lo[i:i + step], hi[i:i + step], M)
        f = _objective(c, layers, x0, goal, u.reshape(-1, d).to(F64)).reshape(-1, M)
        ub[i:i + step] = f.min(1).values
    return ub, ub.min().reshape(1)


def _prune(lo, hi, lb, ub, ids, inc, n_pick, cap):
    """Pruner, pick-out and widest-dimension split of a pool (host arrays): the outputs of the call, zero beyond
    the rows it writes."""
    n, d = lo.shape
    keep = ~(lb.astype(np.float64) > inc)
    alive = np.nonzero(keep)[0]
    if len(alive) <= n_pick:
        picked = alive
    else:
        n1 = min(n_pick, int(math.ceil(np.float32(ETA) * n_pick)))
        by_ub = alive[np.lexsort((ids[alive], ub[alive]))][:n1]
        rest = np.setdiff1d(alive, by_ub)
        picked = np.sort(np.concatenate([by_ub, rest[np.lexsort((ids[rest], lb[rest]))][:n_pick - n1]]))
    rest = np.setdiff1d(alive, picked)
    P = len(picked)
    src = np.concatenate([np.repeat(picked, 2), rest])
    m = len(src)
    out = [np.zeros((cap, d), np.float32), np.zeros((cap, d), np.float32), np.zeros(cap, np.float32),
           np.zeros(cap, np.float32), np.zeros(cap, np.int64)]
    for o, a in zip(out, (lo, hi, lb, ub, ids)):
        o[:m] = a[src]
    j = np.argmax(hi[picked] - lo[picked], axis=1)
    mid = np.float32(0.5) * (lo[picked, j] + hi[picked, j])
    out[1][np.arange(0, 2 * P, 2), j] = mid
    out[0][np.arange(1, 2 * P, 2), j] = mid
    out[4][0:2 * P:2], out[4][1:2 * P:2] = 2 * ids[picked], 2 * ids[picked] + 1
    return [*out, keep.astype(np.uint8), np.array([2 * P, len(rest), m], np.int32)]


def _slopes(flat, dims):
    """[n, H, sumh] slopes as alpha[t][layer]."""
    parts = torch.split(flat, list(dims[1:-1]), dim=2)
    return [[p[:, t] for p in parts] for t in range(flat.shape[1])]


def _optimise(c, dims, bound, pre, steps):
    """Projected Adam ascent of the slopes from the adaptive start: (best bound, final slopes)."""
    al = torch.stack([torch.cat([(zu >= -zl).to(F64) for zl, zu in step], 1) for step in pre], 1)
    m, v, best = torch.zeros_like(al), torch.zeros_like(al), None
    for i in range(1, steps + 1):
        al.requires_grad_(True)
        lb = bound(_slopes(al, dims))
        (g,) = torch.autograd.grad(lb.sum(), al)
        best = lb.detach() if best is None else torch.maximum(best, lb.detach())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        al = (al.detach() + LR * (m / (1 - 0.9 ** i)) / ((v / (1 - 0.999 ** i)).sqrt() + 1e-8)).clamp(0, 1)
    return best, al


def exact(c, seed):
    h, kind, n = _inputs(c, seed), c["kind"], c["n"]
    if kind == "prune":
        o = _prune(h["lo"], h["hi"], h["lb"], h["ub"], h["ids"], h["inc"], c["n_pick"], n + c["n_pick"])
        return [a.astype(np.float64) if a.dtype == np.float32 else a for a in o]
    if kind == "batch":
        # at most about 20 seconds of small launches
        dims = [int(v) for v in h["dims"]]
        row = torch.as_tensor(h["prob"]).cuda().long()
        layers = [(w[row], b[row]) for w, b in _layers(dims, h["params"])]
        x0, goal, lo, hi = _c64(h["x0"])[row], _c64(h["goal"])[row], _c64(h["lo"]), _c64(h["hi"])
        Hrow, rho = torch.as_tensor(h["H"]).cuda()[row], _c64(h["rho"])[row][:, None]
        pre, xs = _intervals(c, layers, x0, lo, hi, c["H"])
        ibp = _lb_intervals(c, xs, goal, rho, lo, hi, c["H"], Hrow)
        best, _ = _optimise(c, dims, lambda al: _crown(c, layers, pre, xs, x0, goal, rho, lo, hi, c["H"], Hrow, al)[0],
                            pre, c["steps"])
        return [best, ibp]
    dims = [int(v) for v in h["dims"]]
    layers, x0, goal = _layers(dims, h["params"]), _c64(h["x0"]), _c64(h["goal"])
    head = []
    if kind == "iteration":
        o = _prune(h["lo"], h["hi"], h["lb"], h["ub"], h["ids"], h["inc"], n // 2, len(h["lb"]) + n // 2)
        head = [a.astype(np.float64) if a.dtype == np.float32 else a for a in o]
        live = min(n, int(o[6][0]))
        h["lo"], h["hi"], h["ids"] = o[0][:live], o[1][:live], o[4][:live]
    if kind in ("rollout", "iteration"):
        flo, fhi = torch.as_tensor(h["lo"]).cuda(), torch.as_tensor(h["hi"]).cuda()
        ub, val = _search(c, layers, x0, goal, flo, fhi, torch.as_tensor(h["ids"]).cuda(), h["seed"])
        # which of several samples of nearly the same objective is picked is a choice, not a value to compare
        if kind == "rollout":
            return [ub, None, val, None]
    lo, hi = _c64(h["lo"]), _c64(h["hi"])
    H, rho, Hrow = c["H"], c["rho"], torch.full((lo.shape[0],), c["H"], device="cuda")
    pre, xs = _intervals(c, layers, x0, lo, hi, H)
    if kind == "ibp":
        cat = lambda e: torch.stack([torch.cat([z[e] for z in step], 1) for step in pre], 1)
        st = lambda e: torch.stack([x[e] for x in xs], 1)
        return [_lb_intervals(c, xs, goal, rho, lo, hi, H, Hrow), cat(0), cat(1), st(0), st(1)]
    bound = lambda al: _crown(c, layers, pre, xs, x0, goal, rho, lo, hi, H, Hrow, al)
    if kind == "crown":
        lb, mu, cst = bound(None)
        return [lb, None, mu, cst]  # the margin is the library's own rounding allowance
    if kind == "alpha":
        return list(_optimise(c, dims, lambda al: bound(al)[0], pre, c["steps"]))
    if kind == "grad":
        al = _c64(h["alpha"]).requires_grad_(True)
        lb = bound(_slopes(al, dims))[0]
        (g,) = torch.autograd.grad(lb.sum(), al)
        return [lb.detach(), g]
    pad = lambda a: torch.cat([a, torch.zeros(n - live, *a.shape[1:], dtype=F64, device="cuda")])
    return head + [pad(ub), None, val, None, pad(bound(None)[0])]
