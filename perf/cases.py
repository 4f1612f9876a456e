"""The measured workloads: what a user of this framework has it do, through its public entry points.

Sizes and input distributions follow ``paper_2110_11226_gb300/synth.py`` (Pagie-1 grids, Higgs-shaped tables, weighted
binary labels, an Epsilon-shaped wide table, ramped half-and-half populations), the tests and ``bench.py``.  Row counts
of real tables are whatever the data gave, so odd ones stand beside the round ones.

A case names one call of a generation: ``evaluate`` (the fused metrics), ``spearman`` (the rank metric), ``predict``,
``host`` (host buffers in, host fitness out), ``tune`` (constant gradient and an Adam step), ``autograd`` (the constants
as a differentiable tensor) and ``breed`` (tournament selection and mutation).  Evaluation and breeding are cases of
their own: winners and children are whole numbers that the last bit of a fitness may decide.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2110_11226_gb300 import gp, synth

SETS = {"basic": synth.BASIC_SET, "paper": synth.PAPER_SET, "full": synth.FULL_SET,
        "extended": synth.EXTENDED_SET}


def listed():
    return [
        # one generation's fitness of a small run: latency and launches
        dict(name="evaluate_pagie_small", kind="evaluate", data="pagie", funcs="basic", depth_min=2,
             depth_max=6, progs=512, rows=4096, feats=2, metric="mse", weighted=False),
        # the headline: Pagie-1 at 16M rows, 4096 programs
        dict(name="evaluate_pagie_16m", kind="evaluate", data="pagie", funcs="full", depth_min=2,
             depth_max=10, progs=4096, rows=1 << 24, feats=2, metric="rmse", weighted=False),
        # regression on a Higgs-shaped table whose row count is no multiple of a vector load
        dict(name="evaluate_table", kind="evaluate", data="table", funcs="full", depth_min=2,
             depth_max=8, progs=2048, rows=2_000_003, feats=28, metric="rmse", weighted=False),
        # classification with class weights, log-loss
        dict(name="evaluate_labels", kind="evaluate", data="labels", funcs="full", depth_min=2,
             depth_max=8, progs=1024, rows=1 << 22, feats=50, metric="logloss", weighted=True),
        # an Epsilon-shaped table: each program touches a few of 2000 columns
        dict(name="evaluate_wide", kind="evaluate", data="labels", funcs="full", depth_min=2,
             depth_max=8, progs=1024, rows=500_000, feats=2000, metric="logloss", weighted=True),
        # the correlation fitness over the fuller function set, weighted rows
        dict(name="evaluate_correlation", kind="evaluate", data="table", funcs="extended", depth_min=2,
             depth_max=8, progs=1024, rows=262_144, feats=28, metric="pearson", weighted=True),
        # the rank fitness
        dict(name="evaluate_rank", kind="spearman", data="pagie", funcs="full", depth_min=2, depth_max=8,
             progs=512, rows=1_000_000, feats=2, metric="spearman", weighted=False),
        # constant tuning between generations: gradient, then one Adam step
        dict(name="tune_pagie", kind="tune", data="pagie", funcs="full", depth_min=4, depth_max=10,
             progs=2048, rows=1 << 20, feats=2, metric="mse", weighted=False),
        # the constants as a tensor of a torch program, small
        dict(name="autograd_small", kind="autograd", data="table", funcs="paper", depth_min=2, depth_max=6,
             progs=256, rows=4099, feats=5, metric="mse", weighted=True),
        # the next population from a fitness array
        dict(name="breed_4096", kind="breed", funcs="full", depth_min=2, depth_max=10, progs=4096, feats=2,
             tourn=20),
        # the predictions of a population on a test table
        dict(name="predict_table", kind="predict", data="table", funcs="full", depth_min=2, depth_max=8,
             progs=256, rows=1_000_003, feats=28),
        # a user with host arrays: copies in, fitness out
        dict(name="evaluate_from_host", kind="host", data="table", funcs="full", depth_min=2, depth_max=8,
             progs=512, rows=100_000, feats=28, metric="mae", weighted=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evaluate"] * 6 + ["spearman", "tune", "tune", "autograd", "breed", "predict", "host"])
    funcs = rng.choice(["basic", "paper", "full", "full", "full", "extended"])
    # a full tree of binary functions alone passes 255 nodes below depth 7, and 16 constants far sooner
    few = kind in ("tune", "autograd")
    deepest = {"basic": 4 if few else 6, "paper": 6 if few else 8}.get(funcs, 10)
    dmin = rng.randint(2, min(4, deepest - 2))
    c = dict(kind=kind, funcs=funcs, depth_min=dmin, depth_max=rng.randint(dmin + 2, deepest))
    if kind == "breed":
        c.update(progs=_log(rng, 200, 8192), feats=rng.choice([2, 5, 28]), tourn=rng.choice([5, 10, 20]))
        return c
    data = rng.choice(["pagie", "table", "labels"])
    feats = 2 if data == "pagie" else rng.choice([1, 3, 8, 28, 50, 200])
    # program-rows of one call, well below the largest listed case's time
    most = dict(evaluate=6e9, spearman=3e8, tune=8e8, autograd=2e8, predict=3e8, host=3e8)[kind]
    if funcs == "extended":
        most /= 4
    progs = _log(rng, 48, 4096)
    rows = _log(rng, 1000, max(2000.0, min(4e6, most / progs, 3e8 / feats)))
    if rng.random() < 0.5:
        rows = max(256, rows // 256 * 256)
    if kind == "spearman":
        metric = "spearman"
    elif kind in ("tune", "autograd"):
        metric = rng.choice(["mse", "mae", "rmse"]) if data != "labels" else "logloss"
    else:
        metric = rng.choice(["mse", "mae", "rmse", "pearson"]) if data != "labels" else "logloss"
    if kind == "host" and metric == "pearson":
        metric = "rmse"
    c.update(data=data, progs=progs, rows=rows, feats=feats)
    if kind != "predict":
        c.update(metric=metric, weighted=rng.random() < 0.4)
    return c


# ---- inputs ------------------------------------------------------------------
def _population(case, seed):
    caps = 16 if case["kind"] in ("tune", "autograd") else None
    return synth.ramped_half_and_half(case["progs"], case["depth_min"], case["depth_max"],
                                      SETS[case["funcs"]], case["feats"], seed, max_consts=caps)


def _hidden(X, g):
    """a smooth target over a few columns, chosen by the generator"""
    F = X.shape[0]
    a, b, c, d = (int(v) for v in torch.randint(0, F, (4,), generator=g, device=X.device).tolist())
    k = torch.rand(3, generator=g, device=X.device) + 0.5
    return k[0] * torch.sin(X[a]) * X[b] + k[1] * X[c].abs() - k[2] * X[d]


def _data(case, seed):
    """X [feats][rows], y, w (or None) on the GPU"""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    F, N = case["feats"], case["rows"]
    if case["data"] == "pagie":
        X = torch.rand(F, N, generator=g, device=dev) * 10.0 - 5.0
        x4 = X.double() ** 4
        y = (x4 / (1.0 + x4)).sum(0).float()
    elif case["data"] == "table":
        X = torch.randn(F, N, generator=g, device=dev)
        heavy = min(4, F)  # the first columns are heavy-tailed
        s = torch.randn(3, heavy, N, generator=g, device=dev).square().mean(0)
        X[:heavy] /= s.sqrt()
        h = _hidden(X, g)
        y = h + 0.1 * h.std() * torch.randn(N, generator=g, device=dev)
    else:
        X = torch.rand(F, N, generator=g, device=dev) * 2.0 - 1.0
        h = _hidden(X, g)
        y = (h > h.median()).float()
        flip = torch.rand(N, generator=g, device=dev) < 0.05
        y = torch.where(flip, 1.0 - y, y)
    w = None
    if case.get("weighted"):
        w = torch.where(y > 0.5, 1.0, 3.0) if case["data"] == "labels" else \
            torch.rand(N, generator=g, device=dev) + 0.5
    return X.contiguous(), y.contiguous(), w


def _pinned(t):
    return None if t is None else t.cpu().pin_memory().numpy()


def prepare(case, seed):
    nodes, off = _population(case, seed)
    s = dict(kind=case["kind"], metric=case.get("metric"))
    if case["kind"] == "breed":
        P = case["progs"]
        g = torch.Generator(device="cuda").manual_seed(seed)
        s.update(progs=gp.nodes_to_device(nodes), off=torch.from_numpy(off).cuda(), feats=case["feats"],
                 fit=torch.randn(P, generator=g, device="cuda").exp(), tourn=case["tourn"], seed=seed,
                 params=gp.make_mut_params(functions=SETS[case["funcs"]]),
                 # the next population's buffers: children are packed, what lies past them stays 0
                 out=torch.zeros(P * 255, dtype=torch.int64, device="cuda"),
                 out_off=torch.zeros(P + 1, dtype=torch.int32, device="cuda"))
        return s
    X, y, w = _data(case, seed)
    if case["kind"] == "host":
        pn = torch.from_numpy(nodes.view(np.int64).copy()).pin_memory().numpy().view(nodes.dtype)
        po = torch.from_numpy(off).pin_memory().numpy()
        s.update(nodes=pn, off=po, X=_pinned(X), y=_pinned(y), w=_pinned(w))
        return s
    s.update(progs=gp.nodes_to_device(nodes), off=torch.from_numpy(off).cuda(), X=X, y=y, w=w)
    if case["kind"] == "tune":
        P = case["progs"]
        s.update(m=torch.zeros(P, 16, device="cuda"), v=torch.zeros(P, 16, device="cuda"), step=0)
    if case["kind"] == "autograd":
        s["consts"] = gp.gp_get_consts(s["progs"], s["off"])
    return s


# ---- one pass ----------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind in ("evaluate", "spearman"):
        return gp.gp_evaluate(s["progs"], s["off"], s["X"], s["y"], s["w"], s["metric"])
    if kind == "predict":
        return gp.gp_predict(s["progs"], s["off"], s["X"])
    if kind == "host":
        return gp.gp_evaluate_host(s["nodes"], s["off"], s["X"], s["y"], s["w"], s["metric"])
    if kind == "tune":
        grad, fit = gp.gp_const_grad(s["progs"], s["off"], s["X"], s["y"], s["w"], s["metric"])
        s["step"] += 1
        gp.gp_adam_step(s["progs"], s["off"], grad, s["m"], s["v"], s["step"])
        return {"grad": grad, "fitness": fit, "consts": gp.gp_get_consts(s["progs"], s["off"]),
                "m": s["m"], "v": s["v"]}
    if kind == "autograd":
        consts = s["consts"].detach().requires_grad_(True)
        fit = gp.fitness_of_constants(consts, s["progs"], s["off"], s["X"], s["y"], s["w"], s["metric"])
        (g,) = torch.autograd.grad(fit.sum(), consts)
        return {"fitness": fit.detach(), "grad": g}
    P = s["fit"].numel()  # breed
    win = gp.gp_tournament_ex(s["fit"], 2 * P, s["tourn"], s["seed"], s["off"], 0.01)
    _, off, mk = gp.gp_mutate(s["progs"], s["off"], s["feats"], win, s["params"], seed=s["seed"] + 1,
                              out=s["out"], out_offsets=s["out_off"])
    return {"winners": win, "progs": s["out"], "offsets": off, "kinds": mk}


# ---- what a pass cannot do without ------------------------------------------
@functools.lru_cache(maxsize=None)
def _mean_nodes(funcs, dmin, dmax, feats, capped):
    """(nodes, function nodes) per program of such a population"""
    nodes, off = synth.ramped_half_and_half(512, dmin, dmax, SETS[funcs], feats, 7,
                                            max_consts=16 if capped else None)
    P = len(off) - 1
    return len(nodes) / P, int((nodes["op"] >= 2).sum()) / P


def work(case):
    L, f = _mean_nodes(case["funcs"], case["depth_min"], case["depth_max"], case["feats"],
                       case["kind"] in ("tune", "autograd"))
    P = case["progs"]
    pop = P * (8.0 * L + 4.0)
    if case["kind"] == "breed":
        # the parents and donors read, the children written; about 12 integer steps per draw
        return {"bytes": 3.0 * pop + 4.0 * P + 8.0 * P, "flops": 24.0 * P * case["tourn"]}
    N = case["rows"]
    used = min(case["feats"], P * (L - f))  # a column that no program names need not be read
    rows = 4.0 * N * (used + (0 if case["kind"] == "predict" else 1) + (1 if case.get("weighted") else 0))
    out = 4.0 * P * (N if case["kind"] == "predict" else 1)
    flops = P * N * (f + (0 if case["kind"] == "predict" else 3))
    if case["kind"] in ("tune", "autograd"):
        out += 4.0 * P * 16 * (5 if case["kind"] == "tune" else 2)
        flops *= 3.0
    if case["kind"] == "spearman":
        flops += P * N * 3.0
    return {"bytes": pop + rows + out, "flops": float(flops)}


# ---- the same in 64 bits, plain torch ----------------------------------------
_BIG = 3.4028234663852886e38  # a value past the float range is infinite, as the entry points say


def _fit32(v):
    return torch.where(v.abs() > _BIG, torch.sign(v) * math.inf, v) if torch.is_tensor(v) else \
        (math.copysign(math.inf, v) if abs(v) > _BIG else v)


def _arity(op):
    return synth.ARITY[int(op)]


_THR = float(np.float32(0.001))


def _apply(op, a, b=None):
    n = synth.OP_NAME[op]
    one, zero = torch.ones((), dtype=torch.float64, device=a.device), torch.zeros((), dtype=torch.float64, device=a.device)
    if n == "add":
        r = a + b
    elif n == "sub":
        r = a - b
    elif n == "mul":
        r = a * b
    elif n == "div":
        r = torch.where(b.abs() < _THR, one, a / b)
    elif n in ("max", "min"):
        left = (a > b) if n == "max" else (a < b)
        r = torch.where(left | a.isnan(), a, b)
    elif n == "sqrt":
        r = a.abs().sqrt()
    elif n == "log":
        r = torch.where(a.abs() < _THR, zero, a.abs().log())
    elif n == "inv":
        r = torch.where(a.abs() < _THR, zero, 1.0 / a)
    elif n == "sq":
        r = a * a
    elif n == "cube":
        r = a * a * a
    elif n == "cbrt":
        r = torch.sign(a) * a.abs().pow(1.0 / 3.0)
    else:
        r = {"exp": torch.exp, "sin": torch.sin, "cos": torch.cos, "tan": torch.tan, "abs": torch.abs,
             "neg": torch.neg, "tanh": torch.tanh, "atan": torch.atan, "sinh": torch.sinh,
             "cosh": torch.cosh}[n](a)
    return _fit32(r)


def _partials(op, a, b, v):
    """d v / d a, d v / d b by the framework's conventions"""
    n = synth.OP_NAME[op]
    z = torch.zeros_like(a)
    if n in ("add", "sub"):
        return z + 1.0, z + (1.0 if n == "add" else -1.0)
    if n == "mul":
        return b, a
    if n == "div":
        p = b.abs() < _THR
        return torch.where(p, z, 1.0 / b), torch.where(p, z, -a / (b * b))
    if n in ("max", "min"):
        left = ((a > b) if n == "max" else (a < b)) | a.isnan()
        return left.double(), (~left).double()
    s = torch.sign(a)
    return {"sqrt": lambda: torch.where(a == 0, z, s / (2.0 * v)), "abs": lambda: s, "neg": lambda: z - 1.0,
            "log": lambda: torch.where(a.abs() < _THR, z, 1.0 / a), "exp": lambda: v,
            "inv": lambda: torch.where(a.abs() < _THR, z, -v * v), "sin": lambda: torch.cos(a),
            "cos": lambda: -torch.sin(a), "tan": lambda: 1.0 + v * v, "sq": lambda: 2.0 * a,
            "cube": lambda: 3.0 * a * a, "cbrt": lambda: torch.where(a == 0, z, 1.0 / (3.0 * v * v)),
            "tanh": lambda: 1.0 - v * v, "atan": lambda: 1.0 / (1.0 + a * a), "sinh": lambda: torch.cosh(a),
            "cosh": lambda: torch.sinh(a)}[n](), None


def _forward(prog, X, tape=None, single=False):
    """the value of one prefix list on every row, by the reverse scan; tape: node -> (value, children);
    single: every value rounded to 32 bits, to see how far that alone moves the outcome"""
    N, dev = X.shape[1], X.device
    stack = []
    for j in range(len(prog) - 1, -1, -1):
        op = int(prog["op"][j])
        if op == 0:
            v, ch = torch.full((N,), float(prog["c"][j]), dtype=torch.float64, device=dev), ()
        elif op == 1:
            v, ch = X[int(prog["feat"][j])].double(), ()
        elif _arity(op) == 1:
            a = stack.pop()
            v, ch = _apply(op, a[1]), (a[0],)
        else:
            a, b = stack.pop(), stack.pop()
            v, ch = _apply(op, a[1], b[1]), (a[0], b[0])
        if single and op >= 2:
            v = v.float().double()
        if tape is not None:
            tape[j] = (v, ch)
        stack.append((j, v))
    return stack[0][1]


def _losses(metric, p, y):
    if metric == "mae":
        return (p - y).abs()
    if metric == "logloss":
        c = torch.where(p >= 0, 1.0 - y, y)
        return torch.where(c == 0, torch.zeros_like(p), c * p.abs()) + torch.log1p(torch.exp(-p.abs()))
    return _fit32((p - y) ** 2)


def _ranks(v):
    """1-based ranks, ties sharing the mean of their positions"""
    s, order = torch.sort(v)
    _, inv, cnt = torch.unique_consecutive(s, return_inverse=True, return_counts=True)
    end = torch.cumsum(cnt, 0).double()
    mean = end - (cnt.double() - 1.0) / 2.0
    r = torch.empty_like(v)
    r[order] = mean[inv]
    return r


def _pearson(a, b, w, sw):
    ma, mb = (w * a).sum() / sw, (w * b).sum() / sw
    da, db = a - ma, b - mb
    va, vb, cov = (w * da * da).sum(), (w * db * db).sum(), (w * da * db).sum()
    if not bool(torch.isfinite(va) & torch.isfinite(cov)):
        return math.nan
    # a constant's rounding is no variance
    if float(va) <= 1e-24 * float(sw) * float(ma * ma) or float(va) <= 0 or float(vb) <= 0:
        return 0.0
    return float(cov.abs() / (va * vb).sqrt())


def _gradient(prog, X, y, w, sw, metric, single=False):
    tape = {}
    p = _forward(prog, X, tape, single)
    loss = _losses(metric, p, y)
    fit = float((w * loss).sum() / sw)
    if metric == "mae":
        d = torch.sign(p - y)
    elif metric == "logloss":
        d = torch.sigmoid(p) - y
    else:
        d = 2.0 * (p - y)
    scale = 1.0 / float(sw)
    if metric == "rmse":
        fit = math.sqrt(fit) if fit == fit and fit >= 0 else fit
        scale = scale / (2.0 * fit) if fit > 0 else 0.0
    adj = {0: w * d}
    grad, k = [0.0] * 16, 0
    for j in range(len(prog)):
        op = int(prog["op"][j])
        v, ch = tape[j]
        g = adj.pop(j)
        if op == 0:
            if k < 16:
                grad[k] = float(g.sum()) * scale
            k += 1
        elif ch:
            a, b = tape[ch[0]][0], tape[ch[1]][0] if len(ch) == 2 else None
            pa, pb = _partials(op, a, b, v)
            adj[ch[0]] = g * pa
            if pb is not None:
                adj[ch[1]] = g * pb
    return fit, grad


def _settled(v, single):
    """v, or None where rounding every value to 32 bits moves it by over 1%: such outputs (the sine of a
    huge argument, a protected operator's decision) have no value that a float evaluation could meet"""
    fine = torch.isfinite(v) & torch.isfinite(single)
    off = torch.linalg.vector_norm((v - single)[fine])
    return v if bool(off <= 0.01 * torch.linalg.vector_norm(v[fine])) else None


def _fitness(prog, X, y, w, sw, metric, yr, single):
    v = _forward(prog, X, single=single)
    if metric == "spearman":
        return math.nan if bool(v.isnan().any()) else _pearson(_ranks(v), yr, w, sw)
    if metric == "pearson":
        return _pearson(v, y, w, sw)
    f = float((w * _losses(metric, v, y)).sum() / sw)
    return math.sqrt(f) if metric == "rmse" and f == f else f


def exact(case, seed):
    if case["kind"] == "breed":
        return None  # whole numbers
    nodes, off = _population(case, seed)
    N, P = case["rows"], case["progs"]
    slow = {"tune": 4.0, "autograd": 4.0, "spearman": 4.0}.get(case["kind"], 1.0) * (2.0 if case["funcs"] == "extended" else 1.0)
    if slow * P * N > 9e9:
        return None
    X, y, w = _data(case, seed)
    progs = [nodes[off[i]:off[i + 1]] for i in range(P)]
    if case["kind"] == "predict":
        out = torch.empty(P, N, dtype=torch.float64, device=X.device)
        one = torch.empty(P, N, dtype=torch.float32, device=X.device)
        for i, p in enumerate(progs):
            out[i] = _forward(p, X)
            one[i] = _forward(p, X, single=True)
        return _settled(out, one.double())
    y = y.double()
    w = torch.ones_like(y) if w is None else w.double()
    sw = w.sum()
    metric = case["metric"]
    if case["kind"] in ("tune", "autograd"):
        both = []
        for single in (False, True):
            got = [_gradient(p, X, y, w, sw, metric, single) for p in progs]
            both.append([torch.tensor([g[k] for g in got], dtype=torch.float64) for k in (0, 1)])
        fit, grad = (_settled(v, s) for v, s in zip(*both))
        if case["kind"] == "autograd":
            return {"fitness": fit, "grad": grad}
        # the first Adam step (lr 0.01, betas 0.9 and 0.999) divides a gradient by its own size: the
        # sign of one that is rounding noise is anyone's, so the constants after it have no such value
        return {"grad": grad, "fitness": fit, "consts": None,
                "m": None if grad is None else 0.1 * grad, "v": None if grad is None else 0.001 * grad * grad}
    yr = _ranks(y) if metric == "spearman" else None
    out, one = (torch.tensor([_fitness(p, X, y, w, sw, metric, yr, single) for p in progs], dtype=torch.float64)
                for single in (False, True))
    out = _settled(out, one)
    return out.numpy() if out is not None and case["kind"] == "host" else out
