"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the package's public entry points, on seeded random formulas of the
kinds that the benchmark and the tests use (weighted and unweighted random 3-SAT, mixed clause
lengths 2..12 with hard clauses, batches of uneven formulas). A case is a dict of plain values;
`prepare` builds what a program holds before the call, `run` makes one pass and returns its
outputs, `work` says what a pass cannot do without and `exact` gives the outputs that have a
64-bit value independent of the library.
"""
from __future__ import annotations

import concurrent.futures
import math
import os

import numpy as np
import torch

import paper_2311_02101_gb300 as ms

FSTAR = [0.068, 0.528]  # the default temperature pair
BUCKET_GAMMA = 0.5


def listed():
    return [
        # a small unweighted formula (the plain-method configuration): 200 rounds of a few
        # thousand clause evaluations each, where launches and latency count
        dict(name="solve_small", kind="solve", n=50, m=215, B=256, steps=200, wmax=1, path=0),
        # a small weighted formula with a ragged number of restarts (the two temperatures meet
        # inside a group of eight chains)
        dict(name="solve_odd", kind="solve", n=317, m=1571, B=500, steps=100, wmax=1000, path=0),
        # the benchmark's formula: weighted Max-3-SAT, 4096 restarts
        dict(name="solve_w3sat", kind="solve", n=1000, m=6000, B=4096, steps=200, wmax=1000,
             path=0),
        # industrial shape: clause lengths 2..12, hard and soft clauses, 1024 restarts
        dict(name="solve_mixed", kind="solve_mixed", n=20000, m=100000, B=1024, steps=100),
        # many formulas of uneven size in one context
        dict(name="solve_batch", kind="solve_batch", count=96, n_lo=100, n_hi=5000, B=256,
             steps=50),
        # the matrix-product formulation asked for by name, on ragged sizes
        dict(name="solve_dense", kind="solve", n=777, m=4001, B=2000, steps=50, wmax=1000, path=1),
        # exact scoring of a block of assignments with the solver's context
        dict(name="eval_w3sat", kind="eval", n=1000, m=6000, B=4096, wmax=1000),
        # the same on mixed clause lengths, with a ragged number of assignments
        dict(name="eval_mixed", kind="eval_mixed", n=20000, m=100000, B=1000),
        # scoring without a context or an allocation, inside a latency-critical loop
        dict(name="eval_noalloc", kind="noalloc", n=250, m=1065, B=100, wmax=1000),
        # a search loop: rounds, unit propagation beside rounds, the merge, rounds, and the
        # whole state read back (as for a checkpoint)
        dict(name="search_up", kind="search_up", n=1000, m=6000, B=1024, steps=100, wmax=1000),
        # one training step of the learned proposal on a batch of formulas
        dict(name="train", kind="train", count=48, n_lo=500, n_hi=2000, layers=3),
        # the learned proposal's prediction for one formula
        dict(name="propose", kind="propose", n=2000, m=12000, layers=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve_mixed", "solve_batch", "solve_dense",
                       "eval", "eval_mixed", "noalloc", "search_up", "train", "propose"])
    if kind in ("solve", "solve_dense"):
        dense = kind == "solve_dense"
        n = _log_int(rng, 50, 2000 if dense else 5000)
        m = int(round(n * rng.uniform(4.0, 8.0)))
        B = _log_int(rng, 64, 4096)
        cap = 4.0e8 if dense else 4.9e9
        steps = int(min(200, max(10, cap / (float(m) * B))))
        while float(m) * B * steps > cap and B > 64:
            B = max(64, B // 2)
        return dict(kind="solve", n=n, m=m, B=B, steps=steps, wmax=rng.choice([1, 100, 1000]),
                    path=1 if dense else 0)
    if kind == "solve_mixed":
        n = _log_int(rng, 500, 20000)
        m = int(n * rng.uniform(3.0, 5.0))
        B = _log_int(rng, 64, 1024)
        return dict(kind=kind, n=n, m=m, B=B,
                    steps=int(min(100, max(20, 1.0e10 / (float(m) * B)))))
    if kind == "solve_batch":
        return dict(kind=kind, count=rng.randint(4, 96), n_lo=100, n_hi=_log_int(rng, 300, 5000),
                    B=rng.choice([64, 200, 256]), steps=rng.randint(10, 50))
    if kind == "eval":
        n = _log_int(rng, 100, 5000)
        return dict(kind=kind, n=n, m=int(round(n * rng.uniform(4.0, 8.0))),
                    B=_log_int(rng, 16, 8192), wmax=rng.choice([1, 1000]))
    if kind == "eval_mixed":
        n = _log_int(rng, 500, 20000)
        return dict(kind=kind, n=n, m=int(n * rng.uniform(3.0, 5.0)), B=_log_int(rng, 16, 1024))
    if kind == "noalloc":
        n = _log_int(rng, 50, 1000)
        return dict(kind=kind, n=n, m=int(round(n * rng.uniform(4.0, 8.0))),
                    B=_log_int(rng, 1, 2048), wmax=rng.choice([1, 1000]))
    if kind == "search_up":
        n = _log_int(rng, 100, 1500)
        return dict(kind=kind, n=n, m=int(round(n * rng.uniform(4.0, 8.0))),
                    B=_log_int(rng, 64, 680), steps=rng.randint(20, 100),
                    wmax=rng.choice([1, 1000]))
    if kind == "train":
        return dict(kind=kind, count=rng.randint(1, 48), n_lo=500, n_hi=_log_int(rng, 600, 2000),
                    layers=rng.choice([1, 2, 3]))
    n = _log_int(rng, 500, 10000)
    return dict(kind="propose", n=n, m=int(round(n * rng.uniform(4.0, 8.0))),
                layers=rng.choice([1, 2, 3]))


# ------------------------------------------------------------------ formulas
def _formula(rng, n, lengths, weights):
    """(n, clause offsets, DIMACS literals, weights): distinct variables per clause, uniform, each
    negated with probability 1/2."""
    m, kmax = len(lengths), int(lengths.max())
    used = np.arange(kmax)[None, :] < lengths[:, None]
    var = rng.integers(0, n, size=(m, kmax))
    while True:
        s = np.sort(np.where(used, var, -1 - np.arange(kmax)[None, :]), axis=1)
        again = np.nonzero((s[:, 1:] == s[:, :-1]).any(axis=1))[0]
        if not len(again):
            break
        var[again] = rng.integers(0, n, size=(len(again), kmax))
    sign = rng.integers(0, 2, size=var.shape) * 2 - 1
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    return n, off, ((var + 1) * sign)[used].astype(np.int32), weights


def _three_sat(rng, n, m, wmax):
    w = rng.integers(1, wmax + 1, size=m).astype(np.int64)
    return _formula(rng, n, np.full(m, 3, np.int64), w)


def _mixed(rng, n, m):
    lengths = np.minimum(1 + rng.geometric(0.4, size=m), 12).astype(np.int64)
    w = rng.integers(1, 101, size=m).astype(np.int64)
    hard = rng.choice(m, size=m // 10, replace=False)
    soft = np.ones(m, bool)
    soft[hard] = False
    w[hard] = 1 + int(w[soft].sum())
    return _formula(rng, n, lengths, w)


def _batch(rng, count, n_lo, n_hi, ratio_lo=4.0, ratio_hi=8.0, wmax=1000):
    """Formulas of uneven size (n log-uniform, m / n uniform); the sizes belong to the case."""
    sizes, out = np.random.default_rng(7919 * count + n_hi), []
    for _ in range(count):
        n = int(round(math.exp(sizes.uniform(math.log(n_lo), math.log(n_hi)))))
        out.append(_three_sat(rng, n, int(round(n * sizes.uniform(ratio_lo, ratio_hi))), wmax))
    return out


def _formulas(case, seed):
    """The formulas of a case (a list), and the generator that goes on drawing its other inputs."""
    rng = np.random.default_rng(1000003 * seed + 17)
    kind = case["kind"]
    if kind in ("solve_mixed", "eval_mixed"):
        return [_mixed(rng, case["n"], case["m"])], rng
    if kind == "solve_batch":
        return _batch(rng, case["count"], case["n_lo"], case["n_hi"]), rng
    if kind == "train":
        return _batch(rng, case["count"], case["n_lo"], case["n_hi"], 6.0, 6.0), rng
    return [_three_sat(rng, case["n"], case["m"], case.get("wmax", 1000))], rng


# ---------------------------------------------------- clause RBMs, fitted once
_SETS = {}


def _fit(key):
    length, bucket, temp = key
    hidden = 3 if length <= 3 else length + 1
    iters = 6000 if length <= 7 else max(1000, 6000 >> (length - 7))
    W, b = ms.maxsat_fit_or_rbm(length, hidden, FSTAR[temp] * (1.0 + bucket * BUCKET_GAMMA), 4,
                                iters)
    return dict(len=length, bucket=bucket, temp=temp, W=W, b=b)


def _params(lengths, path=0):
    """Parameters with the clause RBMs of these lengths (a program fits them once and keeps them)."""
    keys = [(k, j, e) for k in lengths for j in range(4) for e in range(2)]
    todo = [k for k in keys if k not in _SETS]
    if todo:
        with concurrent.futures.ThreadPoolExecutor(max(1, min(16, os.cpu_count() or 1))) as pool:
            _SETS.update(zip(todo, pool.map(_fit, todo)))
    return ms.maxsat_default_params(sets=[_SETS[k] for k in keys], path=path)


def _theta(rng, layers):
    """He-normal weights and zero biases of the proposal network, as one FP32 vector."""
    parts = [rng.normal(0.0, math.sqrt(2.0 / 3), 64 * 3) for _ in range(2)]
    for _ in range(2 * layers):
        parts += [rng.normal(0.0, math.sqrt(2.0 / 128), 64 * 128), np.zeros(64)]
    parts += [rng.normal(0.0, 1.0 / 8, 64), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


def _assignments(rng, B, n):
    return rng.integers(0, 2, size=(B, n), dtype=np.uint8)


def _labels(rng, formulas):
    """Training labels: a variable takes the polarity of most of its occurrences, with noise (what
    a solver's best assignment looks like)."""
    out = []
    for n, _, lits, _ in formulas:
        lean = np.bincount(np.abs(lits) - 1, np.sign(lits), n) + rng.normal(0.0, 3.0, n)
        out.append((lean > 0).astype(np.uint8))
    return np.concatenate(out)


# ------------------------------------------------------------------- the pass
def prepare(case, seed):
    kind = case["kind"]
    formulas, rng = _formulas(case, seed)
    state = dict(kind=kind, case=case, seed=int(rng.integers(1, 2 ** 31)))
    if kind == "noalloc":
        n, off, lits, w = formulas[0]
        state.update(n=n, off=torch.from_numpy(off).cuda(), lits=torch.from_numpy(lits).cuda(),
                     w=None if case["wmax"] == 1 else torch.from_numpy(w).cuda(),
                     x=torch.from_numpy(_assignments(rng, case["B"], n)).cuda(),
                     cost=torch.zeros(case["B"], dtype=torch.int64, device="cuda"))
        return state
    stream = state["stream"] = torch.cuda.Stream()
    mixed = kind in ("solve_mixed", "eval_mixed")
    params = _params(range(2, 13) if mixed else [3], case.get("path", 0))
    if kind in ("solve_batch", "train"):
        state["ctx"] = ms.maxsat_create_batch(formulas, params, stream)
    else:
        state["ctx"] = ms.maxsat_create(*formulas[0], params, stream)
    if kind in ("eval", "eval_mixed"):
        # the context of a solver that has started its chains (and so chosen its path)
        ms.maxsat_reset(state["ctx"], case["B"], state["seed"])
        x = _assignments(rng, case["B"], formulas[0][0])
        state.update(x=torch.from_numpy(x).cuda(),
                     cost=torch.zeros(case["B"], dtype=torch.int64, device="cuda"))
    elif kind in ("train", "propose"):
        state["model"] = ms.maxsat_mp_create(case["layers"], 0)
        ms.maxsat_mp_set_params(state["model"], _theta(rng, case["layers"]))
        if kind == "train":
            state["y"] = torch.from_numpy(_labels(rng, formulas)).cuda()
        else:
            state["prob"] = torch.zeros(formulas[0][0], dtype=torch.float32, device="cuda")
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind in ("solve", "solve_mixed", "solve_batch"):
        cost, best = ms.maxsat_solve(state["ctx"], case["B"], case["steps"], state["seed"])
        return dict(cost=cost, best=best)
    if kind in ("eval", "eval_mixed"):
        ms.maxsat_eval(state["ctx"], state["x"], state["cost"])
        return state["cost"]
    if kind == "noalloc":
        ms.maxsat_eval_noalloc(state["n"], state["off"], state["lits"], state["w"], state["x"],
                               state["cost"])
        return state["cost"]
    if kind == "search_up":
        ctx = state["ctx"]
        ms.maxsat_reset(ctx, case["B"], state["seed"])
        ms.maxsat_step(ctx, case["steps"])
        ms.maxsat_up_begin(ctx)
        ms.maxsat_step(ctx, 20)
        ms.maxsat_up_end(ctx)
        ms.maxsat_step(ctx, 20)
        ms.maxsat_score(ctx)
        return ms.maxsat_get_state(ctx)
    if kind == "train":
        loss = ms.maxsat_mp_gradient(state["model"], state["ctx"], state["y"])
        ms.maxsat_mp_adam(state["model"], state["ctx"], 3e-3)
        theta, grad = ms.maxsat_mp_get_params(state["model"])
        return dict(loss=loss, theta=theta, grad=grad)
    ms.maxsat_mp_forward(state["model"], state["ctx"], state["prob"])
    return state["prob"]


# ------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind in ("solve_batch", "train"):
        mid = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        n = case["count"] * mid
        m = 6.0 * n
    else:
        n, m = float(case["n"]), float(case["m"])
    nnz = m * (3.5 if kind in ("solve_mixed", "eval_mixed") else 3.0)
    formula = 4.0 * nnz + 8.0 * m  # literals and weights
    if kind in ("train", "propose"):
        rows = n + m
        layer = 2.0 * 64 * 128 * rows + 4.0 * 64 * nnz  # dense layers, two signed means
        flops = case["layers"] * layer + 2.0 * 3 * 64 * rows + 2.0 * 64 * n
        if kind == "propose":
            return dict(bytes=formula + 4.0 * n, flops=flops)
        return dict(bytes=formula + n + 12.0 * (449 + 16512 * case["layers"]), flops=3.0 * flops)
    B = float(case["B"])
    if kind in ("eval", "eval_mixed", "noalloc"):
        return dict(bytes=B * n + 8.0 * B + formula, flops=B * (nnz + m))
    # per clause and chain: its literals, its hidden units' draws (five operations of the counter
    # generator and a comparison each), their contributions to its literals; per variable and
    # chain: a draw, the moving average
    units = 5.4 if kind == "solve_mixed" else 3.0
    length = nnz / m
    step = B * (m * (length + 6.0 * units + length) + n * 10.0)
    steps = case["steps"] + (40 if kind == "search_up" else 0)
    out = n + 8.0 if kind != "search_up" else B * (6.0 * n + 20.0)
    return dict(bytes=formula + out, flops=steps * step)


# ------------------------------------------------------------- 64-bit outputs
def _padded(formula):
    """Literals as an m x kmax table (0 where a clause is shorter)."""
    _, off, lits, _ = formula
    lengths = np.diff(off)
    table = np.zeros((len(lengths), int(lengths.max())), np.int64)
    table[np.arange(table.shape[1])[None, :] < lengths[:, None]] = lits
    return table


def _exact_cost(formula, x, weighted):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    table = torch.from_numpy(_padded(formula)).to(dev)
    w = torch.from_numpy(formula[3]).to(dev).double() if weighted else None
    costs = []
    for row in torch.from_numpy(x).to(dev):
        truth = row[(table.abs() - 1).clamp(min=0)].bool() ^ (table < 0)
        unsat = ~(truth & (table != 0)).any(dim=1)
        costs.append((w * unsat).sum().long() if weighted else unsat.sum())
    return torch.stack(costs)


def _exact_network(case, formulas, theta, y):
    """Loss, parameters after one Adam step and gradient (with labels), or the predictions."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    base = np.concatenate([[0], np.cumsum([f[0] for f in formulas])])
    n = int(base[-1])
    lits = np.concatenate([np.sign(f[2]) * (np.abs(f[2]) + b) for f, b in zip(formulas, base)])
    lengths = np.concatenate([np.diff(f[1]) for f in formulas])
    m = len(lengths)
    var = torch.from_numpy((np.abs(lits) - 1).astype(np.int64)).to(dev)
    clause = torch.from_numpy(np.repeat(np.arange(m), lengths)).to(dev)
    sign = torch.from_numpy(np.sign(lits).astype(np.float64)).to(dev)
    length = torch.from_numpy(lengths.astype(np.float64)).to(dev)
    w = torch.from_numpy(np.concatenate([f[3] for f in formulas]).astype(np.float64)).to(dev)
    zero = torch.zeros(n, dtype=torch.float64, device=dev)
    deg, pos = zero.index_add(0, var, sign.abs()), zero.index_add(0, var, (sign > 0).double())
    f = torch.stack([torch.where(deg > 0, pos / deg.clamp(min=1) - 0.5, zero),
                     torch.log1p(deg) / 4, torch.ones_like(zero)], 1)
    g = torch.stack([torch.log(w) / 8, length / 4, torch.ones_like(w)], 1)
    master = torch.from_numpy(theta).to(dev)
    rounded = master.to(torch.bfloat16).double()
    full = master.double()
    at, leaves = 0, []

    def take(shape, weight):
        nonlocal at
        size = math.prod(shape)
        t = (rounded if weight else full)[at:at + size].reshape(shape).clone().requires_grad_()
        at += size
        leaves.append(t)
        return t

    def mean(index, size, rows, count):
        total = torch.zeros(size, 64, dtype=torch.float64, device=dev).index_add(0, index, rows)
        return total / count.clamp(min=1)[:, None]

    hv, hc = torch.relu(f @ take((64, 3), True).T), torch.relu(g @ take((64, 3), True).T)
    for _ in range(case["layers"]):
        Wc, bc = take((64, 128), True), take((64,), False)
        Wv, bv = take((64, 128), True), take((64,), False)
        mc = mean(clause, m, sign[:, None] * hv[var], length)
        hc = torch.relu(torch.cat([mc, hc], 1) @ Wc.T + bc)
        av = mean(var, n, sign[:, None] * hc[clause], deg)
        hv = torch.relu(torch.cat([av, hv], 1) @ Wv.T + bv)
    z = hv @ take((64,), False) + take((1,), False)
    if y is None:
        return torch.sigmoid(z).detach().cpu()
    t = torch.from_numpy(y).to(dev).double()
    loss = (torch.nn.functional.softplus(z) - t * z).mean()
    grads = torch.autograd.grad(loss, leaves, allow_unused=True)
    grad = torch.cat([(torch.zeros_like(p) if d is None else d).reshape(-1)
                      for p, d in zip(leaves, grads)])
    new = full - 3e-3 * grad / (grad.abs() + 1e-8)  # the first Adam step
    return dict(loss=float(loss.detach()), theta=new.cpu(), grad=grad.cpu())


def exact(case, seed):
    kind = case["kind"]
    formulas, rng = _formulas(case, seed)
    rng.integers(1, 2 ** 31)  # the solver's seed
    if kind in ("eval", "eval_mixed", "noalloc"):
        x = _assignments(rng, case["B"], formulas[0][0])
        return _exact_cost(formulas[0], x, kind == "eval_mixed" or case["wmax"] > 1)
    if kind in ("train", "propose"):
        theta = _theta(rng, case["layers"])
        y = _labels(rng, formulas) if kind == "train" else None
        return _exact_network(case, formulas, theta, y)
    return None  # a sampled trajectory: whole numbers, fixed by the seed
