"""Exact costs on packed assignments (maxsat_eval off the dense path,
maxsat_eval_noalloc, the merges): assignment counts around the 32-bit words,
rows that start off a 4-byte boundary, any nonzero byte as true, clause runs
that end inside a warp, weights beyond 2^31 per run, a batch whose formulas
start at odd variables. Whole numbers, equal to the oracle's."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ms():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2311_02101_gb300 as m
    return m


@pytest.fixture(scope="module")
def table():
    return oracle.make_table(list(range(1, 7)), [0.3], n_buckets=1, iters=300)


def random_formula(n, m, kmax, wmax, seed):
    rng = np.random.default_rng(seed)
    cl = [list(rng.integers(1, n + 1, size=k) * (1 - 2 * rng.integers(0, 2, size=k)))
          for k in rng.integers(0, kmax + 1, size=m)]
    return oracle.Instance.from_clauses(n, cl, [int(w) for w in rng.integers(1, wmax, size=m)])


def costs(ms, table, insts, X, offset):
    import torch
    stream = torch.cuda.Stream()
    p = ms.maxsat_default_params(sets=table.sets, n_temps=1, n_buckets=1)
    p.fstar = None
    args = [(i.n, i.off, i.lits, i.w) for i in insts]
    ctx = (ms.maxsat_create_batch(args, p, stream) if len(args) > 1 else
           ms.maxsat_create(*args[0], p, stream))
    buf = torch.zeros(X.size + 8, dtype=torch.uint8, device="cuda")
    xd = buf[offset:offset + X.size].view(X.shape)
    xd.copy_(torch.from_numpy(X))
    out = torch.full((len(insts), X.shape[0]), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(2):  # back to back: the second reuses the packed words
        ms.maxsat_eval(ctx, xd, out)
    torch.cuda.synchronize()
    ms.maxsat_destroy(ctx)
    return out.cpu().numpy()


@pytest.mark.parametrize("n,m,kmax,wmax,B,offset", [
    (1, 1, 1, 2, 1, 0), (37, 33, 3, 9, 31, 1), (128, 512, 3, 1000, 32, 0),
    (129, 513, 6, 2 ** 40, 33, 3), (1000, 6000, 3, 1000, 100, 0), (1003, 777, 6, 5, 1025, 2),
    (4, 0, 3, 5, 70, 0), (1024, 1024, 6, 9, 64, 0), (1025, 1024, 3, 9, 33, 1),
    (1023, 1025, 3, 2 ** 33, 31, 2), (300, 1024, 3, 2 ** 40, 95, 3)])
def test_packed_costs(ms, table, n, m, kmax, wmax, B, offset):
    inst = random_formula(n, m, kmax, wmax, n + B)
    X = np.random.default_rng(B).integers(0, 2, size=(B, n), dtype=np.uint8)
    X[::3] *= 129  # any nonzero byte is true
    got = costs(ms, table, [inst], X, offset)[0]
    assert np.array_equal(got, oracle.evaluate(inst, (X != 0).astype(np.uint8)))


def test_packed_costs_of_a_batch(ms, table):
    insts = [random_formula(n, m, 4, 2000, n) for n, m in
             [(7, 40), (33, 0), (250, 5000), (64, 31), (5, 1)]]
    n = sum(i.n for i in insts)
    X = np.random.default_rng(0).integers(0, 2, size=(67, n), dtype=np.uint8)
    got = costs(ms, table, insts, X, 0)
    at = 0
    for k, i in enumerate(insts):
        assert np.array_equal(got[k], oracle.evaluate(i, X[:, at:at + i.n].copy())), k
        at += i.n


@pytest.mark.parametrize("B", [65, 257, 301])
def test_merges_of_odd_chain_counts(ms, B):
    """2 B candidates, two of them in the last group of four bytes that are
    packed together; the other two bytes are columns that nobody writes, in
    memory where earlier contexts kept floats."""
    import os
    import torch
    tab = oracle.make_table([1, 2, 3], [0.068, 0.528], n_buckets=1, iters=300)
    seed, alpha, tau = 31 + B, 0.05, 0.2
    p = ms.maxsat_default_params(sets=tab.sets, n_temps=2, n_buckets=1, alpha=alpha,
                                 path=ms.MAXSAT_PATH_SPARSE)
    p.fstar = None
    inst = random_formula(400, 1700, 3, 9, B)
    bp2 = (2 * B + 255) // 256 * 256
    # blocks of the candidates' size that held nu: n Bp floats
    olds = [random_formula(400 * bp2 // 1024, 900, 3, 9, k) for k in range(12)]
    held = [ms.maxsat_create(i.n, i.off, i.lits, i.w, p, torch.cuda.Stream()) for i in olds]
    for c in held:
        ms.maxsat_reset(c, 256, 5)
        ms.maxsat_step(c, 20)
    torch.cuda.synchronize()
    for c in held:
        ms.maxsat_destroy(c)
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    prob = np.random.default_rng(B).random(inst.n).astype(np.float32)
    st = oracle.init_chains(inst.n, B, seed)
    kw = dict(n_temps=2, n_buckets=1, alpha=alpha, threads=os.cpu_count() or 4)
    ms.maxsat_reset(ctx, B, seed)
    for _ in range(3):
        ms.maxsat_step(ctx, 2)
        ms.maxsat_up(ctx)
        ms.maxsat_step(ctx, 1)
        ms.maxsat_propose_flips(ctx, prob, tau)
        oracle.gibbs(inst, tab, st, 2, seed, **kw)
        oracle.up_merge(inst, st, oracle.unit_prop(inst, st.x, st.nu32))
        oracle.gibbs(inst, tab, st, 1, seed, **kw)
        oracle.up_merge(inst, st, oracle.flip_proposals(st.x, prob, tau))
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    assert np.array_equal(g["x"], st.x)
    assert np.array_equal(g["nu"], st.nu32)


def test_packed_costs_of_the_largest_batch(ms, table):
    """65535 formulas, one of them with more than 64 slabs of 32 clauses: one
    run of slabs per formula at least, more would not fit a launch's grid."""
    import torch
    n_inst, B, at = 65535, 3, 40000
    big = random_formula(50, 2100, 3, 9, 1)
    w = np.arange(1, n_inst + 1, dtype=np.int64)
    insts = [(1, np.array([0, 1]), np.array([1], np.int32), w[k:k + 1]) for k in range(n_inst)]
    insts[at] = (big.n, big.off, big.lits, big.w)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=1, n_buckets=1)
    p.fstar = None
    ctx = ms.maxsat_create_batch(insts, p, torch.cuda.Stream())
    X = np.random.default_rng(2).integers(0, 2, size=(B, n_inst - 1 + big.n), dtype=np.uint8)
    out = torch.full((n_inst, B), -1, dtype=torch.int64, device="cuda")
    xd = torch.from_numpy(X).cuda()
    torch.cuda.synchronize()
    ms.maxsat_eval(ctx, xd, out)
    torch.cuda.synchronize()
    ms.maxsat_destroy(ctx)
    got = out.cpu().numpy()
    first = np.where(np.arange(n_inst) <= at, np.arange(n_inst), np.arange(n_inst) - 1 + big.n)
    unit = (w[:, None] * (1 - X[:, first].T)).astype(np.int64)
    unit[at] = oracle.evaluate(big, X[:, at:at + big.n].copy())
    assert np.array_equal(got, unit)


def test_evaluations_in_flight_together(ms, table):
    """Evaluations of several assignment blocks launched one after another into
    the same packed words, each overlapping the end of the one before."""
    import torch
    inst = random_formula(1000, 6000, 3, 9, 3)
    stream = torch.cuda.Stream()
    p = ms.maxsat_default_params(sets=table.sets, n_temps=1, n_buckets=1)
    p.fstar = None
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, stream)
    X = np.random.default_rng(4).integers(0, 2, size=(5, 2048, inst.n), dtype=np.uint8)
    xd = torch.from_numpy(X).cuda()
    out = torch.full((60, X.shape[1]), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for k in range(len(out)):
        ms.maxsat_eval(ctx, xd[k % 5], out[k])
    stream.synchronize()
    ms.maxsat_destroy(ctx)
    want = np.stack([oracle.evaluate(inst, x) for x in X])
    assert np.array_equal(out.cpu().numpy(), want[np.arange(len(out)) % 5])
