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
