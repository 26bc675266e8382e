"""Dense rounds on 4-bit hidden patterns where their kernels change form:
tiles of 256 and of 128 chains, octets and quads of chains across two
temperatures, K-blocks that end early, variables in no clause, one to three
literals a clause, and the byte patterns that remain where temperature blocks are
small. Sampled chains against the
oracle, bit for bit (the free energy within the 1e-3 bar of the other parity
tests)."""
import os

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

FSTARS = [0.05, 0.068, 0.12, 0.25, 0.4, 0.528, 0.3]


@pytest.fixture(scope="module")
def ms():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2311_02101_gb300 as m
    return m


_tables = {}


def table_for(temps, Q):
    key = temps, Q
    if key not in _tables:
        table = oracle.make_table([1, 2, 3], FSTARS[:temps], n_buckets=2, Q=Q, iters=1500)
        for s in table.sets:
            s["W"] = 6.0 * np.asarray(s["W"])
        _tables[key] = table
    return _tables[key]


def distinct(n, m, seed):
    """m clauses of 1..3 distinct variables, unequal weights."""
    rng = np.random.default_rng(seed)
    cl = []
    for _ in range(m):
        v = rng.choice(n, size=min(n, int(rng.integers(1, 4))), replace=False) + 1
        cl.append(list(v * (1 - 2 * rng.integers(0, 2, size=v.size))))
    return oracle.Instance.from_clauses(n, cl, [int(w) for w in rng.integers(1, 30, size=m)])


CASES = {
    # name: (instance, chains, temperatures, quantisation bits)
    "one-clause": (lambda: distinct(3, 1, 0), 8, 1, 4),
    "short": (lambda: distinct(129, 515, 1), 260, 2, 4),
    "straddle": (lambda: distinct(127, 700, 2), 300, 7, 4),
    "idle-variables": (lambda: distinct(900, 65, 3), 520, 3, 4),
    "tiles-of-256": (lambda: oracle.Instance(*workloads.random_ksat(2561, 9000, 3, 4, 20)), 1024, 3, 4),
    "many-tiles": (lambda: oracle.Instance(*workloads.random_ksat(1300, 5000, 3, 5)), 4000, 3, 4),
    "thin-temperatures": (lambda: distinct(60, 250, 6), 44, 6, 4),
}


@pytest.mark.parametrize("case", list(CASES))
def test_dense_rounds_match_oracle(ms, case):
    import torch
    make, B, temps, Q = CASES[case]
    inst, alpha, seed, T = make(), 0.05, 23, 5
    table = table_for(temps, Q)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=temps, n_buckets=2, alpha=alpha,
                                 quant_bits=Q, path=ms.MAXSAT_PATH_DENSE, steps_per_graph=2)
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    ms.maxsat_reset(ctx, B, seed)
    ms.maxsat_step(ctx, 2)
    ms.maxsat_step(ctx, T - 2)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    # the chains beside every temperature boundary, the first and the last
    edge = [b + d for e in range(1, temps) for b in [(e * B) // temps] for d in (-1, 0, 1)]
    rows = np.array(sorted({0, B - 1} | {b for b in edge if 0 <= b < B}))
    st = oracle.init_chains(inst.n, len(rows), seed, chain_ids=rows, B_total=B)
    oracle.gibbs(inst, table, st, T, seed, n_temps=temps, n_buckets=2, alpha=alpha,
                 threads=os.cpu_count() or 4)
    assert g["t"] == T
    assert np.array_equal(g["x"][rows], st.x)
    assert np.array_equal(g["nu"][rows], st.nu32)
    for k in ("cost", "best_cost", "best_x"):
        assert np.array_equal(g[k][rows], getattr(st, k)), k
    np.testing.assert_allclose(g["free_energy"][rows], st.free_energy, rtol=1e-3, atol=1e-6)
