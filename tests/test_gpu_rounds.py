"""Rounds where their kernels change form: variables in more than 32 clauses
(several incidence windows), octets of chains across two temperatures,
temperature blocks too small, contributions or weights too large for 4-bit
patterns, several chain tiles, formulas smaller than a block, clauses whose
hidden units fill one to four chunks of three. Every case against the oracle, bit for bit (the free
energy within the 1e-3 bar of the other parity tests)."""
import os

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

FSTARS = [0.05, 0.068, 0.12, 0.25, 0.4, 0.528]


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


def table_for(temps, Q, longest):
    key = temps, Q, longest
    if key not in _tables:
        table = oracle.make_table(list(range(1, longest + 1)), FSTARS[:temps], n_buckets=2, Q=Q,
                                  iters=1500 if longest <= 3 else 100)
        for s in table.sets:
            s["W"] = 6.0 * np.asarray(s["W"])  # on the grid, sized as converged fits are
        _tables[key] = table
    return _tables[key]


def short_clauses(n, m, seed, longest=3, wmax=9):
    """m clauses of 0..longest literals, repeated and opposite literals included."""
    rng = np.random.default_rng(seed)
    cl = [list(rng.integers(1, n + 1, size=k) * (1 - 2 * rng.integers(0, 2, size=k)))
          for k in rng.integers(0, longest + 1, size=m)]
    return oracle.Instance.from_clauses(n, cl, [int(w) for w in rng.integers(1, wmax, size=m)])


CASES = {
    # name: (instance, chains, temperatures, quantisation bits)
    "high-degree": (lambda: oracle.Instance(*workloads.random_ksat(9, 400, 3, 1)), 264, 2, 4),
    "straddle": (lambda: oracle.Instance(*workloads.random_ksat(40, 171, 3, 2, 50)), 300, 3, 4),
    "short": (lambda: short_clauses(23, 90, 3), 520, 6, 4),
    "thin-temperatures": (lambda: short_clauses(23, 90, 4), 44, 6, 4),
    "wide-contributions": (lambda: short_clauses(23, 90, 5), 256, 2, 8),
    "one-clause": (lambda: short_clauses(3, 1, 6), 8, 1, 4),
    "no-clause": (lambda: oracle.Instance.from_clauses(5, [], []), 40, 2, 4),
    "tiles": (lambda: oracle.Instance(*workloads.random_ksat(70, 333, 3, 7, 30000)), 1300, 2, 4),
    "more-variables-than-clauses": (lambda: oracle.Instance(*workloads.random_ksat(900, 20, 3, 8)),
                                    256, 2, 4),
    "lengths-0-9": (lambda: short_clauses(60, 300, 9, 9), 520, 3, 4),
    "lengths-thin-temperatures": (lambda: short_clauses(60, 200, 10, 9), 44, 6, 4),
    "lengths-wide-contributions": (lambda: short_clauses(60, 200, 11, 9), 256, 2, 8),
    "lengths-heavy": (lambda: short_clauses(60, 200, 12, 9, 2 ** 33), 256, 2, 4),
    "lengths-0-12": (lambda: short_clauses(60, 300, 14, 12), 264, 2, 4),
    "lengths-high-degree": (lambda: short_clauses(12, 500, 13, 9), 300, 2, 4),
}


@pytest.mark.parametrize("profiled", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_rounds_match_oracle(ms, case, profiled):
    """`profiled` keeps the two-launch round (events around every launch)."""
    import torch
    make, B, temps, Q = CASES[case]
    inst, alpha, seed = make(), 0.05, 21
    longest = 12 if case == "lengths-0-12" else 9 if case.startswith("lengths") else 3
    table = table_for(temps, Q, longest)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=temps, n_buckets=2, alpha=alpha,
                                 quant_bits=Q, path=ms.MAXSAT_PATH_SPARSE, steps_per_graph=4)
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    ms.maxsat_reset(ctx, B, seed)
    if profiled:
        ms.maxsat_set_profiling(ctx, True)
    for steps in (1, 7, 4):
        ms.maxsat_step(ctx, steps)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    st = oracle.init_chains(inst.n, B, seed)
    oracle.gibbs(inst, table, st, 12, seed, n_temps=temps, n_buckets=2, alpha=alpha,
                 threads=os.cpu_count() or 4)
    assert g["t"] == 12
    assert np.array_equal(g["x"], st.x)
    assert np.array_equal(g["nu"], st.nu32)
    for k in ("cost", "best_cost", "best_x"):
        assert np.array_equal(g[k], getattr(st, k)), k
    np.testing.assert_allclose(g["free_energy"], st.free_energy, rtol=1e-3, atol=1e-6)


@pytest.mark.parametrize("case", [c for c in CASES if not c.startswith("lengths")])
def test_long_steps_match_oracle(ms, case):
    """Steps of eight rounds and more: small formulas take all of a step's
    rounds with one block per octet."""
    import torch
    make, B, temps, Q = CASES[case]
    inst, alpha, seed = make(), 0.05, 22
    table = table_for(temps, Q, 3)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=temps, n_buckets=2, alpha=alpha,
                                 quant_bits=Q, path=ms.MAXSAT_PATH_SPARSE)
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    ms.maxsat_reset(ctx, B, seed)
    for steps in (8, 1, 11):
        ms.maxsat_step(ctx, steps)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    st = oracle.init_chains(inst.n, B, seed)
    oracle.gibbs(inst, table, st, 20, seed, n_temps=temps, n_buckets=2, alpha=alpha,
                 threads=os.cpu_count() or 4)
    assert g["t"] == 20
    assert np.array_equal(g["x"], st.x)
    assert np.array_equal(g["nu"], st.nu32)
    for k in ("cost", "best_cost", "best_x"):
        assert np.array_equal(g[k], getattr(st, k)), k
    np.testing.assert_allclose(g["free_energy"], st.free_energy, rtol=1e-3, atol=1e-6)


def test_contexts_side_by_side_match_oracle(ms):
    """Rounds of several contexts on streams of their own, in flight together:
    blocks of each run whatever shares of its rounds are open, however many of
    them the device has room for."""
    import torch
    table, alpha, B = table_for(2, 4, 3), 0.05, 1300
    p = ms.maxsat_default_params(sets=table.sets, n_temps=2, n_buckets=2, alpha=alpha,
                                 quant_bits=4, path=ms.MAXSAT_PATH_SPARSE)
    insts = [oracle.Instance(*workloads.random_ksat(60 + 25 * k, 300 + 110 * k, 3, 30 + k))
             for k in range(4)]
    ctxs = [ms.maxsat_create(i.n, i.off, i.lits, i.w, p, torch.cuda.Stream()) for i in insts]
    for k, ctx in enumerate(ctxs):
        ms.maxsat_reset(ctx, B, 40 + k)
    for steps in (7, 6, 7):
        for ctx in ctxs:
            ms.maxsat_step(ctx, steps)
    for k, (inst, ctx) in enumerate(zip(insts, ctxs)):
        g = ms.maxsat_get_state(ctx)
        ms.maxsat_destroy(ctx)
        st = oracle.init_chains(inst.n, B, 40 + k)
        oracle.gibbs(inst, table, st, 20, 40 + k, n_temps=2, n_buckets=2, alpha=alpha,
                     threads=os.cpu_count() or 4)
        assert np.array_equal(g["x"], st.x)
        assert np.array_equal(g["nu"], st.nu32)
        for name in ("cost", "best_cost", "best_x"):
            assert np.array_equal(g[name], getattr(st, name)), name


def test_many_temperatures_match_oracle(ms):
    """64 temperatures and 6 clause groups: more (group, temperature) pairs than
    the 256-byte record blocks are built for, in steps of eight rounds and more
    and in shorter ones."""
    import torch
    temps, B, seed, alpha = 64, 520, 23, 0.05
    table = oracle.make_table([1, 2, 3], list(np.linspace(0.05, 0.5, temps)), n_buckets=2, Q=4,
                              iters=50)
    for s in table.sets:
        s["W"] = 6.0 * np.asarray(s["W"])
    inst = short_clauses(23, 90, 15)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=temps, n_buckets=2, alpha=alpha,
                                 quant_bits=4, path=ms.MAXSAT_PATH_SPARSE)
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    ms.maxsat_reset(ctx, B, seed)
    for steps in (8, 1, 11):
        ms.maxsat_step(ctx, steps)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    st = oracle.init_chains(inst.n, B, seed)
    oracle.gibbs(inst, table, st, 20, seed, n_temps=temps, n_buckets=2, alpha=alpha,
                 threads=os.cpu_count() or 4)
    assert np.array_equal(g["x"], st.x)
    assert np.array_equal(g["nu"], st.nu32)
    for k in ("cost", "best_cost", "best_x"):
        assert np.array_equal(g[k], getattr(st, k)), k
    np.testing.assert_allclose(g["free_energy"], st.free_energy, rtol=1e-3, atol=1e-6)
