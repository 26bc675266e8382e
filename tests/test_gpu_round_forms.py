"""One formula on 4-bit patterns in the forms of a round that its size rarely
takes: two launches a round (plain and from graphs) and the cooperative launch,
beside the launches of many rounds."""
import os

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

ALPHA = 0.05
EXACT = ("x", "nu", "cost", "best_cost", "best_x")


@pytest.fixture(scope="module")
def ms():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2311_02101_gb300 as m
    return m


def table_of(Q):
    table = oracle.make_table([1, 2, 3], [0.068, 0.528], n_buckets=1, Q=Q, iters=1500)
    for s in table.sets:
        s["W"] = 6.0 * np.asarray(s["W"])  # on the grid, sized as converged fits are
    return table


def state(ms, table, inst, B, seed, steps, Q=4, persist=0, profiled=False):
    import torch
    p = ms.maxsat_default_params(sets=table.sets, n_temps=2, n_buckets=1, alpha=ALPHA,
                                 quant_bits=Q, path=ms.MAXSAT_PATH_SPARSE, steps_per_graph=3,
                                 persistent_round=persist)
    p.fstar = None
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    ms.maxsat_reset(ctx, B, seed)
    ms.maxsat_set_profiling(ctx, profiled)
    assert ms.maxsat_get_persistent_round(ctx) == (persist if not profiled else 0)
    for s in steps:
        ms.maxsat_step(ctx, s)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    return g


def same_as_oracle(g, table, inst, B, seed, rounds):
    st = oracle.init_chains(inst.n, B, seed)
    oracle.gibbs(inst, table, st, rounds, seed, n_temps=2, n_buckets=1, alpha=ALPHA,
                 threads=os.cpu_count() or 4)
    want = dict(x=st.x, nu=st.nu32, cost=st.cost, best_cost=st.best_cost, best_x=st.best_x)
    for k in EXACT:
        assert np.array_equal(g[k], want[k]), k
    np.testing.assert_allclose(g["free_energy"], st.free_energy, rtol=1e-3, atol=1e-6)


def test_more_tiles_than_places(ms):
    """231 tiles of 256 chains: no resident rounds. The two-launch round from
    graphs of three rounds and the cooperative launch give the same free energy
    too."""
    table, B, seed = table_of(4), 59008, 61
    inst = oracle.Instance(*workloads.random_ksat(12, 40, 3, 61))
    two = state(ms, table, inst, B, seed, (7,))
    per = state(ms, table, inst, B, seed, (2, 5), persist=1)
    for k in EXACT + ("free_energy",):
        assert np.array_equal(two[k], per[k]), k
    same_as_oracle(two, table, inst, B, seed, 7)


def test_cooperative_launch_without_4bit_patterns(ms):
    """Contributions too wide for 4-bit patterns, one formula of 256 chains."""
    table, B, seed = table_of(8), 256, 62
    inst = oracle.Instance(*workloads.random_ksat(50, 215, 3, 62))
    g = state(ms, table, inst, B, seed, (2, 9), Q=8, persist=1)
    same_as_oracle(g, table, inst, B, seed, 11)


def test_many_rounds_a_launch_equal_two_launches_at_full_size(ms):
    """Weighted 3-SAT n = 1000, m = 6000, 4096 chains: launches of seven rounds,
    of at most three, and two launches a round."""
    table, B, seed = table_of(4), 4096, 63
    inst = oracle.Instance(*workloads.random_ksat(1000, 6000, 3, 63, 1000))
    two = state(ms, table, inst, B, seed, (7,), profiled=True)
    for persist in (0, 1):
        many = state(ms, table, inst, B, seed, (7,), persist=persist)
        for k in EXACT:
            assert np.array_equal(two[k], many[k]), (persist, k)
        np.testing.assert_allclose(many["free_energy"], two["free_energy"], rtol=1e-3, atol=1e-6)


@pytest.mark.parametrize("n,m,B", [(50, 215, 300), (60, 300, 1300), (600, 3600, 1024)])
def test_rounds_after_measured_choices(ms, n, m, B):
    """The path choice and the tuner run the forms they choose between (one block
    per octet, shares by ticket) on the chains' own buffers before the reset."""
    import torch
    table, seed, rounds = table_of(4), 64, 13
    inst = oracle.Instance(*workloads.random_ksat(n, m, 3, 64, 50))
    p = ms.maxsat_default_params(sets=table.sets, n_temps=2, n_buckets=1, alpha=ALPHA,
                                 quant_bits=4, path=ms.MAXSAT_PATH_AUTO, tune_blocks=1)
    p.fstar = None
    ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
    for b in (B // 2, B):
        ms.maxsat_reset(ctx, b, seed)
    ms.maxsat_step(ctx, 3)
    ms.maxsat_step(ctx, rounds - 3)
    g = ms.maxsat_get_state(ctx)
    ms.maxsat_destroy(ctx)
    same_as_oracle(g, table, inst, B, seed, rounds)
