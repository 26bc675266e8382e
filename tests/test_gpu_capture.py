"""Resets and rounds inside a caller's stream capture: the captured calls replay,
and the launches of many rounds outside it depend on nothing that a capture
changes on the host without running."""
import os

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

ALPHA, B, SEED = 0.05, 1300, 51


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
    return oracle.make_table([3], [0.068, 0.528], n_buckets=1, iters=1500)


def context(ms, table, inst):
    import torch
    stream = torch.cuda.Stream()
    p = ms.maxsat_default_params(sets=table.sets, n_temps=2, n_buckets=1, alpha=ALPHA,
                                 path=ms.MAXSAT_PATH_SPARSE)
    p.fstar = None
    return ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, stream), stream


def captured(stream, body):
    import torch
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        body()
    return graph


def assert_oracle(ms, table, ctx, inst, rounds):
    g = ms.maxsat_get_state(ctx)
    st = oracle.init_chains(inst.n, B, SEED)
    oracle.gibbs(inst, table, st, rounds, SEED, n_temps=2, n_buckets=1, alpha=ALPHA,
                 threads=os.cpu_count() or 4)
    assert g["t"] == rounds
    assert np.array_equal(g["x"], st.x)
    assert np.array_equal(g["nu"], st.nu32)
    for k in ("cost", "best_cost", "best_x"):
        assert np.array_equal(g[k], getattr(st, k)), k


@pytest.mark.parametrize("steps", [7, 9])
def test_captured_rounds_replay(ms, table, steps):
    """Seven rounds (shares by ticket) or nine (one block per octet)."""
    import torch
    inst = oracle.Instance(*workloads.random_ksat(60, 300, 3, 41))
    ctx, stream = context(ms, table, inst)
    ms.maxsat_reset(ctx, B, SEED)
    ms.maxsat_step(ctx, steps)
    torch.cuda.synchronize()

    def body():
        ms.maxsat_reset(ctx, B, SEED)
        ms.maxsat_step(ctx, steps)

    graph = captured(stream, body)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    stream.synchronize()
    assert_oracle(ms, table, ctx, inst, steps)
    ms.maxsat_step(ctx, 5)
    assert_oracle(ms, table, ctx, inst, steps + 5)
    ms.maxsat_destroy(ctx)


def test_captured_reset_that_never_runs(ms, table):
    """The host starts over at round 0, the chains do not: the same as the round
    of two launches does (profiled)."""
    import torch
    inst = oracle.Instance(*workloads.random_ksat(60, 300, 3, 42))
    states = []
    for profiled in (False, True):
        ctx, stream = context(ms, table, inst)
        ms.maxsat_reset(ctx, B, SEED)
        ms.maxsat_set_profiling(ctx, profiled)
        ms.maxsat_step(ctx, 7)
        torch.cuda.synchronize()
        captured(stream, lambda: ms.maxsat_reset(ctx, B, SEED))
        for steps in (5, 2):
            ms.maxsat_step(ctx, steps)
        states.append(ms.maxsat_get_state(ctx))
        ms.maxsat_destroy(ctx)
    assert states[0]["t"] == states[1]["t"] == 7
    for k in ("x", "nu", "cost", "best_cost", "best_x"):
        assert np.array_equal(states[0][k], states[1][k]), k
