"""Contexts of several host threads, one context per thread: launches of one
thread must not change what another thread's launches may use."""
import threading

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


def test_kernels_of_one_variant_with_different_shared_memory(ms):
    """Evaluations of formulas of 45000 and 20000 variables (180 and 80 KB of
    shared memory a block, the same kernel) from two threads."""
    import torch
    table = oracle.make_table([3], [0.3], n_buckets=1, iters=100)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=1, n_buckets=1)
    p.fstar = None
    wrong, start = [], threading.Barrier(2)

    def work(n):
        try:
            inst = oracle.Instance(*workloads.random_ksat(n, 2000, 3, n))
            stream = torch.cuda.Stream()
            ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, stream)
            X = np.random.default_rng(n).integers(0, 2, size=(32, n), dtype=np.uint8)
            xd = torch.from_numpy(X).cuda()
            out = torch.full((32,), -1, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            start.wait()
            for _ in range(4000):
                ms.maxsat_eval(ctx, xd, out)
            stream.synchronize()
            if not np.array_equal(out.cpu().numpy(), oracle.evaluate(inst, X)):
                wrong.append(f"{n}: costs")
            ms.maxsat_destroy(ctx)
        except Exception as e:  # reported by the main thread
            wrong.append(f"{n}: {e}")

    threads = [threading.Thread(target=work, args=(n,)) for n in (45000, 20000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong


def test_graphs_captured_beside_contexts_that_come_and_go(ms):
    """One thread's rounds are captured into graphs again for every seed, while
    another creates and destroys contexts (which waits for the device, a call
    that a capture in flight refuses and that invalidates it)."""
    import os
    import torch
    table = oracle.make_table([1, 2, 3, 4], [0.068, 0.528], n_buckets=1, iters=300)
    p = ms.maxsat_default_params(sets=table.sets, n_temps=2, n_buckets=1, alpha=0.05,
                                 steps_per_graph=3, path=ms.MAXSAT_PATH_SPARSE)
    p.fstar = None
    inst = oracle.Instance(*workloads.random_ksat(60, 200, 4, 71))
    small = oracle.Instance(*workloads.random_ksat(20, 60, 3, 72))
    wrong, start, done = [], threading.Barrier(2), threading.Event()

    def rounds():
        try:
            ctx = ms.maxsat_create(inst.n, inst.off, inst.lits, inst.w, p, torch.cuda.Stream())
            start.wait()
            for seed in range(400):
                ms.maxsat_reset(ctx, 256, seed)
                ms.maxsat_step(ctx, 7)
            g = ms.maxsat_get_state(ctx)
            ms.maxsat_destroy(ctx)
            st = oracle.init_chains(inst.n, 256, 399)
            oracle.gibbs(inst, table, st, 7, 399, n_temps=2, n_buckets=1, alpha=0.05,
                         threads=os.cpu_count() or 4)
            if not (np.array_equal(g["x"], st.x) and np.array_equal(g["cost"], st.cost)):
                wrong.append("states")
        except Exception as e:
            wrong.append(f"rounds: {e}")
        done.set()

    def contexts():
        try:
            start.wait()
            while not done.is_set():
                ctx = ms.maxsat_create(small.n, small.off, small.lits, small.w, p,
                                       torch.cuda.Stream())
                ms.maxsat_reset(ctx, 64, 1)
                ms.maxsat_step(ctx, 4)
                ms.maxsat_destroy(ctx)
        except Exception as e:
            wrong.append(f"contexts: {e}")

    threads = [threading.Thread(target=f) for f in (rounds, contexts)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
