"""sim_batch_step on handles with step graphs runs them beside one another, as the graph of a whole
batch does."""
import threading
import time

import pytest

import paper_2303_00689_gb300 as kx
from tests.test_gpu_eigen import lattice

pytestmark = pytest.mark.gpu


def per_step(step):
    """Shortest of five timings of 8 steps, in seconds a step."""
    step(8)                                             # captures what is captured on first use
    best = 1e9
    for _ in range(5):
        t = time.perf_counter()
        step(8)
        best = min(best, time.perf_counter() - t)
    return best / 8


@pytest.mark.parametrize("n,count", [(480, 12), (720, 8)])
def test_handles_with_graphs_are_stepped_together(n, count):
    hs = [lattice(n, kx.SIM_PREC_MIXED, i, kernel=kx.SIM_KERNEL_KRYLOV) for i in range(2 * count)]
    batch = kx.sim_batch_create(hs[count:])
    try:
        for h in hs[:count]:
            kx.sim_enable_graphs(h)
        one_graph = per_step(lambda k: kx.sim_batch_run(batch, k))
        graphs = per_step(lambda k: kx.sim_batch_step(hs[:count], k))
        # one after the other, or two at a time, they take more than twice as long
        assert graphs <= 1.5 * one_graph
    finally:
        kx.sim_batch_destroy(batch)
        for h in hs:
            kx.sim_destroy(h)


def test_handles_stepped_by_threads_of_their_own_share_the_device():
    """Eight threads, a handle of n = 480 each: large eigensolver grids fit two at a time, so steps that
    meet take small ones, as a batch does (and the thread of a handle alone the large one again)."""
    hs = [lattice(480, kx.SIM_PREC_MIXED, i, kernel=kx.SIM_KERNEL_KRYLOV) for i in range(8)]
    try:
        for h in hs:
            kx.sim_enable_graphs(h)
        together = per_step(lambda k: kx.sim_batch_step(hs, k))

        def threads(k):
            ts = [threading.Thread(target=kx.sim_step, args=(h, k)) for h in hs]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        assert per_step(threads) <= 1.3 * together
    finally:
        for h in hs:
            kx.sim_destroy(h)
