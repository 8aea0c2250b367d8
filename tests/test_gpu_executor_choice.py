"""Which executor a graph runs on when its launch shape is left to the library,
as its statistics report it: 1 block of 128 or 512 threads (inside one block),
blocks of 32 threads (owned chunks) or more (the ring). The results are the
oracle's whichever it is."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph
from test_gpu_block_exec import explicit, layered

pytestmark = pytest.mark.gpu


def shape_of(tr, iters, config=None):
    """(blocks, threads) of one execution, its results checked."""
    ensure_built()
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=iters)
    g.analyze()
    if config:
        g.exec_config(*config)
    g.execute()
    g.sync()
    st = g.stats()
    assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=iters)[1])
    g.close()
    return st["exec_blocks"], st["exec_threads"]


def roots_then_chain(roots, n):
    """Tasks 0 .. roots - 1 without predecessors, then a chain: edges of one task, a front as wide as the roots."""
    v = np.arange(roots, n)
    return explicit(n, np.stack([v, v - 1], 1))


def test_many_roots_of_long_bodies_leave_the_block():
    """Short edges alone do not make a front narrow: the roots are ready together."""
    assert shape_of(explicit(701, np.zeros((0, 2))), 30000)[0] > 1
    assert shape_of(roots_then_chain(700, 1401), 20000)[0] > 1
    # of short bodies, or few, they stay: in a block of 16 warps, and of 4 only where those hold them
    assert shape_of(explicit(701, np.zeros((0, 2))), 8) == (1, 512)
    assert shape_of(roots_then_chain(200, 900), 8) == (1, 512)
    assert shape_of(roots_then_chain(70, 900), 8) == (1, 128)
    assert shape_of(explicit(60, np.zeros((0, 2))), 1000) == (1, 128)


def random_steps(w, t, seed, longest=False):
    """w x t tasks of random fan-in 5; longest: and an edge from the first to the last."""
    tr = tg.taskbench(w, t, "random", seed=seed, encode="explicit")
    rows = np.stack([np.repeat(np.arange(tr.n), np.diff(tr.pred_off)), tr.pred], 1)
    return explicit(tr.n, np.concatenate([rows, [[tr.n - 1, 0]]]) if longest else rows)


def test_wide_small_graphs_are_not_put_in_one_block():
    """Steps of a thousand tasks want more than one SM's lanes, however few tasks there are in all."""
    assert shape_of(random_steps(1024, 20, 3), 8) == (32, 32)
    assert shape_of(layered(1000, 20, 8), 64) == (32, 32)
    assert shape_of(random_steps(600, 90, 4, longest=True), 8)[0] > 32  # the ring
    assert shape_of(layered(100, 300, 8, longest=True), 8)[0] > 32
    # a few hundred wide, or dense and narrow, with edges too long for owned chunks: the queue in a block
    assert shape_of(random_steps(300, 90, 4, longest=True), 8) == (1, 512)
    assert shape_of(layered(40, 600, 8, longest=True), 8) == (1, 512)
    # a handful of tasks
    assert shape_of(explicit(200, [(v, 0) for v in range(1, 200)] + [(199, v) for v in range(1, 199)]), 8) == (1, 512)


@pytest.mark.parametrize("n,iters,in_blocks", [(1000, 16000, False), (1000, 500, True), (300, 3000, False),
                                               (4000, 8, False), (64, 8000, True)])
def test_batches_of_long_independent_bodies(n, iters, in_blocks):
    """Graphs whose roots alone outweigh one SM's lanes run on the grid; the block executors never count idle polls."""
    ensure_built()
    tr = explicit(n, np.concatenate([[[n - 1, 0]], [[n - 2, 0]]]))
    want = oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=iters)[1]
    graphs = [gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=iters) for _ in range(3)]
    for g in graphs:
        g.analyze()
    b = grt.Batch(graphs)
    for _ in range(2):
        for g in graphs:
            g.out.zero_()
        b.execute(replays=2)
        b.sync()
        c = b.counters()
        assert c["tasks"] == 6 * n and (c["idle"] == 0) == in_blocks
        for g in graphs:
            assert np.array_equal(g.out.cpu().numpy(), want)
    b.close()
    for g in graphs:
        g.close()


def test_owned_chunks_hold_a_whole_step_and_no_long_bodies():
    ensure_built()
    assert shape_of(tg.taskbench(1024, 70, "stencil"), 8) == (32, 32)
    assert shape_of(tg.taskbench(2000, 40, "stencil"), 8) == (64, 32)
    assert shape_of(tg.taskbench(3000, 30, "stencil"), 1000) == (128, 32)
    assert shape_of(tg.taskbench(1024, 40, "random", seed=2), 1000) == (32, 32)
    assert shape_of(tg.taskbench(2000, 10, "stencil"), 2500)[1] == 64  # two warps a block: the ring


def test_window_of_sixteen_warps_and_long_bodies():
    ensure_built()
    assert shape_of(tg.taskbench(100, 60, "stencil"), 500) == (1, 512)
    assert shape_of(tg.taskbench(100, 60, "stencil"), 1200) == (32, 32)
    assert shape_of(tg.taskbench(60, 60, "stencil"), 1200) == (1, 128)
