"""Executors chosen by a graph's size and shape when the launch shape is left to
the library: inside one block with a queue of ready tasks (up to 65534 tasks) or
with counters for a window of program order (short edges, any number of tasks),
over owned chunks (longer edges), and the same for batches and stitched replay.
COUNTER bodies on chains show a missing or early dependence as a lost update."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


def chains(n, counters, reach, seed, extra=3):
    """Task v adds to counter v % counters after task v - counters, and after up
    to `extra` tasks at most `reach` before it."""
    rng = np.random.default_rng(seed)
    cnt = np.zeros(n, np.int64)
    preds = []
    for v in range(n):
        p = {v - counters} if v >= counters else set()
        if v >= counters and reach > 0:
            p |= {int(x) for x in rng.integers(max(0, v - reach), v, int(rng.integers(0, extra + 1)))}
        cnt[v] = len(p)
        preds += sorted(p)
    return tg._finish(1, [0], [0], np.zeros(n, np.int64), np.zeros(0, np.int64), np.zeros(0, np.int64),
                      np.zeros(0, np.uint8), pred_counts=cnt, pred=np.array(preds, np.int64),
                      body_arg=np.arange(n) % counters, name=f"chains{n}_{counters}_{reach}")


def want(tr, counters, runs):
    return np.bincount(np.asarray(tr.body_arg), minlength=counters) * runs


# (tasks, counters, reach, extra): the window's small and large blocks up to its
# longest edge, past it (queue in a block, owned chunks), many successors per
# task, and sizes around a chunk, the queue's shared part and the id limit
SIZES = [(1, 1, 0, 0), (2, 2, 0, 0), (31, 5, 7, 3), (33, 40, 0, 0), (1000, 16, 160, 3), (5000, 161, 161, 3),
         (5000, 7, 2100, 3), (20000, 900, 2101, 4), (9000, 3, 8999, 12), (65534, 1000, 60000, 1),
         (65535, 1000, 60000, 1), (70000, 64, 100, 2), (70000, 2000, 2100, 3), (80000, 1500, 5000, 3),
         (70000, 40, 16000, 20)]


@pytest.mark.parametrize("n,counters,reach,extra", SIZES, ids=["-".join(map(str, s)) for s in SIZES])
def test_counter_chains_in_every_executor(n, counters, reach, extra):
    ensure_built()
    tr = chains(n, counters, reach, seed=n + reach, extra=extra)
    g = gpu_graph(tr, body=grt.RT_BODY_COUNTER, state_elems=counters)
    g.analyze()
    g.execute()
    g.sync()
    assert np.array_equal(g.state.cpu().numpy(), want(tr, counters, 1))
    for _ in range(2):
        g.replay(3)
        g.sync()
    assert np.array_equal(g.state.cpu().numpy(), want(tr, counters, 7))
    g.close()


@pytest.mark.parametrize("body", [grt.RT_BODY_COUNTER, grt.RT_BODY_SPIN])
@pytest.mark.parametrize("n,counters,reach,extra", [(3001, 60, 0, 0), (3001, 500, 0, 0), (3001, 50, 60, 40), (3001, 500, 600, 40)],
                         ids=["small", "large", "small-wide", "large-wide"])
def test_window_records(n, counters, reach, extra, body):
    """Windows of both sizes, with and without successors past the trigger record."""
    ensure_built()
    tr = chains(n, counters, reach, seed=counters, extra=extra)
    if body == grt.RT_BODY_SPIN:
        g = gpu_graph(tr, body=body, spin_iters=9)
        g.analyze()
        g.replay(2)
        g.sync()
        assert np.array_equal(g.out.cpu().numpy()[:n], oracle.run_bodies(tr, body, spin_iters=9)[1])
    else:
        g = gpu_graph(tr, body=body, state_elems=counters)
        g.analyze()
        g.replay(5)
        g.sync()
        assert np.array_equal(g.state.cpu().numpy(), want(tr, counters, 5))
    g.close()


@pytest.mark.parametrize("body", [grt.RT_BODY_SPIN, grt.RT_BODY_FMA])
def test_bodies_of_wide_and_deep_graphs(body):
    ensure_built()
    for tr in (tg.taskbench(32, 300, "stencil"), tg.taskbench(1024, 70, "random", seed=4),
               tg.taskbench(2000, 40, "stencil"), tg.random_rects(grid=(64, 64), n=3000, side=(2, 24), seed=5)):
        g = gpu_graph(tr, body=body, spin_iters=21)
        g.analyze()
        want_out = oracle.run_bodies(tr, body, spin_iters=21)[1]
        for run in (g.execute, lambda: g.replay(2)):
            g.out.zero_()
            run()
            g.sync()
            assert np.array_equal(g.out.cpu().numpy()[:tr.n], want_out), tr.name
        g.close()


def test_batch_of_every_kind():
    """A batch whose graphs take all four kinds of block, empty and single-task
    graphs among them; each replay adds each task once."""
    ensure_built()
    specs = [(1, 1, 0, 0), (500, 9, 100, 3), (3000, 300, 900, 7), (4000, 5, 3999, 2), (20000, 40, 19000, 2)] * 3
    traces = [chains(n, c, r, seed=k, extra=e) for k, (n, c, r, e) in enumerate(specs)]
    graphs = []
    for tr, (n, c, r, e) in zip(traces, specs):
        g = gpu_graph(tr, body=grt.RT_BODY_COUNTER, state_elems=c)
        g.analyze()
        graphs.append(g)
    b = grt.Batch(graphs)
    for _ in range(3):  # direct, then captured and relaunched
        b.execute(replays=2)
        b.sync()
    assert b.counters()["tasks"] == 2 * sum(t.n for t in traces)
    for tr, g, (n, c, r, e) in zip(traces, graphs, specs):
        assert np.array_equal(g.state.cpu().numpy(), want(tr, c, 6)), tr.name
    b.close()
    for g in graphs:
        g.close()


@pytest.mark.parametrize("pieces,steps,replays", [(3, 2, 40), (16, 30, 7), (90, 11, 3), (700, 5, 25)])
def test_stitched_counters(pieces, steps, replays):
    ensure_built()
    one = tg.stencil_1d(pieces, steps, 16)
    g = gpu_graph(tg.concat([one, one]), body=grt.RT_BODY_COUNTER, state_elems=pieces)
    g.analyze()
    for k in range(2):
        g.execute_stitched(replays)
        assert np.array_equal(g.state.cpu().numpy(), np.full(pieces, steps * replays * (k + 1)))
    g.close()
