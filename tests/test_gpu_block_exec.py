"""The executor that runs a graph inside one block from a queue of ready tasks:
graphs of up to 65534 tasks whose edges are too long for a window of program
order."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


def explicit(n, preds, counters=1):
    """A trace of n tasks without rectangles; preds: (task, predecessor) rows, task v adds to counter v % counters."""
    preds = np.unique(np.asarray(preds, np.int64).reshape(-1, 2), axis=0)
    return tg._finish(1, [0], [0], np.zeros(n, np.int64), np.zeros(0, np.int64), np.zeros(0, np.int64),
                      np.zeros(0, np.uint8), pred_counts=np.bincount(preds[:, 0], minlength=n), pred=preds[:, 1],
                      body_arg=np.arange(n) % counters, name=f"explicit{n}_{len(preds)}")


def chain(n, *more):
    """One chain of n tasks and an edge from the first to the last, longer than any window."""
    v = np.arange(1, n)
    return explicit(n, np.concatenate([np.stack([v, v - 1], 1), [[n - 1, 0]], *[np.asarray(m).reshape(-1, 2) for m in more]]))


@pytest.mark.parametrize("n", [17000, 20000, 65534])
def test_every_run_runs_every_task(n):
    """Each launch runs all of its tasks, whichever warp finds the queue empty first."""
    ensure_built()
    tr = chain(n, [(v, v - 700) for v in range(701, n, 3)])
    g = gpu_graph(tr, body=grt.RT_BODY_COUNTER, state_elems=1)
    g.analyze()
    for k in range(60):
        g.execute()
        g.sync()
        st = g.stats()
        assert (st["exec_blocks"], st["exec_threads"]) == (1, 512)
        assert st["exec_counters"]["tasks"] == n
    assert int(g.state.cpu()[0]) == 60 * n
    g.close()


def test_a_run_past_its_limit_reports_and_recovers():
    """A limit far below the time between two reports: the launch ends with RT_ERR_TIMEOUT, the graph stays usable."""
    ensure_built()
    tr = chain(17000)
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=900, timeout_ns=100_000)
    g.analyze()
    with pytest.raises(grt.GrtError) as e:
        g.execute()
        g.sync()
    assert e.value.status == grt.RT_ERR_TIMEOUT
    g.close()
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=900)
    g.analyze()
    g.execute()
    g.sync()
    st = g.stats()
    assert (st["exec_blocks"], st["exec_threads"], st["exec_counters"]["tasks"]) == (1, 512, tr.n)
    g.close()


def test_a_warp_that_never_waits_reports_its_progress():
    """A chain runs in one warp, which always keeps its next task: 60000 tasks take several times the limit, the 4096
    between two reports a small part of it."""
    ensure_built()
    n = 60000
    tr = chain(n)
    g = gpu_graph(tr, body=grt.RT_BODY_COUNTER, state_elems=1, timeout_ns=15_000_000)
    g.analyze()
    g.execute()
    g.sync()
    st = g.stats()
    assert (st["exec_blocks"], st["exec_threads"]) == (1, 512)
    assert int(g.state.cpu()[0]) == n
    g.close()


@pytest.mark.parametrize("longest", [False, True], ids=["window", "queue"])
def test_edges_of_many_replays_are_counted_in_64_bits(longest):
    """255 layers of 256 tasks, each after all of the layer before it: 16.6M edges a run, over 2^32 in 264 runs."""
    ensure_built()
    w, t, runs = 256, 255, 264
    v = np.repeat(np.arange(w, w * t), w)
    preds = np.stack([v, (v // w - 1) * w + np.tile(np.arange(w), w * (t - 1))], 1)
    if longest:
        preds = np.concatenate([preds, [[w * t - 1, 0]]])
    tr = explicit(w * t, preds, counters=w)
    g = gpu_graph(tr, body=grt.RT_BODY_COUNTER, state_elems=w, timeout_ns=2_000_000_000)
    g.analyze()
    if longest:  # a batch of one
        b = grt.Batch([g])
        b.execute(replays=runs)
        b.sync()
        c = b.counters()
        b.close()
    else:
        g.replay(runs)
        g.sync()
        st = g.stats()
        assert (st["exec_blocks"], st["exec_threads"]) == (1, 512)
        c = st["exec_counters"]
    assert c["tasks"] == runs * tr.n
    assert c["edges"] == runs * len(preds) > 1 << 32
    assert np.array_equal(g.state.cpu().numpy(), np.full(w, t * runs))
    g.close()


def layered(w, t, d, longest=False):
    """t steps of w tasks, each after d tasks of the step before it; longest: and an edge from the first to the last."""
    v = np.arange(w, w * t)
    p = (v // w - 1)[:, None] * w + ((v % w)[:, None] * 7 + np.arange(d)[None, :] * (w // d)) % w
    rows = np.stack([np.repeat(v, d), p.reshape(-1)], 1)
    return explicit(w * t, np.concatenate([rows, [[w * t - 1, 0]]]) if longest else rows)


def test_a_full_queue_is_shared_out_in_batches():
    """Steps of 1000 ready tasks of degree 8: the warps take batches, not a task each."""
    ensure_built()
    tr = layered(1000, 30, 8)
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=9)
    g.analyze()
    b = grt.Batch([g])
    for _ in range(2):
        g.out.zero_()
        b.execute(replays=2)
        b.sync()
        assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=9)[1])
        c = b.counters()
        assert c["tasks"] == 2 * tr.n and c["edges"] == 2 * g.stats()["n_edges"]
        assert 4 * c["claims"] < c["tasks"]
    b.close()
    g.close()
