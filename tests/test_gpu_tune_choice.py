"""The tuners' answers include what the library does untuned."""
import time

import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


def run_ms(g):
    """The quickest of 20 runs, host time."""
    best = 1e9
    for _ in range(20):
        t0 = time.perf_counter()
        g.execute()
        g.sync()
        best = min(best, (time.perf_counter() - t0) * 1e3)
    return best


@pytest.mark.parametrize("width,steps,untuned", [(32, 400, (1, 128)), (256, 200, (1, 512)), (5000, 40, (256, 32))])
def test_a_tuned_graph_is_no_slower_than_an_untuned_one(tmp_path, width, steps, untuned):
    ensure_built()
    cache = tmp_path / "tune.txt"
    tr = tg.taskbench(width, steps, "stencil")
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=8)
    g.analyze()
    before = run_ms(g)
    st = g.stats()
    assert (st["exec_blocks"], st["exec_threads"]) == untuned
    c = g.tune(cache)
    assert run_ms(g) < 1.3 * before
    st = g.stats()
    if untuned[0] == 1:
        assert c["blocks"] == 1 and (st["exec_blocks"], st["exec_threads"]) == untuned
    g.out.zero_()
    g.execute()
    g.sync()
    want = oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=8)[1]
    assert np.array_equal(g.out.cpu().numpy(), want)
    g.exec_config()
    again = g.tune(cache)  # answered from the cache
    assert again["trials"] == 0 and all(again[k] == c[k] for k in ("blocks", "warps", "claim", "keep", "policy"))
    g.out.zero_()
    g.replay(3)
    g.sync()
    assert g.stats()["exec_blocks"] == st["exec_blocks"]
    assert np.array_equal(g.out.cpu().numpy(), want)
    g.close()


def test_one_block_of_eight_warps_runs_what_does_not_fit_on_the_ring():
    """The shape lets a graph run inside one block; one that does not fit keeps the ring in that shape."""
    ensure_built()
    for tr, iters, threads in ((tg.taskbench(300, 20, "stencil"), 8, 512), (tg.taskbench(2000, 5, "stencil"), 8, 256),
                               (tg.taskbench(1, 50, "stencil"), 8, 128)):
        g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=iters)
        g.analyze()
        g.exec_config(1, 8, 4, 8)
        g.execute()
        g.sync()
        st = g.stats()
        assert (st["exec_blocks"], st["exec_threads"]) == (1, threads)
        assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=iters)[1])
        g.close()


def test_a_batch_in_blocks_is_tuned_without_a_grid(tmp_path):
    """No bound on the blocks, and the time reported is that of the launch as it runs."""
    ensure_built()
    cache = tmp_path / "tune.txt"
    traces = [tg.taskbench(40 + 13 * k, 60, tg.PATTERNS[k % 3] if k % 3 != 1 else "stencil", seed=k) for k in range(24)]
    graphs = [gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=7) for tr in traces]
    for g in graphs:
        g.analyze()
    b = grt.Batch(graphs)
    b.execute(replays=4)
    b.sync()
    c = b.tune(replays=4, cache_path=cache)
    assert c["trials"] >= 10
    if c["policy"] == grt.RT_EXEC_RING:
        assert (c["blocks"], c["warps"]) == (0, 0)
    assert cache.read_text().startswith("batch3/")
    best = 1e9
    for _ in range(5):
        b.execute(replays=4, blocks=c["blocks"], warps=c["warps"], claim=c["claim"], keep=c["keep"])
        best = min(best, b.sync())
    assert best < 1.3 * c["ms"]
    for tr, g in zip(traces, graphs):
        assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=7)[1])
    assert b.tune(replays=4, cache_path=cache)["trials"] == 0
    b.close()
    for g in graphs:
        g.close()


def test_the_caches_entries_are_of_the_current_kernels(tmp_path):
    """An entry of an older sweep or executor does not answer: its tile or shape was the best of other kernels."""
    ensure_built()
    cache = tmp_path / "tune.txt"
    tr = tg.random_rects(grid=(200, 200), n=900, rects=(1, 3), side=(1, 30), seed=5)
    grt.rt_tune_tile(tr, cache)
    key = cache.read_text().split(" ")[0]
    assert key.startswith("tile4/")
    for old in ("tile", "tile2", "tile3"):
        cache.write_text(f"{old}/{key.split('/', 1)[1]} 8 8 0.001\n")
        assert grt.rt_tune_tile(tr, cache)[2] > 0.001


def test_a_tuned_graph_takes_larger_launches():
    """Tuned for launches that run inside one block, then cleared and given ones that do not."""
    ensure_built()
    small, large = tg.taskbench(32, 100, "stencil"), tg.taskbench(1024, 100, "stencil")
    g = grt.Graph(2, large.dom_lo, large.dom_hi)
    for tr in (small, large):
        g.clear()
        g.launch_trace(tr)
        g.analyze()
        if tr is small:
            assert g.tune()["blocks"] == 1
        g.execute()
        g.sync()
        st = g.stats()
        assert (st["exec_blocks"] == 1) == (tr is small) and st["exec_counters"]["tasks"] == tr.n
    g.close()
