"""A caller's bound on a batch's blocks holds where each graph runs inside one."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [(20,), (150,), (20, 150)], ids=["small", "large", "both"])
def test_blocks_in_flight_are_bounded(widths):
    """64 like graphs one or two at a time take many times what they take side by side."""
    ensure_built()
    traces = [tg.taskbench(widths[k % len(widths)], 40, "stencil") for k in range(64)]
    graphs = []
    for tr in traces:
        g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=5)
        g.analyze()
        graphs.append(g)
    b = grt.Batch(graphs)
    ms = {}
    for blocks in (0, 1, 2, 3, 304, 1):
        for g in graphs:
            g.out.zero_()
        b.execute(replays=4, blocks=blocks)
        b.sync()
        for _ in range(2):  # captured, relaunched
            b.execute(replays=4, blocks=blocks)
            ms[blocks] = b.sync()
        assert b.counters()["tasks"] == 4 * sum(t.n for t in traces)
        for tr, g in zip(traces, graphs):
            assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=5)[1])
    assert ms[1] > 8 * ms[0] and ms[1] > 8 * ms[304] and ms[2] > 4 * ms[0] and ms[3] > 3 * ms[0]
    b.close()
    for g in graphs:
        g.close()
