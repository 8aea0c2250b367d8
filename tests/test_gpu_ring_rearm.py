"""Counters re-armed by the tasks themselves: runs on the ring and over owned
chunks of one graph, one after another in any order, each find them at the
in-degrees."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tr", [tg.taskbench(700, 20, "random", seed=2), tg.random_rects(grid=(60, 60), n=900, side=(2, 20), seed=4)],
                         ids=["random", "rects"])
def test_runs_in_any_order(tr):
    ensure_built()
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=3)
    g.analyze()
    want = oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=3)[1]
    rng = np.random.default_rng(1)
    for k in range(60):
        policy, shape, replays = [(grt.RT_EXEC_RING, (152, 4, 4, 8), 1), (grt.RT_EXEC_RING, (152, 2, 8, 16), 1),
                                  (grt.RT_EXEC_RING, (40, 8, 1, 2), 3), (grt.RT_EXEC_OWNED, (32, 1, 1, 0), 1),
                                  (grt.RT_EXEC_OWNED, (64, 1, 4, 0), 2), (grt.RT_EXEC_RING, (0, 0, 0, 0), 1)][rng.integers(6)]
        g.exec_policy(policy)
        g.exec_config(*shape)
        g.out.zero_()
        g.replay(replays) if replays > 1 else g.execute()
        g.sync()
        assert np.array_equal(g.out.cpu().numpy(), want), k
    g.close()
