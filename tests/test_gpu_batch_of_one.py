"""A batch of a single graph, on every executor a batch has."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [grt.RT_EXEC_RING, grt.RT_EXEC_OWNED])
@pytest.mark.parametrize("tr", [tg.random_rects(grid=(30, 30), n=300, side=(1, 9), seed=2),
                                tg.random_rects(grid=(900, 900), n=6000, side=(1, 9), seed=3)],
                         ids=["few_roots", "many_roots"])
def test_batch_of_one_graph(tr, policy):
    """CHECK bodies (never inside one block) and SPIN bodies of a graph of few and of thousands of roots."""
    ensure_built()
    for body in (grt.RT_BODY_CHECK, grt.RT_BODY_SPIN):
        g = gpu_graph(tr, body=body, spin_iters=9)
        g.analyze()
        b = grt.Batch([g])
        b.exec_policy(policy)
        want_state, want_out = oracle.run_bodies(tr, body, spin_iters=9)
        b.execute(replays=1)
        b.sync()
        assert b.counters()["tasks"] == tr.n
        if body == grt.RT_BODY_CHECK:
            assert np.array_equal(g.state.cpu().numpy(), want_state)
        assert np.array_equal(g.out.cpu().numpy(), want_out)
        for _ in range(2):  # the ring as the launch before left it, from a captured launch
            b.execute(replays=3)
            b.sync()
            assert b.counters()["tasks"] == 3 * tr.n
        b.close()
        g.close()
