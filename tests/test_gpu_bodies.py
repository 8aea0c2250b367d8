"""The SPIN and FMA bodies at iteration counts on both sides of their loops'
turns (32 steps, 8 steps, single ones), in the executors that inline them."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph

pytestmark = pytest.mark.gpu

TRACE = tg.taskbench(40, 9, "stencil")
COUNTS = (0, 1, 7, 8, 9, 24, 31, 32, 33, 40, 63, 64, 65, 127, 300)


@pytest.mark.parametrize("body", [grt.RT_BODY_SPIN, grt.RT_BODY_FMA])
@pytest.mark.parametrize("config", [(0, 0, 0, 0), (8, 2, 0, 0)], ids=["default", "ring"])
def test_iteration_counts(body, config):
    ensure_built()
    for iters in COUNTS:
        g = gpu_graph(TRACE, body=body, spin_iters=iters)
        g.analyze()
        g.exec_config(*config)
        g.execute()
        g.sync()
        want = oracle.run_bodies(TRACE, body, spin_iters=iters)[1]
        assert np.array_equal(g.out.cpu().numpy(), want), iters
        g.exec_policy(grt.RT_EXEC_OWNED)
        g.out.zero_()
        g.execute()
        g.sync()
        assert np.array_equal(g.out.cpu().numpy(), want), iters
        g.close()


def test_no_executor_runs_a_body_quicker_than_it_runs_alone():
    """The rate that efficiencies are measured against is the body's best: a chain of long bodies takes at least that."""
    ensure_built()
    alone = grt.rt_microbench_atomics()["fma_body_ns_per_iter"]
    iters, tr = 60000, tg.taskbench(1, 40, "stencil")
    for config in ((8, 2, 1, 4), (0, 0, 0, 0)):
        g = gpu_graph(tr, body=grt.RT_BODY_FMA, spin_iters=iters, flags=grt.RT_GRAPH_PROFILE)
        g.analyze()
        g.exec_config(*config)
        for _ in range(3):
            g.execute()
            g.sync()
            assert g.stats()["ms_exec_kernel"] * 1e6 > 0.98 * alone * iters * tr.n
        g.close()
