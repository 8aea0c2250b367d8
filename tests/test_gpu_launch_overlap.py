"""rt_launch_batch of a large host batch while its stream is busy."""
import time

import numpy as np
import pytest
import torch

from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, ensure_built, oracle_csr

pytestmark = pytest.mark.gpu


def occupy(stream, seconds):
    """Queues about that much work."""
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with torch.cuda.stream(stream):
        a.record()
        torch.cuda._sleep(10_000_000)
        b.record()
        b.synchronize()
        torch.cuda._sleep(int(10_000_000 * seconds * 1e3 / a.elapsed_time(b)))


@pytest.mark.parametrize("bad", [False, True], ids=["valid", "invalid"])
def test_a_large_host_batch_does_not_wait_for_work_queued_before_it(bad):
    """0.3 s of work are queued; the call takes no longer than checking on the host and copying."""
    ensure_built()
    tr = tg.taskbench(512, 100, "random", seed=3, encode="explicit")
    assert tr.n + len(tr.pred) > 65536
    pred = np.array(tr.pred, np.int32)
    if bad:
        pred[-1] = tr.n
    arrays = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
              for a in (tr.req_off, tr.lo, tr.hi, tr.priv, tr.pred_off, pred)]
    stream = torch.cuda.Stream()
    g = grt.Graph(2, tr.dom_lo, tr.dom_hi, stream=stream)
    if not bad:
        g.launch(*arrays)  # everything loaded and allocated
        g.clear()
    torch.cuda.synchronize()
    occupy(stream, 0.3)
    t0 = time.perf_counter()
    if bad:
        with pytest.raises(grt.GrtError) as e:
            g.launch(*arrays)
        assert e.value.status == grt.RT_ERR_INVALID
    else:
        g.launch(*arrays)
    took = time.perf_counter() - t0
    assert not stream.query()  # the work queued before it still runs
    assert took < 0.1
    if not bad:
        g.analyze()
        assert_csr_equal(g, tr, oracle_csr(tr))
    g.close()
