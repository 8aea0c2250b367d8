"""Owned chunks that the library picks, on a device that others hold: their warps
start together or not yet, so neither a resident server nor kernels that leave
them a few places make a run give up."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph
from test_gpu_block_exec import explicit

pytestmark = pytest.mark.gpu

WIDE = tg.taskbench(1024, 70, "stencil")
TRACE = tg.taskbench(600, 10, "stencil")


def crowd(sms, seconds):
    """A batch whose blocks (two fill an SM's registers) take all places but one for about that long, launched on a
    stream of its own: (batch, its graph)."""
    stream = torch.cuda.Stream()
    v = np.arange(1, 200)  # a chain of long bodies, with edges of 100 tasks: a block of 16 warps
    tr = explicit(200, np.concatenate([np.stack([v, v - 1], 1), np.stack([v[99:], v[99:] - 100], 1)]))
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=1200, stream=stream)
    g.analyze()
    b = grt.Batch([g] * (2 * sms - 1), stream=stream)
    b.execute(replays=20, blocks=2 * sms - 1)
    ms = b.sync()
    b.execute(replays=min(4096, int(20 * seconds * 1e3 / ms)), blocks=2 * sms - 1)
    return b, g


@pytest.mark.parametrize("what", ["execute", "replay", "stitch"])
def test_runs_on_a_few_places(what):
    """The limit is a tenth of the time for which others hold the rest of the device."""
    ensure_built()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    stream = torch.cuda.Stream()
    tr = tg.concat([TRACE, TRACE]) if what == "stitch" else WIDE
    R = {"execute": 1, "replay": 3, "stitch": 60}[what]
    out = torch.zeros(TRACE.n * R if what == "stitch" else WIDE.n, dtype=torch.int32, device="cuda")
    g = grt.Graph(2, tr.dom_lo, tr.dom_hi, body=grt.RT_BODY_SPIN, spin_iters=8, out=out, stream=stream,
                  timeout_ns=50_000_000)
    g.launch_trace(tr)
    g.analyze()
    run = {"execute": lambda: g.execute(), "replay": lambda: g.replay(3), "stitch": lambda: g.execute_stitched(R)}[what]
    run()  # everything loaded and allocated
    g.sync()
    out.zero_()
    torch.cuda.synchronize()
    b, bg = crowd(sms, 0.5)
    time.sleep(0.02)  # the crowd has started
    run()
    g.sync()
    assert b.sync() > 300  # the others held their places for all that time
    one = oracle.run_bodies(TRACE if what == "stitch" else WIDE, oracle.oracle.BODY_SPIN, spin_iters=8)[1]
    assert np.array_equal(out.cpu().numpy(), np.tile(one, R) if what == "stitch" else one)
    for x in (b, bg, g):
        x.close()


def test_runs_beside_a_resident_server():
    """Everything is created, loaded and run once before the server starts, and closed after it has stopped."""
    ensure_built()
    cases = []
    for tr in (WIDE, tg.taskbench(100, 90, "stencil"), tg.taskbench(3000, 20, "stencil")):
        g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=8, stream=torch.cuda.Stream())
        g.analyze()
        cases.append((g, oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=8)[1]))
    batch = grt.Batch([g for g, _ in cases], stream=torch.cuda.Stream())
    R = 40
    out = torch.zeros(R * TRACE.n, dtype=torch.int32, device="cuda")
    two = grt.Graph(2, TRACE.dom_lo, TRACE.dom_hi, body=grt.RT_BODY_SPIN, spin_iters=8, out=out,
                    stream=torch.cuda.Stream())
    two.launch_trace(tg.concat([TRACE, TRACE]))
    two.analyze()
    one = oracle.run_bodies(TRACE, oracle.oracle.BODY_SPIN, spin_iters=8)[1]

    def everything():
        for g, _ in cases:
            g.out.zero_()
        out.zero_()
        torch.cuda.current_stream().synchronize()
        for g, _ in cases:
            g.execute()
        for g, want in cases:
            g.sync()
            assert np.array_equal(g.out.cpu().numpy(), want)
            g.out.zero_()
        torch.cuda.current_stream().synchronize()
        two.execute_stitched(R)
        assert np.array_equal(out.cpu().numpy(), np.tile(one, R))
        batch.execute(replays=3)
        batch.sync()
        for g, want in cases:
            assert np.array_equal(g.out.cpu().numpy(), want)

    everything()
    everything()  # the batch's launch captured
    requests = [tg.random_rects(grid=(256, 256), n=300 + 40 * k, side=(1, 40), seed=k) for k in range(8)]
    srv = grt.Server(2, [0, 0], [255, 255], body=grt.RT_BODY_SPIN, spin_iters=4, max_inflight=16, max_tasks=4096,
                     workers=2, keep_results=True, budget_bytes=1 << 30)
    for _ in range(5):
        tickets = [srv.submit(t) for t in requests]
        everything()
    srv.drain(120_000_000_000)
    assert all(srv.poll(t)["status"] == grt.RT_OK for t in tickets)
    srv.close()
    batch.close()
    for x in (two, *(g for g, _ in cases)):
        x.close()
