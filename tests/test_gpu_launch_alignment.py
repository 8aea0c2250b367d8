"""rt_launch_batch from device arrays at any byte address: what a kernel cannot
load from there is copied."""
import numpy as np
import pytest
import torch

from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, ensure_built, oracle_csr

pytestmark = pytest.mark.gpu


def at_offset(a, offset):
    """(device address `offset` bytes past a 256-byte boundary that holds the array, what keeps it alive)."""
    raw = np.frombuffer(np.ascontiguousarray(a).tobytes(), np.uint8)
    buf = torch.zeros(len(raw) + 512, dtype=torch.uint8, device="cuda")
    start = -buf.data_ptr() % 256 + offset
    buf[start:start + len(raw)] = torch.from_numpy(raw.copy()).cuda()
    return buf.data_ptr() + start, buf


@pytest.mark.parametrize("bounds", [np.int32, np.int64])
@pytest.mark.parametrize("offset", [0, 1, 2, 4, 8, 12])
def test_device_arrays_at_any_address(bounds, offset):
    ensure_built()
    tr = tg.random_rects(grid=(60, 50), n=700, rects=(1, 3), side=(1, 12), seed=9)
    held = [at_offset(a, offset) for a in (tr.req_off, tr.lo.astype(bounds), tr.hi.astype(bounds), tr.priv)]
    torch.cuda.synchronize()
    g = grt.Graph(2, tr.dom_lo, tr.dom_hi)
    launch = grt.rt_launch_batch32 if bounds is np.int32 else grt.rt_launch_batch
    launch(g.h, tr.n, *[h[0] for h in held], None, None, None, grt.RT_LAUNCH_DEVICE)
    g.analyze()
    assert_csr_equal(g, tr, oracle_csr(tr))
    g.close()
