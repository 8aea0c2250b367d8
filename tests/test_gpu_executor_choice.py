"""Which executor a graph runs on when its launch shape is left to the library,
as its statistics report it: 1 block of 128 or 512 threads (inside one block),
blocks of 32 threads (owned chunks) or more (the ring). The results are the
oracle's whichever it is."""
import numpy as np
import pytest

import oracle
from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import ensure_built, gpu_graph
from test_gpu_block_exec import explicit

pytestmark = pytest.mark.gpu


def shape_of(tr, iters, config=None):
    """(blocks, threads) of one execution, its results checked."""
    ensure_built()
    g = gpu_graph(tr, body=grt.RT_BODY_SPIN, spin_iters=iters)
    g.analyze()
    if config:
        g.exec_config(*config)
    g.execute()
    g.sync()
    st = g.stats()
    assert np.array_equal(g.out.cpu().numpy(), oracle.run_bodies(tr, oracle.oracle.BODY_SPIN, spin_iters=iters)[1])
    g.close()
    return st["exec_blocks"], st["exec_threads"]


def roots_then_chain(roots, n):
    """Tasks 0 .. roots - 1 without predecessors, then a chain: edges of one task, a front as wide as the roots."""
    v = np.arange(roots, n)
    return explicit(n, np.stack([v, v - 1], 1))


def test_many_roots_of_long_bodies_leave_the_block():
    """Short edges alone do not make a front narrow: the roots are ready together."""
    assert shape_of(explicit(701, np.zeros((0, 2))), 30000)[0] > 1
    assert shape_of(roots_then_chain(700, 1401), 20000)[0] > 1
    # of short bodies, or few, they stay: in a block of 16 warps, and of 4 only where those hold them
    assert shape_of(explicit(701, np.zeros((0, 2))), 8) == (1, 512)
    assert shape_of(roots_then_chain(200, 900), 8) == (1, 512)
    assert shape_of(roots_then_chain(70, 900), 8) == (1, 128)
    assert shape_of(explicit(60, np.zeros((0, 2))), 1000) == (1, 128)
