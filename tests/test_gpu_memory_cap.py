"""Analysis under a graph's memory cap (as the server sets one for each batch it
analyses): what is only there for speed gives way to it."""
import ctypes

import numpy as np
import pytest

from paper_2508_16522_gb300 import grt
from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, ensure_built, gpu_graph, oracle_csr

pytestmark = pytest.mark.gpu


def internals():
    """The two calls the server makes, by their C++ names."""
    lib = grt.load()
    size, cap = lib._ZN3grt15graph_footprintEP8rt_graph, lib._ZN3grt17graph_set_mem_capEP8rt_graphm
    size.argtypes, size.restype = [ctypes.c_void_p], ctypes.c_size_t
    cap.argtypes, cap.restype = [ctypes.c_void_p, ctypes.c_size_t], None
    return size, cap


def test_the_sweep_by_windows_gives_way_to_the_cap():
    """Writes of whole tiles, tens of thousands to a tile and no pair filter: the sweep by windows asks for twice the
    pair buffer, 16 bytes an entry more; with half of that missing the tiles are swept without it."""
    ensure_built()
    size, cap = internals()
    n = 70000
    tr = tg._finish(2, [0, 0], [31, 15], np.ones(n, np.int64), np.stack([16 * (np.arange(n) % 2), np.zeros(n)], 1)
                    .astype(np.int64).reshape(-1), np.stack([16 * (np.arange(n) % 2) + 15, np.full(n, 15)], 1)
                    .astype(np.int64).reshape(-1), np.ones(n, np.uint8))
    ref = oracle_csr(tr)
    g = gpu_graph(tr, tile=(16, 16))
    g.analyze()
    whole, st = size(g.h), g.stats()
    assert st["n_entries"] == n and st["pair_filter_bits"] == 0
    assert_csr_equal(g, tr, ref)
    g.close()
    g = gpu_graph(tr, tile=(16, 16))
    cap(g.h, whole - 8 * n)
    g.analyze()
    assert_csr_equal(g, tr, ref)
    assert size(g.h) <= whole - 8 * n
    g.close()
