"""Rows of the CSR by buckets that are sorted by one warp, in registers up to 256
candidate pairs and in shared memory past that: row lengths on both sides of
every step, with and without duplicate pairs; the CSR equals the oracle's."""
import numpy as np
import pytest

from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, gpu_graph

pytestmark = pytest.mark.gpu

LENGTHS = [31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024]


def test_explicit_rows():
    """Sources of every length in turn, their successors spread over later tasks."""
    rng = np.random.default_rng(3)
    k, n = len(LENGTHS), 3000
    preds = [set() for _ in range(n)]
    for v in range(3 * k):
        for c in rng.choice(np.arange(3 * k, n), LENGTHS[v % k], replace=False):
            preds[c].add(v)
    z = np.zeros(0, np.int64)
    tr = tg._finish(1, [0], [0], np.zeros(n, np.int64), z, z, np.zeros(0, np.uint8), pred_counts=[len(p) for p in preds],
                    pred=[x for p in preds for x in sorted(p)], name="rows")
    g = gpu_graph(tr)
    g.analyze()
    assert g.stats()["csr_by_buckets"] == 1
    assert_csr_equal(g, tr)
    g.close()


@pytest.mark.parametrize("readers,tiles", [(17, 2), (32, 2), (33, 2), (43, 3), (64, 2), (65, 2), (85, 3), (86, 3), (128, 2),
                                           (129, 2), (120, 5), (500, 2)])
def test_rows_with_duplicates(readers, tiles):
    """A writer of the whole domain, then readers of it: each pair once a tile."""
    n = 3 * (readers + 1)
    priv = np.where(np.arange(n) % (readers + 1) == 0, 1, 0)
    tr = tg._finish(1, [0], [64 * tiles - 1], np.ones(n, np.int64), np.zeros(n, np.int64), np.full(n, 64 * tiles - 1),
                    priv, name=f"readers{readers}_{tiles}")
    g = gpu_graph(tr, tile=(64, 1))
    g.analyze()
    assert_csr_equal(g, tr)
    g.close()
