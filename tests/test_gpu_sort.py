"""The entry sort at its block sizes: inputs of one-cell rectangles, one entry
each, on both sides of a block (3072 keys, 1024 in small sorts) and of the line
between the two, in two passes; the CSR equals the oracle's."""
import numpy as np
import pytest

from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, gpu_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 98303, 98304, 98305, 32 * 3072, 33 * 3072 - 1, 33 * 3072,
                               33 * 3072 + 1, 301059])
def test_entry_sort(n):
    rng = np.random.default_rng(n)
    at = rng.integers(0, 512, (n, 2))
    at[: n // 3] //= 16  # a third of them in one corner: long digit runs
    tr = tg._finish(2, [0, 0], [511, 511], np.ones(n, np.int64), at, at, rng.choice(3, n, p=(0.3, 0.5, 0.2)),
                    name=f"cells{n}")
    g = gpu_graph(tr, tile=(8, 8))
    g.analyze()
    assert g.stats()["n_entries"] == n
    assert_csr_equal(g, tr)
    g.close()
