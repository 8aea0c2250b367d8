"""Which sweep an analysis took, as its statistics report it, at tile shapes and
inputs for each form of the sweep by windows; the CSR equals the oracle's."""
import numpy as np
import pytest

from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, gpu_graph, oracle_csr
from test_gpu_windows import _boxes, dense

pytestmark = pytest.mark.gpu


def many_large_rects(seed):
    """Tasks of up to 40 overlapping rectangles, each a good part of a 48 x 48 domain."""
    rng = np.random.default_rng(seed)
    counts = rng.choice([1, 2, 3, 9, 15, 40], size=300)
    boxes, priv = [], []
    for _ in range(int(counts.sum())):
        x, y = rng.integers(0, 14, 2)
        w, h = rng.integers(20, 34, 2)
        boxes.append([[x, y], [min(x + w, 47), min(y + h, 47)]])
        priv.append(rng.choice(3, p=(0.6, 0.3, 0.1)))
    return _boxes(2, (48, 48), counts, boxes, priv, f"many_large{seed}")


def runs_of(readers):
    """Readers and reducers of the whole domain in turn, `readers` of each: that many squared pairs a change."""
    priv = np.repeat([0, 2, 0, 2, 0, 2], readers)
    return _boxes(2, (8, 8), np.ones(len(priv), np.int64), [[[0, 0], [7, 7]]] * len(priv), priv, f"runs{readers}")


# (input, tile, what the windows left, whether the pair filter was in use). Boxes with many edges in a wide tile make
# more class cells of a window than it takes, so some of those are left
CASES = [
    ("small_tiles", lambda: dense((200, 168), 700, (4, 90), 3), (16, 16), "none", True),
    ("wide_tiles", lambda: dense((512, 512), 500, (150, 400), 4), (64, 64), "any", True),
    ("flat_tiles", lambda: dense((512, 512), 500, (150, 400), 5), (128, 16), "any", True),
    ("tall_tiles", lambda: dense((512, 512), 500, (150, 400), 6), (16, 128), "any", True),
    ("ragged_tiles", lambda: dense((517, 300), 500, (100, 250), 7), (33, 31), "any", True),
    ("one_row", lambda: dense((997, 1), 800, (300, 900), 8), (32, 1), "none", True),
    ("one_dim", lambda: dense((4001,), 1800, (60, 900), 9), (100, 1), "any", False),
    ("one_tile", lambda: dense((48, 48), 3000, (20, 40), 10, rects=(1, 2)), (48, 48), "some", False),
    ("large_tasks", lambda: many_large_rects(1), (48, 48), "some", False),
    ("small_boxes", lambda: dense((200, 168), 700, (1, 3), 11), (16, 16), "not run", False),
    ("overflow_filtered", lambda: runs_of(300), (2, 2), "overflow", True),
    ("overflow", lambda: runs_of(300), (8, 8), "overflow", False),
]


@pytest.mark.parametrize("name,make,tile,path,filtered", CASES, ids=[c[0] for c in CASES])
def test_the_sweep_taken(name, make, tile, path, filtered):
    tr = make()
    g = gpu_graph(tr, tile=tile)
    g.analyze()
    st = g.stats()
    assert_csr_equal(g, tr, oracle_csr(tr))
    assert (st["pair_filter_bits"] > 0) == filtered
    left = st["windows_left"]
    assert {"none": left == 0, "some": left > 0, "any": left >= 0, "not run": left == -1, "overflow": left == -2}[path], left
    g.close()
