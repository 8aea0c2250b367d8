"""The sweep by windows (dense inputs), and the tile sweep without classes
(rectangles of a few cells): the CSR equals the oracle's where they can go
wrong -- tile shapes on both sides of 32 columns and rows, 1-D
tiles, windows cut inside a task of many rectangles, tasks of more candidates
than a window takes, runs of readers longer than a walk, thinly covered domain
borders, and more distinct pairs than the buffer's first guess."""
import numpy as np
import pytest

from paper_2508_16522_gb300 import tracegen as tg

from gpu_helpers import assert_csr_equal, gpu_graph, oracle_csr

pytestmark = pytest.mark.gpu


def _boxes(ndim, ext, counts, boxes, priv, name):
    b = np.asarray(boxes, np.int64).reshape(-1, 2, ndim)
    return tg._finish(ndim, [0] * ndim, [e - 1 for e in ext], counts, b[:, 0].reshape(-1), b[:, 1].reshape(-1),
                      np.asarray(priv, np.uint8), name=name)


def dense(grid, n, side, seed, rects=(1, 4), probs=(0.6, 0.3, 0.1)):
    return tg.random_rects(grid=grid, n=n, rects=rects, side=side, seed=seed, probs=probs, ndim=len(grid))


def many_rects(seed):
    """Tasks of up to 40 overlapping rectangles on a small domain: tasks that a
    window cuts, and tasks of more candidates in a tile than one takes."""
    rng = np.random.default_rng(seed)
    counts = rng.choice([1, 2, 3, 9, 17, 40], size=300)
    boxes, priv = [], []
    for _ in range(int(counts.sum())):
        x, y = rng.integers(0, 40, 2)
        w, h = rng.integers(6, 24, 2)
        boxes.append([[x, y], [min(x + w, 47), min(y + h, 47)]])
        priv.append(rng.choice(3, p=(0.6, 0.3, 0.1)))
    return _boxes(2, (48, 48), counts, boxes, priv, f"many_rects{seed}")


def long_runs(readers, seed):
    """Readers, then reducers, then writers of the whole domain, with small boxes
    between: runs of several blocks of 32 candidates."""
    rng = np.random.default_rng(seed)
    boxes, priv = [], []
    for kind, m in ((0, readers), (2, readers // 2), (1, 3), (0, 40), (2, 5), (0, readers)):
        for _ in range(m):
            boxes.append([[0, 0], [23, 23]])
            priv.append(kind)
            if rng.random() < 0.2:
                x, y = rng.integers(0, 20, 2)
                boxes.append([[x, y], [x + 3, y + 3]])
                priv.append(rng.integers(0, 3))
    return _boxes(2, (24, 24), np.ones(len(priv), np.int64), boxes, priv, f"runs{readers}")


def few_large(seed):
    """Boxes of one or two cells, one in a thousand the whole domain: the tile
    sweep that keeps every cell its own class."""
    rng = np.random.default_rng(seed)
    boxes, priv = [], []
    for k in range(4000):
        x, y = rng.integers(0, 45, 2)
        boxes.append([[0, 0], [47, 39]] if k % 1000 == 7 else [[x, min(y, 39)], [min(x + rng.integers(0, 2), 47), min(y, 39)]])
        priv.append(rng.choice(3, p=(0.6, 0.3, 0.1)))
    counts = rng.integers(1, 4, 4000)
    counts = counts[:int(np.searchsorted(np.cumsum(counts), 4000))]
    counts = np.append(counts, 4000 - counts.sum())
    return _boxes(2, (48, 40), counts, boxes, priv, f"few_large{seed}")


CASES = [
    ("few_large", lambda: few_large(6), [(16, 16), (8, 8), (32, 4), (48, 20), (7, 9)]),
    ("tiles", lambda: dense((200, 168), 700, (4, 90), 3), [(16, 16), (16, 32), (32, 32), (32, 4), (33, 31), (64, 64), (128, 16)]),
    ("thin", lambda: dense((256, 256), 1500, (20, 120), 5, probs=(0.9, 0.02, 0.08)), [(16, 16), (32, 32), (64, 32)]),
    ("ragged", lambda: dense((97, 1), 400, (1, 60), 7), [(16, 16), (32, 1), (97, 1)]),
    ("one_dim", lambda: dense((4001,), 1800, (60, 900), 9), [(16, 1), (100, 1), (1024, 1), (1000, 1)]),
    ("stencil_1d", lambda: tg.stencil_1d(7, 90, 512), [(0, 0), (512, 1), (100, 1)]),
    ("many_rects", lambda: many_rects(1), [(8, 8), (16, 16), (48, 48)]),
    ("runs", lambda: long_runs(60, 2), [(8, 8), (16, 32)]),
    ("long_runs", lambda: long_runs(550, 4), [(16, 16)]),
    ("one_task", lambda: dense((64, 64), 1, (20, 60), 1), [(8, 8)]),
]


@pytest.mark.parametrize("name,make,tiles", CASES, ids=[c[0] for c in CASES])
def test_csr_by_windows_equals_the_oracle(name, make, tiles):
    tr = make()
    ref = oracle_csr(tr)
    for tile in tiles:
        g = gpu_graph(tr, tile=tile)
        g.analyze()
        assert_csr_equal(g, tr, ref)
        g.close()
