"""Wide LCC at the edges of its row paths (empty rows, 1, 8, 31 to 33, 127 to
129, 1023 to 1025 and several thousand entries, at every offset within a bitmap
word), for each number of edge labels a kernel is built for, with multiplicity
classes met early, late and not at all.  Everything is integer and must equal
the oracle."""
import numpy as np
import pytest

from paper_1912_08453_gb300 import workloads as wl
from tests.test_gpu_wide import check

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 1023, 1024, 1025, 4000, 8161, 8192, 8193, 9400]


def stars(copies, seed):
    rng = np.random.default_rng(seed)
    lengths = LENGTHS * copies
    hubs, leaves = len(lengths), 9500
    edges = set()
    for h, d in enumerate(lengths):
        edges.update((h, hubs + int(v)) for v in rng.choice(leaves, d, replace=False))
    edges.update((hubs + int(a), hubs + int(b)) for a, b in rng.integers(0, leaves, (3000, 2)) if a < b)
    labels = rng.choice(5, hubs + leaves, p=[.3, .3, .3, .09, .01])
    labels[:hubs] = np.arange(hubs) % 3
    return wl.graph_from_edge_list(hubs + leaves, sorted(edges), labels)


# (labels, edges): nested needs on one label, a wheel, a path and a clique
TEMPLATES = [
    ([0, 1, 1, 1, 2, 2, 3], [(0, 1), (0, 2), (0, 3), (0, 4), (0, 5), (4, 6)]),
    ([0, 1, 2, 1, 2, 1, 2, 0, 0], [(0, i) for i in range(1, 7)] + [(1, 2), (3, 4), (1, 7), (3, 8)]),
    ([2] + [1] * 40, [(0, i) for i in range(1, 41)]),
    ([0, 1, 2, 4, 2, 1, 0, 1], [(i, i + 1) for i in range(7)]),
    ([0, 1], [(0, 1)]),
]


@pytest.fixture(scope="module")
def ctx():
    from paper_1912_08453_gb300 import ccpm
    return ccpm.Context(0)


@pytest.mark.parametrize("n_el", [1, 2, 3, 6])
@pytest.mark.parametrize("copies", [1, 5])
def test_row_paths(ctx, copies, n_el):
    g = stars(copies, copies)
    el = wl.edge_labels(g.row_ptr, g.col, n_el, seed=n_el, weights=[6] + [1] * (n_el - 1))
    for i, (tl, te) in enumerate(TEMPLATES):
        tel = [j % n_el if i % 2 == 0 or j % 3 == 0 else 0 for j in range(len(te))]
        check(ctx, g, tl, te, tel, el)
        check(ctx, g, tl, te)                    # no edge labels
    for seed in range(3):
        tl, te, tel = wl.sampled_template(g, el, 10 + 15 * seed, 6, seed=seed)
        check(ctx, g, tl, te, tel, el)
