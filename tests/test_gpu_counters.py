"""The counters a caller divides by: LCC rounds that ran, and only those.  Rounds
are queued before it is known whether they are needed (behind a check that may
change nothing, past the fixpoint); what returns at once is no round."""
import pytest

from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# a triangle, a 4-cycle with a chord, two triangles that share a vertex
TEMPLATES = [
    ([0, 1, 2], [(0, 1), (1, 2), (0, 2)]),
    ([0, 1, 2, 1], [(0, 1), (1, 2), (2, 3), (3, 0), (0, 2)]),
    ([0, 1, 2, 1, 2], [(0, 1), (1, 2), (0, 2), (0, 3), (3, 4), (0, 4)]),
]


def disjoint_triangles(k):
    """Every vertex lies in a triangle: the cycle checks eliminate nothing."""
    edges = [(3 * i + a, 3 * i + b) for i in range(k) for a, b in ((0, 1), (1, 2), (0, 2))]
    return wl.graph_from_edge_list(3 * k, edges, [0, 1, 2] * k)


# a million triangles: rows of more than 2^22 entries, the rounds evaluate changes only
@pytest.mark.parametrize("graph", ["triangles", "many triangles", "rmat"])
@pytest.mark.parametrize("split", [0, 1])
def test_launches_are_the_rounds_that_ran(graph, split):
    from paper_1912_08453_gb300 import ccpm
    if graph == "rmat":
        g = wl.rmat_graph(12, seed=4, labels="zipf", n_labels=3)
    elif graph == "triangles":
        g = disjoint_triangles(50)
    else:
        import numpy as np
        k = 1 << 20
        v = np.arange(3 * k, dtype=np.int64)
        other = np.sort(np.stack([v // 3 * 3 + (v + 1) % 3, v // 3 * 3 + (v + 2) % 3], 1), axis=1)
        g = wl.Graph(3 * k, 2 * np.arange(3 * k + 1, dtype=np.int64), other.reshape(-1).astype(np.int32),
                     (v % 3).astype(np.uint8))
    ctx = ccpm.Context(0)
    dev = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels)
    unchanged = 0
    for tl, te in TEMPLATES:
        t = ccpm.Template(ctx, tl, te)
        r = ccpm.prune(ctx, dev, t, ccpm.options(search_split=split, run_final=0))
        rounds = r.phase_rounds()
        assert r.counts()["lcc_launches"] == sum(rounds), rounds
        unchanged += rounds[1:].count(0)
        r.close()
        t.close()
    if graph != "rmat":
        assert unchanged > 0                      # a check that changed nothing was among them
    dev.close()
    ctx.close()
