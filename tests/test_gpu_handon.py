"""Searches over long label groups: the stretches a search hands to other
warps (edges of 32-candidate windows and of the 32 parts a group is cut into)
and the sampled join cache (edges of its 128 ids), against the oracle.

The graph: two hubs of label 0 and one of label 2, joined to one another and
to `common` vertices of label 1; some of these also carry edges among
themselves, so triangles and 4-cycles end in long groups that are scanned as
well as looked up.  All results are integers and must be equal."""
import numpy as np
import pytest

from oracle import pipeline
from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TEMPLATES = [
    ([0, 1, 2], [(0, 1), (1, 2), (0, 2)]),
    ([0, 1, 0, 1], [(0, 1), (1, 2), (2, 3), (3, 0)]),
    ([0, 1, 1, 2], [(0, 1), (1, 2), (0, 2), (2, 3), (1, 3)]),
]


def hub_graph(common, seed):
    rng = np.random.default_rng(seed)
    edges = {(0, 1), (0, 2), (1, 2)}
    for v in range(3, 3 + common):
        edges.update((h, v) for h in range(3) if rng.random() < 0.9)
    for _ in range(common // 8):
        a, b = (int(x) for x in rng.integers(3, 3 + common, 2))
        if a != b:
            edges.add((min(a, b), max(a, b)))
    labels = [0, 0, 2] + [1] * common
    return wl.graph_from_edge_list(3 + common, sorted(edges), labels)


@pytest.mark.parametrize("common", [31, 33, 127, 129, 1025, 4200])
def test_long_groups_equal_the_oracle(common):
    from paper_1912_08453_gb300 import ccpm
    g = hub_graph(common, common)
    ctx = ccpm.Context(0)
    graph = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels)
    for tl, te in TEMPLATES:
        if len(tl) == 4 and tl[1] == tl[3] and common > 2000:
            continue                                  # 10^7 4-cycles: slow on the oracle's side
        ref = pipeline.run(g.row_ptr, g.col, g.labels, tl, te)
        t = ccpm.Template(ctx, tl, te)
        for split in (0, 1, 5) + ((-1,) if common < 1000 else ()):   # -1: whole searches, expanded up front
            for cap in (1 << 32, 100):                # past the cap: the existence searches
                r = ccpm.prune(ctx, graph, t, ccpm.options(search_split=split, max_embeddings=cap),
                               allow_budget=True)
                np.testing.assert_array_equal(r.omega(), ref.omega)
                np.testing.assert_array_equal(r.edge_bitmap(), ref.ebits)
                c = r.counts()
                assert c["count_valid"] == int(ref.match_embeddings <= cap)
                if c["count_valid"]:
                    assert c["match_embeddings"] == ref.match_embeddings
                n, lst, vc, ec = r.matches(t, list_cap=64, vertex_counts=True, entry_counts=True,
                                           opts=ccpm.options(search_split=split))
                assert n == ref.match_embeddings
                assert int(vc.sum()) == n * len(tl) and int(ec.sum()) == 2 * n * len(te)
                assert len({tuple(x) for x in lst.tolist()}) == min(n, 64)
                r.close()
        t.close()
    graph.close()
    ctx.close()
