"""Searches that are spread up front (no handing on, or a caller's own budget): a
level whose items do not fit the item list (2^22 for a small graph) leaves the
search at the level before, and it runs from there.

The graph: a hub with leaves of one label and a few edges among them, so that the
second of two equal leaves gives leaves * (leaves - 1) items."""
import numpy as np
import pytest

from oracle import pipeline
from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def hub(leaves):
    rng = np.random.default_rng(leaves)
    edges = {(0, v) for v in range(1, leaves + 1)}
    edges |= {(int(a), int(b)) for a, b in np.sort(rng.integers(1, leaves + 1, (300, 2)), axis=1) if a < b}
    return wl.graph_from_edge_list(leaves + 1, sorted(edges), [1] + [0] * leaves)


# the counting search: 2040 * 2039 items fit, 2060 * 2059 do not
@pytest.mark.parametrize("leaves", [2040, 2060])
@pytest.mark.parametrize("tl,te", [([1, 0, 0, 0], [(0, 1), (0, 2), (0, 3)]),
                                   ([1, 0, 0, 0, 0], [(0, 1), (0, 2), (0, 3), (0, 4), (1, 2)])])
def test_expansion_that_does_not_fit(leaves, tl, te):
    from paper_1912_08453_gb300 import ccpm
    g = hub(leaves)
    ref = pipeline.run(g.row_ptr, g.col, g.labels, tl, te, max_embeddings=1000)
    assert not ref.count_valid
    ctx = ccpm.Context(0)
    dev, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, tl, te)
    for opts in ({"search_split": -1}, {"search_budget": 1 << 22}, {"search_split": -1, "search_budget": 1 << 22}):
        r = ccpm.prune(ctx, dev, t, ccpm.options(max_embeddings=1000, **opts), allow_budget=True)
        np.testing.assert_array_equal(r.omega(), ref.omega)
        np.testing.assert_array_equal(r.edge_bitmap(), ref.ebits)
        assert not r.counts()["count_valid"] and r.phase_rounds() == ref.phase_rounds
        r.close()
    for x in (t, dev, ctx):
        x.close()
