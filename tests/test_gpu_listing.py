"""Match listings on both kinds of rows: rows copied from the result (the first
listing of a graph, and large results of templates over hubs) and the graph's own
label-grouped rows.  Matches, and participation counts, equal the oracle's."""
import numpy as np
import pytest

import oracle
from oracle import pipeline
from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # degree labels: hubs, with few and with many entries in the result
    (15, [5, 12, 11, 11, 5, 7], [(0, 1), (1, 2), (2, 3), (3, 0), (2, 4), (3, 4), (4, 5)]),
    (15, [11, 10, 12], [(0, 1), (1, 2), (0, 2)]),
    (15, [5, 11, 4, 12], [(0, 1), (1, 2), (2, 3)]),
    (14, [5, 4, 8, 7, 4, 5], [(0, 1), (1, 2), (1, 3), (3, 4), (3, 5), (2, 3)]),
    (13, [11, 3, 6, 8, 7, 9], [(0, 1), (1, 2), (1, 3), (3, 4), (4, 5)]),
]


def ordered(maps):
    """A 64-bit key of every distinct row, in order."""
    odd = np.random.default_rng(1).integers(1, 1 << 62, maps.shape[1]).astype(np.uint64) * np.uint64(2) + np.uint64(1)
    return np.unique((maps.astype(np.uint64) * odd).sum(axis=1, dtype=np.uint64))


@pytest.mark.parametrize("scale,tl,te", CASES)
def test_both_kinds_of_rows(scale, tl, te):
    from paper_1912_08453_gb300 import ccpm
    g = wl.rmat_graph(scale, seed=6)
    ref = pipeline.run(g.row_ptr, g.col, g.labels, tl, te, max_embeddings=1 << 24)
    og = oracle.Graph(g.row_ptr, g.col, g.labels)
    count, lst, vc, ec = oracle.matches(og, tl, te, ref.omega, ref.A, list_cap=1 << 22)
    want = ordered(lst)
    assert 0 < count == ref.match_embeddings == len(want)
    ctx = ccpm.Context(0)
    dev, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, tl, te)
    exact = ccpm.prune(ctx, dev, t)
    states = [exact, ccpm.prune(ctx, dev, t, ccpm.options(lcc_only=1)),
              ccpm.prune(ctx, dev, t, ccpm.options(max_embeddings=1), allow_budget=True)]
    for r in states:
        for opts in ({}, {}, {"search_split": -1}, {"hub_degree": 16}):     # the first one copies
            n, got, v, e = r.matches(t, list_cap=count + 5, vertex_counts=True, entry_counts=True,
                                     opts=ccpm.options(**opts))
            assert n == count
            np.testing.assert_array_equal(ordered(got), want)
            np.testing.assert_array_equal(v, vc)
            np.testing.assert_array_equal(e, ec)
            n, got, _, _ = r.matches(t, list_cap=7, device=True)
            assert n == count
            assert len(ordered(np.concatenate([lst, got.cpu().numpy()]))) == count      # all of them listed above
    for x in (*states, t, dev, ctx):
        x.close()


def test_sizes_on_both_sides_of_the_rule():
    """What the cases above rely on: results below and above 2^14 entries."""
    from paper_1912_08453_gb300 import ccpm
    ctx = ccpm.Context(0)
    entries = []
    for scale, tl, te in CASES:
        g = wl.rmat_graph(scale, seed=6)
        dev, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, tl, te)
        r = ccpm.prune(ctx, dev, t)
        entries.append(r.counts()["active_e_dir"])
        for x in (r, t, dev):
            x.close()
    ctx.close()
    assert min(entries) < 1 << 14 and sum(e >= 1 << 14 for e in entries) >= 2, entries
