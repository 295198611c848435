"""LCC rounds on frontiers of every size class: rows of 1, 16, 17, 32, 64, 65,
1024 and 1025 entries (edges of the row paths), from a few rows to more than
one per resident warp, and templates whose label-multiplicity classes coincide
(one counted mask serves several template vertices).  Everything is integer
and must equal the oracle: omega, the edge bitmap, rounds, scanned entries."""
import numpy as np
import pytest

import oracle
from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CLIQUE5 = [(a, b) for a in range(5) for b in range(a + 1, 5)]
TEMPLATES = [
    ([0, 1], [(0, 1)]),
    ([0, 1, 1], [(0, 1), (0, 2)]),
    ([0, 1, 0, 1, 2], CLIQUE5),                                            # six pairs, two masks
    ([0, 1, 1, 1, 2, 2, 0], [(0, 1), (0, 2), (0, 3), (0, 4), (0, 5), (4, 6)]),
    ([0, 0, 1, 1, 2, 2, 3, 3, 4, 4, 5], [(a, 10) for a in range(10)] + [(0, 2), (1, 3), (4, 6)]),   # five masks
]


def stars(copies, seed):
    """Hubs of the listed row lengths over shared leaves, labels at random."""
    rng = np.random.default_rng(seed)
    lengths = [1, 16, 17, 32, 64, 65, 1024, 1025] * copies
    hubs, leaves = len(lengths), 3000
    edges = set()
    for h, d in enumerate(lengths):
        edges.update((h, hubs + int(v)) for v in rng.choice(leaves, d, replace=False))
    edges.update((h, h + 1) for h in range(0, hubs - 1, 3))
    return wl.graph_from_edge_list(hubs + leaves, sorted(edges), rng.integers(0, 6, hubs + leaves))


@pytest.mark.parametrize("graph", ["stars1", "stars8", "rmat12", "rmat17"])
@pytest.mark.parametrize("offset", [0, 1])
def test_rounds_equal_the_oracle(graph, offset):
    """offset: the columns start that many elements past a 16-byte boundary."""
    import torch
    from paper_1912_08453_gb300 import ccpm
    if graph.startswith("stars"):
        g = stars(int(graph[5:]), 5)
    else:
        g = wl.rmat_graph(int(graph[4:]), seed=9, labels="zipf", n_labels=6)
    ctx = ccpm.Context(0)
    col = torch.zeros(g.m_dir + offset, dtype=torch.int32, device="cuda:0")[offset:]
    col.copy_(torch.from_numpy(g.col))
    torch.cuda.synchronize()
    dev = ccpm.Graph(ctx, torch.from_numpy(g.row_ptr).cuda(), col, torch.from_numpy(g.labels).cuda())
    for tl, te in TEMPLATES:
        og = oracle.Graph(g.row_ptr, g.col, g.labels)
        omega, active = oracle.init(og, tl, te)
        rounds, scanned = oracle.lcc(og, tl, te, omega, active)
        t = ccpm.Template(ctx, tl, te)
        for opts in ({}, {"short_rows": 1}, {"short_rows": 1024}, {"hub_degree": 16}, {"hub_degree": 4096},
                     {"entry_labels": 1}, {"compact": 1}, {"compact": -1}):
            r = ccpm.prune(ctx, dev, t, ccpm.options(lcc_only=1, **opts))
            np.testing.assert_array_equal(r.omega(), omega)
            np.testing.assert_array_equal(r.edge_bitmap(), oracle.pack_bits(active))
            assert r.phase_rounds()[0] == rounds
            assert r.counts()["edges_scanned_lcc"] == scanned
            r.close()
        t.close()
    dev.close()
    ctx.close()
