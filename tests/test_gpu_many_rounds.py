"""Fixpoints that take hundreds of rounds: more than the 8-bit marks of the wide
LCC tell apart, and more groups of queued rounds than any sampled graph needs.

The graph: a path whose ends lose one vertex a round (every template vertex has
two neighbours, so a vertex with one active neighbour dies), its middle joined
to one of two hubs that share all their leaves and stay.  Nothing near the hubs
changes for as long as the path lasts, and then the joined hub's row does."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1912_08453_gb300 import workloads as wl
from tests.test_gpu_wide import check

pytestmark = pytest.mark.gpu

TRIANGLE = ([0, 0, 0], [(0, 1), (1, 2), (0, 2)])


def path_and_hubs(length, leaves):
    hubs = [length, length + 1]
    edges = [(i, i + 1) for i in range(length - 1)] + [(length // 2, hubs[0])]
    edges += [(h, length + 2 + i) for h in hubs for i in range(leaves)]
    return wl.graph_from_edge_list(length + 2 + leaves, edges, [0] * (length + 2 + leaves))


# rows of the hubs: short, one warp, a block, chunks
@pytest.mark.parametrize("length,leaves", [(511, 20), (514, 500), (1301, 2000), (600, 9000)])
def test_wide(length, leaves):
    from paper_1912_08453_gb300 import ccpm
    g = path_and_hubs(length, leaves)
    ctx = ccpm.Context(0)
    check(ctx, g, *TRIANGLE)
    el = np.zeros(g.m_dir, np.uint8)
    check(ctx, g, *TRIANGLE, [0, 0, 0], el)
    ctx.close()


@pytest.mark.parametrize("limits", [(1 << 62, 0, 0), (0, 0, 0), (1 << 62, 1 << 62, 1 << 62)])
@pytest.mark.parametrize("length,leaves", [(511, 20), (514, 500), (1301, 2000)])
def test_prune(length, leaves, limits):
    from paper_1912_08453_gb300 import ccpm
    g = path_and_hubs(length, leaves)
    og = oracle.Graph(g.row_ptr, g.col, g.labels)
    omega, active = oracle.init(og, *TRIANGLE)
    rounds, scanned = oracle.lcc(og, *TRIANGLE, omega, active)
    assert rounds > length // 2
    ctx = ccpm.Context(0)
    f = ccpm.lib.ccpm_test_round_limits
    f.argtypes, f.restype = [ctypes.c_void_p] + 3 * [ctypes.c_int64], None
    f(ctx.h, *limits)
    dev, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, *TRIANGLE)
    for opts in ({}, {"hub_degree": 64}, {"compact": 1}):
        r = ccpm.prune(ctx, dev, t, ccpm.options(lcc_only=1, **opts))
        np.testing.assert_array_equal(r.omega(), omega)
        np.testing.assert_array_equal(r.edge_bitmap(), oracle.pack_bits(active))
        assert r.phase_rounds() == [rounds]
        assert r.counts()["edges_scanned_lcc"] == scanned
        assert r.counts()["lcc_launches"] == rounds
        r.close()
    for x in (t, dev, ctx):
        x.close()
