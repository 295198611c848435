"""Every round kernel on graphs the oracle can check.  Which kernel a round takes
depends on the entries in the active rows, and the lines lie at 2^22 and 2^28
entries: here they are moved, so that small graphs take the kernels of huge
ones, with each width of the narrow omega (1 and 2 bytes, none), with and
without multiplicity classes, changes of rounds and of non-local checks, and
other row splits.  Everything is integer and must equal the oracle."""
import ctypes
import math
from collections import Counter

import numpy as np
import pytest

import oracle
from oracle import pipeline
from paper_1912_08453_gb300 import workloads as wl
from tests.test_gpu_rounds import TEMPLATES, stars

pytestmark = pytest.mark.gpu

NEVER = 1 << 62
# (huge, inline, delta): k_rows everywhere, deltas or not; k_lcc_round with deltas; long rows of the
# first round inside k_first_round or after it
LIMITS = [(0, 0, 0), (0, NEVER, 0), (0, 0, NEVER), (NEVER, 0, 0), (NEVER, NEVER, 0), (NEVER, 0, NEVER)]


def context(limits):
    from paper_1912_08453_gb300 import ccpm
    ctx = ccpm.Context(0)
    f = ccpm.lib.ccpm_test_round_limits
    f.argtypes, f.restype = [ctypes.c_void_p] + 3 * [ctypes.c_int64], None
    f(ctx.h, *limits)
    return ctx


def sampled(g, n0, extra):
    """A template that matches: its LCC leaves something for rounds to work on.
    Loading a template counts its automorphisms one by one, so samples with many
    equal leaves are passed over."""
    for seed in range(10000):
        tl, te, _ = wl.sampled_template(g, np.zeros(g.m_dir, np.uint8), n0, extra, seed)
        ends = np.bincount(np.asarray(te).ravel())
        leaves = Counter((a + b - v, tl[v]) for a, b in te for v in (a, b) if ends[v] == 1)
        if math.prod(math.factorial(k) for k in leaves.values()) <= 1000:
            return tl, te
    raise AssertionError("no such sample")


@pytest.fixture(scope="module")
def cases():
    """Graphs, templates and the oracle's LCC fixpoints."""
    out = []
    for name, g in (("stars", stars(4, 5)), ("rmat", wl.rmat_graph(13, seed=9, labels="zipf", n_labels=12)),
                    ("degree", wl.rmat_graph(13, seed=2))):
        templates = list(TEMPLATES) if name == "stars" else TEMPLATES[2:4]
        # 1-byte omega, 2-byte, none; few and many classes
        templates += [sampled(g, n0, extra) for n0, extra in ((6, 0), (8, 3), (9, 0), (16, 4), (17, 2), (32, 6))]
        ref = []
        og = oracle.Graph(g.row_ptr, g.col, g.labels)
        for tl, te in templates:
            omega, active = oracle.init(og, tl, te)
            rounds, scanned = oracle.lcc(og, tl, te, omega, active)
            ref.append((tl, te, omega, oracle.pack_bits(active), rounds, scanned))
        out.append((g, ref))
    return out


@pytest.mark.parametrize("limits", LIMITS)
def test_first_fixpoint(cases, limits):
    from paper_1912_08453_gb300 import ccpm
    ctx = context(limits)
    for g, ref in cases:
        dev = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels)
        for tl, te, omega, bits, rounds, scanned in ref:
            t = ccpm.Template(ctx, tl, te)
            for opts in ({}, {"hub_degree": 16, "short_rows": 1024}, {"hub_degree": 100}, {"short_rows": 300},
                         {"entry_labels": 1}, {"compact": 1}, {"no_edge_elimination": 1}):
                r = ccpm.prune(ctx, dev, t, ccpm.options(lcc_only=1, **opts))
                what = f"{len(tl)} vertices, {opts}"
                np.testing.assert_array_equal(r.omega(), omega, err_msg=what)
                if "no_edge_elimination" not in opts:
                    np.testing.assert_array_equal(r.edge_bitmap(), bits, err_msg=what)
                    assert r.phase_rounds() == [rounds], what
                    assert r.counts()["edges_scanned_lcc"] == scanned, what
                    # and from that state: nothing left to do
                    again = ccpm.prune(ctx, dev, t, ccpm.options(lcc_only=1, resume=1, **opts), result=r)
                    np.testing.assert_array_equal(again.omega(), omega, err_msg=what)
                    np.testing.assert_array_equal(again.edge_bitmap(), bits, err_msg=what)
                r.close()
            t.close()
        dev.close()
    ctx.close()


# labels that repeat, cycles: checks that eliminate, and rounds after them
CHECKED = [
    ([5, 4, 8, 7, 4, 5], [(0, 1), (1, 2), (1, 3), (3, 4), (3, 5), (2, 3)]),
    ([7, 8, 7, 4, 4, 6], [(0, 1), (1, 2), (2, 3), (3, 0), (0, 4), (4, 5)]),
    ([6, 7, 6, 7, 8], [(0, 1), (0, 2), (0, 3), (0, 4), (1, 2), (1, 3), (1, 4), (2, 3), (2, 4), (3, 4)]),
    ([5, 6, 7, 8, 6, 5, 4, 7, 5], [(0, 1), (1, 2), (2, 3), (3, 0), (3, 4), (4, 5), (5, 6), (6, 7), (7, 4), (2, 8)]),
]


@pytest.fixture(scope="module")
def checked():
    g = wl.rmat_graph(13, labels="degree", seed=4)
    ref = [pipeline.run(g.row_ptr, g.col, g.labels, tl, te, max_embeddings=1 << 20) for tl, te in CHECKED]
    assert sum(sum(r.phase_rounds[1:]) for r in ref) > 0     # rounds after a check that eliminated
    return g, ref


@pytest.mark.parametrize("limits", LIMITS)
def test_rounds_after_checks(checked, limits):
    from paper_1912_08453_gb300 import ccpm
    g, refs = checked
    ctx = context(limits)
    dev = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels)
    for (tl, te), ref in zip(CHECKED, refs):
        t = ccpm.Template(ctx, tl, te)
        for opts in ({}, {"hub_degree": 16}, {"compact": -1}, {"compact": -1, "hub_degree": 100, "short_rows": 1024},
                     {"search_split": 1}, {"compact": 1}):
            r = ccpm.prune(ctx, dev, t, ccpm.options(max_embeddings=1 << 20, **opts), allow_budget=True)
            c = r.counts()
            np.testing.assert_array_equal(r.omega(), ref.omega, err_msg=str(opts))
            np.testing.assert_array_equal(r.edge_bitmap(), ref.ebits, err_msg=str(opts))
            assert r.phase_rounds() == ref.phase_rounds, opts
            assert c["edges_scanned_lcc"] == ref.lcc_scanned, opts
            assert c["lcc_launches"] == sum(ref.phase_rounds), opts
            r.close()
        t.close()
    dev.close()
    ctx.close()
