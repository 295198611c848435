"""Which kernels the LCC rounds of a prune are queued as, by template and size (on
a stand-in for the CUDA runtime that counts launches by name)."""
import ctypes

import pytest

from paper_1912_08453_gb300 import ccpm
from paper_1912_08453_gb300 import workloads as wl
from tests.fake_cuda import fake, fake_library  # noqa: F401

PATH8 = ([0, 1, 2, 3, 4, 5, 6, 7], [(i, i + 1) for i in range(7)])
STAR8 = ([0, 1, 1, 2, 2, 3, 4, 5], [(0, i) for i in range(1, 8)])               # two classes
PATH9 = ([0, 1, 2, 3, 4, 5, 6, 7, 8], [(i, i + 1) for i in range(8)])
PATH17 = (list(range(17)), [(i, i + 1) for i in range(16)])
FOUR = ([0, 1, 1, 2, 2, 3, 3, 4, 4], [(0, i) for i in range(1, 9)])      # four classes
FIVE = ([5, 0, 0, 1, 1, 2, 2, 3, 3, 4, 4], [(0, i) for i in range(1, 11)])      # five classes


@pytest.mark.parametrize("huge,tmpl,rows", [
    (0, PATH8, True), (0, STAR8, True), (1 << 40, PATH8, False),
    (0, PATH9, False), (0, PATH17, False), (0, FOUR, False), (0, FIVE, False)])
def test_later_rounds(fake, huge, tmpl, rows):  # noqa: F811
    g = wl.rmat_graph(6, seed=3)
    ctx = ccpm.Context(0)
    f = ccpm.lib.ccpm_test_round_limits
    f.argtypes, f.restype = [ctypes.c_void_p] + 3 * [ctypes.c_int64], None
    for delta in (0, 1 << 40):
        f(ctx.h, huge, 1 << 40, delta)
        graph, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, *tmpl)
        before = [fake.fake_calls(k) for k in (b"k_rows", b"k_lcc_round", b"k_first_round", b"k_push")]
        ccpm.prune(ctx, graph, t, ccpm.options(lcc_only=1)).close()
        n_rows, n_lcc, n_first, n_push = (
            fake.fake_calls(k) - b for k, b in zip((b"k_rows", b"k_lcc_round", b"k_first_round", b"k_push"), before))
        # six rounds are queued; the first is k_first_round and k_rows over what it leaves, unless the
        # template has more than four classes
        first = int(tmpl is not FIVE)
        assert n_first == first
        assert (n_rows, n_lcc) == ((6, 0) if rows else (first, 6 - first))
        assert n_push == (4 if delta == 0 else 0)
        t.close()
        graph.close()
    ctx.close()
