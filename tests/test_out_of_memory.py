"""A refused allocation is an error of its call and of no other: the next call
on the same context finds a whole workspace, or makes one, and no stale error."""
import numpy as np
import pytest

from paper_1912_08453_gb300 import ccpm
from paper_1912_08453_gb300 import workloads as wl
from tests.fake_cuda import fake, fake_library  # noqa: F401

TL, TE = [5, 4, 8, 7, 4, 5], [(0, 1), (1, 2), (1, 3), (3, 4), (3, 5), (2, 3)]


@pytest.fixture()
def env(fake):  # noqa: F811
    g = wl.rmat_graph(6, seed=3)
    ctx = ccpm.Context(0)
    graph, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, TL, TE)
    yield fake, g, ctx, graph, t
    for x in (t, graph, ctx):            # before the library is the real one again
        x.close()


def fails_then_works(f, call, attempts):
    """Refuse the 1st, 2nd, ... allocation of call(k), and those after it: it reports
    CCPM_ENOMEM, and the same call then works and touches no missing buffer."""
    refused = 0
    for k in range(1, attempts + 1):
        f.fake_fail_at(k)
        try:
            call(k)
        except ccpm.CcpmError as e:
            assert e.code == ccpm.CCPM_ENOMEM, (k, str(e))
            refused += 1
        else:
            assert f.fake_allocs() < k, f"allocation {k} was refused, and the call went on"
        f.fake_fail_at(0)
        call(k)
        assert f.fake_bad() == 0, f"after refusing allocation {k}"
    assert 0 < refused < attempts            # every allocation was refused once


@pytest.mark.parametrize("kind", ["prune", "lcc_only", "matches", "explore", "batch"])
def test_pruning(env, kind):
    f, g, ctx, graph, t = env
    kept = ccpm.prune(ctx, graph, t)

    def call(k):
        # another piece length each time: the workspace is made again
        o = ccpm.options(hub_degree=16 + k, batch_workers=1, lcc_only=int(kind == "lcc_only"))
        if kind == "matches":
            kept.matches(t, vertex_counts=True, opts=o)
        elif kind == "explore":
            ccpm.explore(ctx, graph, t, 1, o)[1].close()
        elif kind == "batch":
            for r in ccpm.prune_batch(ctx, graph, [t], o):
                r.close()
        else:
            ccpm.prune(ctx, graph, t, o).close()

    fails_then_works(f, call, 60)
    kept.close()


def test_wide(env):
    f, g, ctx, graph, t = env
    fails_then_works(f, lambda k: ccpm.lcc_wide(ctx, graph, TL, TE), 4)


def test_network(env):
    f, g, ctx, graph, t = env
    x, y = np.zeros((64, 16), np.float32), np.zeros(64, np.float32)

    def call(k):
        net = ccpm.Mlp(ctx, seed=1)
        try:
            net.train(x, y, steps=2, batch=64)
            net.gradient(x, y)
            net.forward(x)
        finally:
            net.close()

    fails_then_works(f, call, 8)


@pytest.mark.parametrize("kind", ["prune", "lcc_only", "resume", "matches", "explore"])
def test_pruning_takes_less_where_memory_is_short(env, kind, monkeypatch):
    """Half of the item lists (64 B each, 2^22 and 2^20 of them for a small graph)
    and the lists of delta rounds (16 B a vertex) are wanted, not needed."""
    f, g, ctx, graph, t = env
    o = ccpm.options(lcc_only=int(kind == "lcc_only"))
    first = ccpm.prune(ctx, graph, t, o)
    state = first.export_state()
    first.close()
    o.resume = int(kind == "resume")

    def need(limit):
        """The call's peak, on a context of its own and with this much memory."""
        c = ccpm.Context(0)
        r = ccpm.state_import(c, graph, t, state) if kind in ("resume", "matches") else None
        before = f.fake_in_use()
        f.fake_limit(limit)
        try:
            if kind == "matches":
                monkeypatch.setattr(graph, "ctx", c)      # the context the call runs on
                r.matches(t, vertex_counts=True, entry_counts=True)
            elif kind == "explore":
                r = ccpm.explore(c, graph, t, 1, o)[1]
            else:
                r = ccpm.prune(c, graph, t, o, result=r)
            return f.fake_peak() - before
        finally:
            f.fake_limit(1 << 60)
            if r is not None:
                r.close()
            c.close()
            assert f.fake_bad() == 0

    wanted = need(1 << 60)
    least = wanted - 32 * (2**22 + 2**20) - 16 * g.n
    for limit in (wanted, wanted - 1, wanted - 4 * g.n, wanted - 2**20, least):
        assert need(limit) <= limit
    with pytest.raises(ccpm.CcpmError) as e:
        need(least // 2)
    assert e.value.code == ccpm.CCPM_ENOMEM
