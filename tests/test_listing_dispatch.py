"""Which rows a match listing reads, on a stand-in for the CUDA runtime that counts
launches by name: the first listing of a graph copies the result's rows, later
ones of a small result read the graph's grouped rows, made once, unless there is
no room for these."""
import pytest

from paper_1912_08453_gb300 import ccpm
from paper_1912_08453_gb300 import workloads as wl
from tests.fake_cuda import fake, fake_library  # noqa: F401


@pytest.mark.parametrize("room", [True, False])
def test_listing_rows(fake, room):  # noqa: F811
    g = wl.rmat_graph(14, seed=3)
    ctx = ccpm.Context(0)
    graph, t = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels), ccpm.Template(ctx, [5, 4, 6, 3], [(0, 1), (1, 2), (2, 3)])
    r = ccpm.prune(ctx, graph, t, ccpm.options(run_final=0))      # (the final step groups the rows itself)
    calls = [b"k_live_entries", b"k_label_sort", b"k_final_items"]
    seen = []
    before = fake.fake_in_use()
    for i in range(3):
        if i == 1 and not room:
            fake.fake_limit(5 * g.m_dir // 2)                     # the grouped copy takes 5 bytes an entry
        assert r.matches(t, vertex_counts=True, device=False)[0] == 0
        seen.append([fake.fake_calls(c) for c in calls])
    assert fake.fake_bad() == 0
    copies = [x[0] for x in seen]
    assert copies == ([1, 1, 1] if room else [1, 2, 3])
    assert [x[1] for x in seen] == ([0, 1, 1] if room else [0, 0, 0])
    assert (fake.fake_in_use() - before >= 5 * g.m_dir) == room
    for x in (r, t, graph, ctx):
        x.close()
