"""Loading a graph from arrays on the device waits for what makes the arrays on
the default stream, and not for other streams' work."""
import numpy as np
import pytest

from paper_1912_08453_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TL, TE = [5, 4, 8, 7, 4, 5], [(0, 1), (1, 2), (1, 3), (3, 4), (3, 5), (2, 3)]


def on_device(g):
    import torch
    return [torch.from_numpy(x).cuda() for x in (g.row_ptr, g.col, g.labels)]


def test_other_streams_are_not_waited_for():
    import torch
    from paper_1912_08453_gb300 import ccpm
    g = wl.rmat_graph(12, seed=3)
    arrays = on_device(g)
    ctx = ccpm.Context(0)
    ccpm.Graph(ctx, *arrays).close()              # first use of the context and its kernels
    torch.cuda.synchronize()
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2 * 10**9)              # about a second
        done.record()
    dev = ccpm.Graph(ctx, *arrays)
    assert not done.query()
    done.synchronize()
    dev.close()
    ctx.close()


def test_the_default_stream_is():
    import torch
    from paper_1912_08453_gb300 import ccpm
    g = wl.rmat_graph(12, seed=3)
    ready = on_device(g)
    late = [torch.zeros_like(x) for x in ready]
    ctx = ccpm.Context(0)
    torch.cuda.synchronize()
    torch.cuda._sleep(2 * 10**8)
    for x, y in zip(late, ready):
        x.copy_(y)
    dev = ccpm.Graph(ctx, *late)                  # counts the labels
    host = ccpm.Graph(ctx, g.row_ptr, g.col, g.labels)
    t = ccpm.Template(ctx, TL, TE)
    a, b = ccpm.prune(ctx, dev, t), ccpm.prune(ctx, host, t)
    np.testing.assert_array_equal(a.omega(), b.omega())
    # a state names its graph by the label counts among others
    c = ccpm.state_import(ctx, host, t, a.export_state())
    for x in (a, b, c, dev, host, t, ctx):
        x.close()
