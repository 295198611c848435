"""Host side of the ordering network on a stand-in for the CUDA runtime: what a
single GPU cannot show (a second device, a device that takes no cluster)."""
import numpy as np
import pytest

from paper_1912_08453_gb300 import ccpm
from tests.fake_cuda import fake, fake_library  # noqa: F401

X, Y = np.zeros((5000, 16), np.float32), np.zeros(5000, np.float32)


@pytest.mark.parametrize("batch", [64, 5000])       # the fused loop, the kernels per step
def test_every_device_runs_it(fake, batch):  # noqa: F811
    """The kernels' shared memory is allowed for each device by itself."""
    for device in (0, 1, 0):
        ctx = ccpm.Context(device)
        net = ccpm.Mlp(ctx, seed=1)
        net.train(X, Y, steps=3, batch=batch)
        net.gradient(X, Y)
        net.forward(X)
        net.close()
        ctx.close()
    assert fake.fake_bad() == 0


@pytest.mark.parametrize("batch,clusters,fused", [(64, 1, True), (4096, 1, True), (4097, 1, False), (64, 0, False)])
def test_training_takes_the_kernels_per_step_without_a_cluster(fake, batch, clusters, fused):  # noqa: F811
    fake.fake_clusters(clusters)
    ctx = ccpm.Context(0)
    net = ccpm.Mlp(ctx, seed=1)
    net.train(X, Y, steps=3, batch=batch)
    assert fake.fake_calls(b"k_mlp_train") == int(fused)
    assert fake.fake_calls(b"k_mlp_backward") == fake.fake_calls(b"k_mlp_adam") == (0 if fused else 3)
    net.close()
    ctx.close()
