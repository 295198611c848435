"""The gradient a training step uses, parameter by parameter, against the gradient
kernel on the same rows.

Adam's first step moves a parameter by lr g / (|g| + 1e-8).  With inputs, targets
and biases of about 1e-9 every g lies far below 1e-8, where this is linear in g,
so that the step gives g back; and lr = 1e10 makes the step as large as the
parameters, so that little is lost in p - step.

Tolerance, per parameter: both sides round the same operands to BF16 and sum the
64 rows of a tile in the same order; what may differ is the order of the tiles'
sums, by tiles * 2^-23 of the sum of their magnitudes (taken from the gradient
of each tile).  Reading g back costs 2^-23 of the larger of p before and after,
and some ten FP32 roundings of the step.  A lost or doubled tile, a wrong
1/batch or a row of padding that counts is larger than that a thousand times over."""
import numpy as np
import pytest

from tests.test_gpu_train import BLOCKS, sample

pytestmark = pytest.mark.gpu

U = 2.0 ** -23


@pytest.mark.parametrize("batch", [1, 5, 63, 64, 65, 256, 257, 500, 512, 513, 1000, 4095, 4096, 4097])
def test_gradient_of_a_step(batch):
    from paper_1912_08453_gb300 import ccpm
    ctx = ccpm.Context(0)
    rng = np.random.default_rng(batch)
    n, lr, seed = 5000, 1e10, 77
    X = (1e-9 * rng.normal(size=(n, 16))).astype(np.float32)
    T = (1e-9 * rng.normal(size=n)).astype(np.float32)
    net = ccpm.Mlp(ctx, seed=batch)
    p0 = net.params()
    for name, a, b in BLOCKS:
        if name[0] == "b":
            p0[a:b] = 1e-9 * rng.normal(size=b - a)
    net.set_params(p0)
    rows = sample(n, batch, seed, 0)
    want, want_loss = net.gradient(X[rows], T[rows])
    tiles = [rows[i:i + 64] for i in range(0, batch, 64)]
    sums = sum(len(t) / batch * np.abs(net.gradient(X[t], T[t])[0].astype(np.float64)) for t in tiles)
    net.set_params(p0)
    loss = net.train(X, T, steps=1, batch=batch, lr=lr, seed=seed)
    p1 = net.params().astype(np.float64)
    d = (p0 - p1) / lr
    got = 1e-8 * d / (1 - np.abs(d))
    tol = (len(tiles) + 1) * U * sums + 1e-8 * U * np.maximum(np.abs(p0), np.abs(p1)) / lr + 20 * U * np.abs(want)
    assert abs(loss - want_loss) <= (len(tiles) + 64) * U * want_loss
    for name, a, b in BLOCKS:
        off = np.abs(got[a:b] - want[a:b])
        assert np.all(off <= tol[a:b]), (name, float((off / tol[a:b]).max()))
        assert np.abs(want[a:b]).max() > 1000 * tol[a:b].min()      # what is compared is well above the tolerance
    net.close()
    ctx.close()
