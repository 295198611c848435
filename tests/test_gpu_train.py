"""The fused training loop against single steps made of the gradient kernel and
an Adam update in float64, on the same sampled rows, at the edges of its row
split (64-row tiles, one to eight blocks at work) and of the rule that selects it.

Tolerance: both sides round the same operands to BF16, so gradients differ by
the order of FP32 sums and by the odd activation that rounds to the neighbouring
BF16 value, about r = 2^-9 of a block's typical entry at the worst.  Adam's step
is lr times a function of the gradient's direction: an entry below r of the
typical one (a share of about r) can move by up to 2 lr the other way, which is
2 sqrt(r) = 0.09 of the displacement's norm; a block that is wrong is off by
more than 1.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BLOCKS = [("W1", 0, 1024), ("b1", 1024, 1088), ("W2", 1088, 5184), ("b2", 5184, 5248),
          ("w3", 5248, 5312), ("b3", 5312, 5313)]
M64 = (1 << 64) - 1


def sample(n, batch, seed, step):
    idx = []
    for i in range(batch):
        z = (seed + 0x9E3779B97F4A7C15 * (step * batch + i + 1)) & M64
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
        idx.append((z ^ (z >> 31)) % n)
    return np.array(idx)


@pytest.mark.parametrize("batch,n", [(1, 1), (5, 700), (32, 700), (33, 700), (64, 3), (65, 700), (256, 700),
                                     (257, 5000), (500, 5000), (4096, 5000), (4097, 5000)])
def test_training_steps(batch, n):
    from paper_1912_08453_gb300 import ccpm
    ctx = ccpm.Context(0)
    rng = np.random.default_rng(batch)
    X = rng.normal(size=(n, 16)).astype(np.float32)
    T = (rng.normal(size=n) + 2).astype(np.float32)
    net, one = ccpm.Mlp(ctx, seed=batch), ccpm.Mlp(ctx, seed=batch)
    p0 = net.params().astype(np.float64)
    p0[1024:1088] = rng.normal(size=64) * 0.1
    p0[5184:5248] = rng.normal(size=64) * 0.1
    net.set_params(p0.astype(np.float32))
    p0 = net.params().astype(np.float64)
    lr, seed, steps = 1e-3, 77, 3
    p, m1, m2 = p0.copy(), np.zeros_like(p0), np.zeros_like(p0)
    for s in range(steps):
        one.set_params(p.astype(np.float32))
        rows = sample(n, batch, seed, s)
        g, want_loss = one.gradient(X[rows], T[rows])
        g = g.astype(np.float64)
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        p = p - lr * (m1 / (1 - 0.9 ** (s + 1))) / (np.sqrt(m2 / (1 - 0.999 ** (s + 1))) + 1e-8)
    loss = net.train(X, T, steps=steps, batch=batch, lr=lr, seed=seed)
    assert abs(loss - want_loss) <= 1e-2 * abs(want_loss)
    got = net.params().astype(np.float64)
    for name, a, b in BLOCKS:
        d, ref = got[a:b] - p[a:b], p[a:b] - p0[a:b]
        assert np.linalg.norm(d) <= 0.09 * np.linalg.norm(ref) + 1e-7, (name, np.linalg.norm(d), np.linalg.norm(ref))


def test_training_is_repeatable():
    from paper_1912_08453_gb300 import ccpm
    ctx = ccpm.Context(0)
    rng = np.random.default_rng(5)
    X = rng.normal(size=(900, 16)).astype(np.float32)
    T = rng.normal(size=900).astype(np.float32)
    out = []
    for _ in range(2):
        net = ccpm.Mlp(ctx, seed=9)
        net.train(X, T, steps=40, batch=200, lr=1e-3, seed=3)
        out.append(net.params())
    assert np.array_equal(out[0], out[1])
