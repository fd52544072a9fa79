"""A training pass of several mini-batches against the same steps restated: the
seeded order of the pairs, the library's own gradient of each mini-batch (set as
a model, another kernel) and Adam with the decayed rate and bias corrections in
numpy float32.  Pins what a pass carries from step to step: the rows of the next
batch, the model rewritten in between, the moments, the schedule, a shorter last
batch, several rounds of a batch in the cluster's blocks, and the next pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NP = 13 * 64 + 64 + 64 * 64 + 64 + 64 * 3 + 3
M64 = (1 << 64) - 1
f32 = np.float32


def _splitmix(z):
    z = (z + np.uint64(0x9E3779B97F4A7C15))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _order(n, key):
    """The pass's permutation: a four-round Feistel network on [0, 4^h), its
    cycle walked until the value falls below n."""
    h = 1
    while (1 << (2 * h)) < n:
        h += 1
    mask = np.uint64((1 << h) - 1)

    def rounds(x):
        L, R = x >> np.uint64(h), x & mask
        for r in range(4):
            f = _splitmix(np.uint64((key + 0x632BE59BD9B4E019 * r) & M64) + R) & mask
            L, R = R, L ^ f
        return (L << np.uint64(h)) | R

    with np.errstate(over="ignore"):
        x = rounds(np.arange(n, dtype=np.uint64))
        while (x >= n).any():
            out = x >= n
            x[out] = rounds(x[out])
    return x.astype(np.int64)


@pytest.mark.parametrize("n,batch,epochs", [(300, 120, 1), (2500, 1000, 1), (700, 256, 3), (129, 64, 4), (9000, 4096, 1),
                                            (20001, 20000, 1), (12000, 5000, 2)])
@pytest.mark.parametrize("weighted", [False, True])
def test_steps_of_a_pass(n, batch, epochs, weighted):
    from paper_1211_2293_gb300 import tc

    rng = np.random.default_rng(n + batch)
    X = rng.standard_normal((n, 13)).astype(f32)
    T = (X[:, :3] * 0.3 + 0.05 * rng.standard_normal((n, 3))).astype(f32)
    W = rng.uniform(0.5, 2.0, n).astype(f32) if weighted else None
    lr, seed = 1e-3, 7
    ctx = tc.Context()
    ctx.mlp_train(X, T, W, epochs=epochs, batch=batch, lr=lr, seed=seed)
    got = ctx.mlp_get()[0][:NP]
    ref = tc.Context()
    ref.mlp_train(X, T, W, epochs=1, batch=batch, lr=1e-30, seed=seed)  # the fresh parameters and the maps
    model = ref.mlp_get()[0]
    p, maps = model[:NP].copy(), model[NP:].copy()
    m, v = np.zeros(NP, f32), np.zeros(NP, f32)
    b1, b2 = f32(0.9), f32(0.999)
    steps = (n + batch - 1) // batch
    clear = np.ones(NP, bool)
    key = seed
    for ep in range(epochs):
        key = (key * 6364136223846793005 + 1442695040888963407) & M64
        order = _order(n, key)
        assert np.array_equal(np.sort(order), np.arange(n))
        for k in range(steps):
            rows = order[k * batch:(k + 1) * batch]
            ref.mlp_set(np.concatenate([p, maps]), 0.5)
            g = ref.mlp_loss_grad(X[rows], T[rows], None if W is None else W[rows])[1]
            clear &= np.abs(g) > 1e-2 * np.abs(g).max()
            t = ep * steps + k
            rate = f32(0.5 * lr * (1 + np.cos(np.pi * t / (epochs * steps))))
            c1, c2 = f32(1) - b1 ** f32(t + 1), f32(1) - b2 ** f32(t + 1)
            m = ((1 - b1).astype(np.float64) * g + b1 * m).astype(f32)
            v = (((1 - b2) * g).astype(np.float64) * g + b2 * v).astype(f32)
            p = p - rate * (m / c1) / (np.sqrt(v / c2) + f32(1e-8))
    moved = np.abs(p - model[:NP])
    assert clear.sum() >= 30  # (the last batch of 129 pairs in 64s is one row)
    # float32 rounding of a few operations a step moves a parameter by some
    # 1e-6 of the rate; where that turns the BF16 rounding of a weight the next
    # gradients change by 2^-9 of that weight's share of them, far below 0.05
    # of a gradient that is a hundredth of the largest.  Rows, a model or
    # moments of another step change the normalised update by tenths
    err = np.abs(got - p)
    assert err[clear].max() <= 0.05 * lr + 2.0**-22
    assert np.median(err) <= 1e-3 * lr + 2.0**-22
    assert moved[clear].max() > 0.5 * lr
