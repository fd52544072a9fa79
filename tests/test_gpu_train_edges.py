"""A training pass (one cooperative launch) against the same steps taken one
gradient at a time, at batch sizes around its tiles (16 rows), blocks (64 rows)
and last, shorter mini-batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NP = 13 * 64 + 64 + 64 * 64 + 64 + 64 * 3 + 3


def _pairs(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, 13)).astype(np.float32)
    T = (X[:, :3] * 0.3 + 0.05 * rng.standard_normal((n, 3))).astype(np.float32)
    return X, T, rng.uniform(0.5, 2.0, n).astype(np.float32)


@pytest.mark.parametrize("n,batch", [(16, 16), (17, 16), (63, 64), (64, 64), (65, 64), (130, 64), (1000, 1024),
                                     (2049, 1024), (20000, 20000), (20001, 20000)])
def test_one_step_is_gradient_and_adam(n, batch):
    """After a pass of one step (or two) the parameters are the fresh ones
    moved by Adam with the library's own gradient of each mini-batch, within
    the float32 rounding of the update (the first step moves every parameter
    by lr g / (|g| + eps), so a gradient at rounding level may go either way:
    those are held to the step's size)."""
    from paper_1211_2293_gb300 import tc

    X, T, W = _pairs(n, n + batch)
    lr, seed = 1e-3, 7
    ctx = tc.Context()
    ctx.mlp_train(X, T, W, epochs=1, batch=batch, lr=lr, seed=seed)
    got, _ = ctx.mlp_get()
    # a pass at a vanishing learning rate leaves the fresh parameters and maps
    ref = tc.Context()
    loss0 = ref.mlp_train(X, T, W, epochs=1, batch=batch, lr=1e-30, seed=seed)
    fresh, _ = ref.mlp_get()
    assert np.array_equal(got[NP:], fresh[NP:])  # the maps come from the data alone
    if n <= batch:
        loss, g = ref.mlp_loss_grad(X, T, W)
        assert abs(loss - loss0[0]) <= 1e-5 * abs(loss)
        step = (fresh[:NP] - got[:NP]).astype(np.float64)
        exp = lr * g.astype(np.float64) / (np.abs(g) + 1e-8)
        clear = np.abs(g) > 1e-4 * np.abs(g).max()
        assert np.all(np.abs(step - exp)[clear] <= 2.0**-22 * np.abs(fresh[:NP][clear]) + 1e-3 * lr)
        assert np.all(np.abs(step) <= lr * 1.001 + 2.0**-22 * np.abs(fresh[:NP]))
    else:
        # two Adam steps, the second at the decayed rate
        assert 0 < np.abs(fresh[:NP] - got[:NP]).max() <= 2 * lr * 1.001 + 1e-6
    again = tc.Context()
    again.mlp_train(X, T, W, epochs=1, batch=batch, lr=lr, seed=seed)
    assert np.array_equal(again.mlp_get()[0], got)
