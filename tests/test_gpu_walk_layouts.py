"""The split walk's body layouts (bodies per lane x list slices, chosen by a
group's size) at the sizes where they change, against FP64 direct sums."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

EDGES64 = [1, 2, 15, 16, 17, 31, 32, 33, 39, 40, 41, 47, 48, 49, 63, 64]
EDGES128 = EDGES64 + [65, 95, 96, 97, 127, 128]


def _check(ctx, p, m, off, eps, theta, pot):
    ctx.forces(theta, eps)
    out = ctx.get_acc(with_pot=pot)
    acc, ph = out if pot else (out, None)
    e2 = float(np.float32(eps)) ** 2
    for a, b in zip(off[:-1], off[1:]):
        x, w = p[a:b].astype(np.float64), m[a:b].astype(np.float64)
        for i in range(0, b - a, 512):  # rows of bodies
            r = slice(i, min(i + 512, b - a))
            d = x[None, :, :] - x[r, None, :]
            ri = 1.0 / np.sqrt((d * d).sum(2) + e2)
            t = d * (w[None, :] * ri**3)[:, :, None]
            ex, mag = t.sum(1), np.linalg.norm(t, axis=2).sum(1)
            # the sums' float32 rounding, as for every walk of the library
            err = np.linalg.norm(acc[a:b][r] - ex, axis=1)
            assert np.all(err <= 2e-5 * np.linalg.norm(ex, axis=1) + 32 * 2.0**-24 * mag)
            if pot:
                assert np.all(np.abs(ph[a:b][r] + ri @ w - w[r] / np.sqrt(e2)) <= 2e-5 * (ri @ w))


@pytest.mark.parametrize("gmax,repeat", [(64, 1), (64, 24), (64, 110), (128, 1), (128, 60)])
@pytest.mark.parametrize("precise,pot,tile", [(1, 0, 128), (1, 1, 64), (0, 1, 256)])
def test_group_sizes(gmax, repeat, precise, pot, tile):
    """One group per system: every layout, with eight, two and one part per
    group as the bodies grow in number; theta = 0 sums every body."""
    from paper_1211_2293_gb300 import tc

    sizes = (EDGES64 if gmax == 64 else EDGES128) * repeat
    n = sum(sizes)
    p, _, m = inputs.plummer(n, seed=n, with_velocity=False)
    off = np.concatenate([[0], np.cumsum(sizes)])
    ctx = tc.Context(gmax=gmax, precise=precise, want_pot=pot, tile=tile)
    ctx.build_batch(p, m, off, 4)
    _check(ctx, p, m, off[: len(EDGES128) + 1], 0.05, 0.0, bool(pot))


@pytest.mark.parametrize("n", [700, 1500, 4000])
@pytest.mark.parametrize("warps", [1, 2, 3, 4])
def test_lists_of_many_tiles(n, warps):
    """Groups whose list spans many tiles, with one to four teams in a block."""
    from paper_1211_2293_gb300 import tc

    p, _, m = inputs.plummer(n, seed=n, with_velocity=False)
    ctx = tc.Context(want_pot=1, warps=warps)
    ctx.build(p, m, 8)
    _check(ctx, p, m, np.array([0, n]), 0.02, 0.0, True)


def test_one_leaf_of_coincident_bodies():
    """A level-21 leaf of more bodies than leaf_max allows elsewhere."""
    from paper_1211_2293_gb300 import tc

    n = 4400
    p = np.full((n, 3), 0.25, np.float32)
    p[:60] = inputs.plummer(60, seed=1, with_velocity=False)[0]
    m = np.full(n, 1.0 / n, np.float32)
    ctx = tc.Context(want_pot=1)
    ctx.build(p, m, 8)
    _check(ctx, p, m, np.array([0, n]), 0.1, 0.0, True)
