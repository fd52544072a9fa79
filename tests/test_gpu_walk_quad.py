"""The quadrupole walk on producer and consumer warps against the one-warp
walk: the same lists, and sums that agree to the float32 rounding of both; at
group sizes where the layout changes, with lists of a few cells and of many
tiles, in one and in eight parts per group."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

EPS = 0.05


def _both(p, m, off, leaf, theta, **cfg):
    from paper_1211_2293_gb300 import tc

    out = []
    for split in (0, 1):
        ctx = tc.Context(quad=1, quadrupole=1, want_pot=1, verify=1, split=split, **cfg)
        ctx.build_batch(p, m, off, leaf)
        ctx.forces(theta, EPS)
        out.append((ctx.lists(), *ctx.get_acc(with_pot=True)))
        ctx.close()
    (l0, a0, p0), (l1, a1, p1) = out
    for k in l0:
        assert np.array_equal(l0[k], l1[k]), k
    # each walk's sums: 2e-5 of the result and 32 roundings of the terms'
    # magnitudes; a monopole term is at most its potential / EPS and its
    # quadrupole term at most that again
    lim = 2e-5 * np.linalg.norm(a0, axis=1) + 64 * 2.0**-24 * np.abs(p0) / EPS
    assert np.all(np.linalg.norm(a1 - a0, axis=1) <= 2 * lim)
    assert np.all(np.abs(p1 - p0) <= 4e-5 * (np.abs(p0) + m / EPS))


@pytest.mark.parametrize("gmax", [32, 64])
@pytest.mark.parametrize("n,leaf,theta", [(1, 1, 0.5), (70, 1, 1.0), (3000, 1, 0.6), (20000, 4, 0.4), (80000, 8, 0.7)])
def test_quad_systems(n, leaf, theta, gmax):
    p, _, m = inputs.plummer(max(n, 2), seed=n, with_velocity=False)
    _both(p[:n], m[:n], np.array([0, n]), leaf, theta, gmax=gmax)


@pytest.mark.parametrize("repeat", [1, 40])
def test_quad_group_sizes(repeat):
    """Systems of 1 to 64 bodies: one group each."""
    sizes = [1, 2, 15, 16, 17, 31, 32, 33, 40, 41, 47, 48, 49, 63, 64] * repeat
    off = np.concatenate([[0], np.cumsum(sizes)])
    p, _, m = inputs.plummer(int(off[-1]), seed=5, with_velocity=False)
    _both(p, m, off, 2, 0.8)
