"""The learned walk on producer and consumer warps, the producers running the
network, against the one-warp walk: in eight, four, two and one parts per
group, with bands of no cell, of fewer than 32 and of many; repeats bit for
bit."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

EPS = 0.05
NP = 13 * 64 + 64 + 64 * 64 + 64 + 64 * 3 + 3


def _model(tc):
    rng = np.random.default_rng(11)
    m = np.zeros(tc.MLP_NMODEL, np.float32)
    m[:NP] = 0.2 * rng.standard_normal(NP)
    m[NP:] = 1.0
    return m


@pytest.mark.parametrize("n,theta,band", [(1, 0.6, 0.5), (300, 0.9, 0.2), (5000, 0.67, 0.67), (5000, 0.67, 0.6),
                                          (20000, 0.67, 0.3), (50000, 0.6, 0.5), (70000, 0.67, 0.55)])
@pytest.mark.parametrize("gmax", [32, 64])
def test_learned_split(n, theta, band, gmax):
    from paper_1211_2293_gb300 import tc

    p, _, m = inputs.plummer(max(n, 2), seed=n, with_velocity=False)
    p, m = p[:n], m[:n]
    plain = tc.Context(want_pot=1)
    plain.build(p, m, 8)
    plain.forces(theta, EPS)
    phi = plain.get_acc(with_pot=True)[1]
    out = []
    for split in (0, 1):
        ctx = tc.Context(quad=1, split=split, gmax=gmax, verify=1)
        ctx.mlp_set(_model(tc), band)
        ctx.set_config(learned=1)
        ctx.build(p, m, 8)
        ctx.forces(theta, EPS)
        a = ctx.get_acc()
        out.append((ctx.lists(), ctx.mlp_evals(), a))
        ctx.forces(theta, EPS)
        assert np.array_equal(ctx.get_acc(), a)
    (l0, e0, a0), (l1, e1, a1) = out
    for k in l0:
        assert np.array_equal(l0[k], l1[k]), k
    assert e0 == e1
    # the walks' sums, and the same corrections added in another order: a
    # term F x label is at most some 4 times its cell's monopole term, itself
    # at most its potential / EPS, and takes at most 64 roundings
    lim = 2e-5 * np.linalg.norm(a0, axis=1) + 256 * 2.0**-24 * np.abs(phi) / EPS
    assert np.all(np.linalg.norm(a1 - a0, axis=1) <= 2 * lim)
