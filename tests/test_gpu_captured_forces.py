"""A force phase that the caller captures into a CUDA graph of its own: replayed
on trees built later it gives what a direct call gives, and capturing it does
not count as having run it."""
import numpy as np
import pytest
import torch

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

CFGS = [dict(), dict(split=0), dict(quad=1, quadrupole=1), dict(gmax=128, want_pot=1)]
# in parts and in tree order, in parts and ordered, whole and ordered
SIZES = [3000, 10007, 100003]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _clouds(n):
    """As many bodies, and other numbers of groups."""
    rng = np.random.default_rng(n)
    p, _, m = inputs.plummer(n, 5)
    q = rng.random((n, 3)).astype(np.float32)
    r = (0.5 + 0.01 * rng.random((n, 3))).astype(np.float32)
    r[: n // 3] = q[: n // 3]
    return (p, q, r), m


def _direct(tc, cfg, x, m):
    ctx = tc.Context(**cfg)
    ctx.build(_dev(x), _dev(m), 8)
    ctx.forces(0.6, 0.05)
    return ctx.get_acc()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("cfg", CFGS)
@pytest.mark.parametrize("warm", [True, False])
def test_replayed_on_later_trees(cfg, n, warm):
    """warm: forces and their groups' order are there before the capture;
    else the tree has just been built."""
    from paper_1211_2293_gb300 import tc

    clouds, m = _clouds(n)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = tc.Context(**cfg)
        # the node tables have room for every cloud before the capture (a
        # larger tree would move them away from under the graph)
        for x in (clouds[1], clouds[2], clouds[0]):
            ctx.build(_dev(x), _dev(m), 8)
        ctx.forces(0.6, 0.05)
        ctx.sync()
        if not warm:
            ctx.build(_dev(clouds[1]), _dev(m), 8)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.forces(0.6, 0.05)
        # captured, not run: a direct call does the whole phase
        ctx.forces(0.6, 0.05)
        assert np.array_equal(ctx.get_acc(), _direct(tc, cfg, clouds[0 if warm else 1], m))
        for x in (clouds[1], clouds[2], clouds[0]):
            ctx.build(_dev(x), _dev(m), 8)
            ctx.forces(0.9, 0.05)  # (other forces on the tree in between)
            g.replay()
            assert np.array_equal(ctx.get_acc(), _direct(tc, cfg, x, m))
        # another size of groups and back: the graph's buffers are still its own
        if cfg.get("gmax", 64) == 64:
            ctx.set_config(gmax=128 if not cfg.get("quadrupole") else 32)
            ctx.forces(0.6, 0.05)
            ctx.set_config(gmax=64)
            ctx.forces(0.9, 0.05)
            g.replay()
            assert np.array_equal(ctx.get_acc(), _direct(tc, cfg, clouds[0], m))


@pytest.mark.parametrize("n", SIZES)
def test_first_force_phase_captured(n):
    """No force phase before the capture: nothing is allocated in it, and the
    groups are walked whole (the sums differ from those of parts by the float32
    rounding of the lists' order)."""
    from paper_1211_2293_gb300 import tc

    (x, _, _), m = _clouds(n)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = tc.Context(want_pot=1)
        ctx.build(_dev(x), _dev(m), 8)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.forces(0.6, 0.05)
        g.replay()
        acc, pot = ctx.get_acc(with_pot=True)
        ref = tc.Context(want_pot=1)
        ref.build(_dev(x), _dev(m), 8)
        ref.forces(0.6, 0.05)
        a0, p0 = ref.get_acc(with_pot=True)
    # each sum within 2e-5 of the result and 32 roundings of the terms'
    # magnitudes, and a term is at most its potential / eps
    lim = 2e-5 * np.linalg.norm(a0, axis=1) + 32 * 2.0**-24 * np.abs(p0) / 0.05
    assert np.all(np.linalg.norm(acc - a0, axis=1) <= 2 * lim)
    assert np.all(np.abs(pot - p0) <= 4e-5 * (np.abs(p0) + m / 0.05))
