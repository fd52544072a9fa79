"""A rebuild that fails leaves the context without a tree: every call that needs
one says so (TC_ESTATE), nothing works from the failed tree's sizes, and the
next state or build that succeeds recovers."""
import numpy as np
import pytest
import torch

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

N = 3000


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _context(tc):
    p, v, m = inputs.plummer(N, 61)
    ctx = tc.Context(quad=1, want_pot=1, verify=1)
    ctx.build(_dev(p), _dev(m), 8)
    ctx.forces(0.6, 0.01)
    ctx.get_acc()
    return ctx, p, v, m


def _refused(tc, ctx):
    lists = np.zeros(4, np.int64)
    calls = [lambda: ctx.forces(0.6, 0.01), lambda: ctx.step(1e-3), lambda: ctx.fmm(0.5, 0.01), ctx.tree, ctx.systems,
             ctx.cube, ctx.lists, ctx.get_acc, lambda: ctx.group_list(0, 0.6), lambda: ctx.autotune(0.6, 0.01, reps=1),
             lambda: ctx.mlp_pairs(0.6, 0.01, 0.5, 1.0, 1, 100), ctx.fmm_stats]
    for call in calls:
        with pytest.raises(tc.TcError) as e:
            call()
        assert e.value.code == tc.TC_ESTATE, call
    lib, h = ctx._lib, ctx._h
    assert lib.tc_get_nodes(h, lists.ctypes.data, None, None, None, None, None, None, None, None) == tc.TC_ESTATE
    assert lib.tc_get_groups(h, lists.ctypes.data, None, None) == tc.TC_ESTATE


def _same_as_fresh(tc, ctx, p, m):
    ctx.forces(0.6, 0.01)
    acc = ctx.get_acc()
    ref = tc.Context(quad=1, want_pot=1, verify=1)
    ref.build(_dev(p), _dev(m), 8)
    ref.forces(0.6, 0.01)
    assert np.array_equal(acc, ref.get_acc())
    a, b = ctx.tree(), ref.tree()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_failed_state(tc, bad):
    ctx, p, v, m = _context(tc)
    sizes = ctx.sizes()
    # a state whose tree would be another one: far fewer or far more nodes
    for q in (np.zeros_like(p), np.random.default_rng(1).random((N, 3)).astype(np.float32)):
        q = q.copy()
        q[N // 2, 1] = bad
        with pytest.raises(tc.TcError) as e:
            ctx.set_state(_dev(q), _dev(v))
        assert e.value.code == tc.TC_EINVAL
        _refused(tc, ctx)
        assert ctx.sizes() == sizes
        x, _ = ctx.get_state()  # the bodies are there
        assert np.array_equal(x, q, equal_nan=True)
    # another configuration is no rebuild of what has no tree
    ctx.set_config(gmax=32)
    _refused(tc, ctx)
    ctx.set_config(gmax=64)
    ctx.set_state(_dev(p), _dev(v))
    _same_as_fresh(tc, ctx, p, m)


def test_failed_build(tc):
    ctx, p, v, m = _context(tc)
    q = p.copy()
    q[3, 0] = np.nan
    with pytest.raises(tc.TcError) as e:
        ctx.build(_dev(q), _dev(m), 8)
    assert e.value.code == tc.TC_EINVAL
    for call in (ctx.get_acc, ctx.sizes, lambda: ctx.step(1e-3), lambda: ctx.set_state(_dev(p), _dev(v))):
        with pytest.raises(tc.TcError) as e:
            call()
        assert e.value.code == tc.TC_ESTATE
    ctx.build(_dev(p), _dev(m), 8)
    _same_as_fresh(tc, ctx, p, m)


def test_step_that_outgrows_the_table(tc):
    """Bodies on two points that a step scatters: the step's tree does not fit,
    and afterwards the sizes are those of the tables, not of that tree."""
    n = 20000
    pos = np.zeros((n, 3), np.float32)
    pos[n // 2:] = 1.0
    vel = np.random.default_rng(0).standard_normal((n, 3)).astype(np.float32)
    mass = np.full(n, 1.0 / n, np.float32)
    ctx = tc.Context(quad=1, want_pot=1, verify=1)
    ctx.build(_dev(pos), _dev(mass), 8)
    ctx.set_velocity(_dev(vel))
    ctx.forces(0.5, 0.01)
    sizes = ctx.sizes()
    ctx.step(1.0)
    ctx.step(1.0)  # (enqueued behind the stopped one)
    with pytest.raises(tc.TcError) as e:
        ctx.sync()
    assert e.value.code == tc.TC_EDEVICE and "capacity" in str(e.value)
    assert ctx.sizes() == sizes
    _refused(tc, ctx)
    x, v = ctx.get_state()
    ctx.set_state(_dev(x), _dev(v))
    ctx.forces(0.5, 0.01)
    acc = ctx.get_acc()
    ref = tc.Context(quad=1, want_pot=1, verify=1)
    ref.build(_dev(x), _dev(mass), 8)
    ref.forces(0.5, 0.01)
    assert np.array_equal(acc, ref.get_acc())
