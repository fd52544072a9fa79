"""A captured step belongs to what it was captured from: after a change of that,
replayed steps give the same bits as steps launched one by one."""
import numpy as np
import pytest
import torch

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _state(ctx):
    return (*ctx.get_state(), ctx.get_acc())


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_other_split_of_the_same_bodies():
    """Batches of as many bodies and systems, split elsewhere: four and three
    bounding-box chunks, the root cubes far apart in size."""
    from paper_1211_2293_gb300 import tc

    n = 3072
    p, v, m = inputs.plummer(n, 71)
    offs = [np.array([0, 1500, n]), np.array([0, 1024, n])]
    out = []
    for graph in (0, 1):
        ctx = tc.Context(graph=graph)
        got = []
        ctx.build_batch(_dev(p), _dev(m), offs[0], 8)  # (room for four chunks before the first capture)
        for k in (1, 0, 1, 0):
            q = p.copy()
            q[offs[k][1]:] *= 7.0 + k
            ctx.build_batch(_dev(q), _dev(m), offs[k], 8)
            ctx.set_velocity(_dev(v))
            ctx.forces(0.6, 0.01)
            for _ in range(2):
                ctx.step(0.5)
            got.append((*_state(ctx), ctx.systems()[1]))
        out.append(got)
    for a, b in zip(*out):
        _same(a, b)


@pytest.mark.parametrize("shallow_again", [False, True])
def test_deeper_tree_built_since_the_capture(shallow_again):
    """A step captured on an even cloud, then a state of as many bodies and
    nodes with 20000 of them in a cube of side 1e-4, more than a step orders
    within a run of equal digits: its steps sort the digits of that tree."""
    from paper_1211_2293_gb300 import tc

    n, tight = 40000, 20000
    rng = np.random.default_rng(81)
    p = rng.random((n, 3)).astype(np.float32)
    q = p.copy()
    q[:tight] = (0.3 + 1e-4 * rng.random((tight, 3))).astype(np.float32)
    v, m = np.zeros_like(p), np.full(n, 1.0 / n, np.float32)
    out = []
    for graph in (0, 1):
        ctx = tc.Context(graph=graph)
        ctx.build(_dev(p), _dev(m), 16)
        got = []
        for x in (p, q, p) if shallow_again else (p, q):
            ctx.set_state(_dev(x), _dev(v))
            ctx.forces(0.7, 0.01)
            for _ in range(2):
                ctx.step(1e-6)
            got.append(_state(ctx))
        out.append(got)
    for a, b in zip(*out):
        _same(a, b)


@pytest.mark.parametrize("cfg", [dict(quad=1, quadrupole=1), dict(want_pot=1, gmax=128)])
@pytest.mark.parametrize("between", ["list", "other"])
def test_timed_step_after_another_walk(cfg, between):
    """With phase timing the walk follows the graph: it is the configuration's,
    whatever walk ran between two steps."""
    from paper_1211_2293_gb300 import tc

    p, v, m = inputs.plummer(5000, 91)
    out = []
    for timing in (False, True):
        ctx = tc.Context(**cfg)
        ctx.set_timing(timing)
        ctx.build(_dev(p), _dev(m), 8)
        ctx.set_velocity(_dev(v))
        ctx.forces(0.6, 0.01)
        ctx.group_list(3, 0.3)  # (its scratch: a buffer that grows drops the graph)
        ctx.step(1e-3)
        if between == "list":
            ctx.group_list(3, 0.9)
        else:
            keep = ctx.config()
            ctx.set_config(quadrupole=0, split=0)
            ctx.forces(0.6, 0.01)
            ctx.set_config(**keep)
        ctx.step(1e-3)
        out.append(_state(ctx))
    _same(*out)
