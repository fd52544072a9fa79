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
