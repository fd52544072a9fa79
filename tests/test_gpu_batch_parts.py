"""Parts of the groups of a batch, which follow the size of the system a body is
in: on both sides of the sizes where their number changes, the one-warp walk's
lists and sums, and a replayed step the bits of steps launched one by one."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs
from tests.test_gpu_walk_parts import _both, _compare, EPS

pytestmark = pytest.mark.gpu

# bodies of a system: a part per 64 (few tasks) or 512 (more tasks than teams)
SIZES = [[7] * 300, [127] * 20, [128] * 20, [511] * 20, [512] * 20, [300] * 50, [1023] * 30, [1024] * 30, [64] * 700,
         [1] * 50 + [2000], [3000, 1, 1, 9, 64]]


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: f"{len(s)}x{s[-1]}")
def test_parts_of_batches(sizes):
    from paper_1211_2293_gb300 import tc

    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])
    p, v, m = inputs.plummer(n, seed=n)

    def make(split):
        ctx = tc.Context(want_pot=1, verify=1, split=split)
        ctx.build_batch(p, m, off, 8)
        return ctx

    _compare(_both(make, lambda ctx: ctx.forces(0.5, EPS)), m)
    out = []
    for graph in (0, 1):
        ctx = tc.Context(graph=graph)
        ctx.build_batch(p, m, off, 8)
        ctx.set_velocity(v)
        ctx.forces(0.5, EPS)
        ctx.step(1e-3)
        ctx.step(1e-3)
        out.append((*ctx.get_state(), ctx.get_acc()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
