"""The sort of one block where runs of equal top digits are as long as it ranks,
one longer, most of the bodies or all of them: built again on the depth of an
even cloud, and inside a step, the order is the full sort's, bit for bit."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import _ctx, _dev

pytestmark = pytest.mark.gpu


def _compare_tree(ctx, t):
    """Order and nodes (the moments of cells as small as the coordinates'
    rounding have no bound to be held to)."""
    tr = ctx.tree()
    for k in ("perm", "keys", "level", "prefix", "first", "count", "child_first", "nchild"):
        assert np.array_equal(tr[k], getattr(t, k)), k


def _cloud(n, runs, spread, seed):
    rng = np.random.default_rng(seed)
    p = rng.random((n, 3))
    at = 0
    for k, r in enumerate(runs):
        p[at:at + r] = 0.1 + 0.2 * k + spread * rng.random((r, 3))
        at += r
    return rng.permutation(p).astype(np.float32)


@pytest.mark.parametrize("n,runs", [(300, [63, 1]), (300, [64]), (300, [65]), (1000, [128, 129]), (1025, [63, 64, 65, 66]),
                                    (4096, [1000, 300]), (4096, [4096]), (4095, [2048, 64, 65])])
@pytest.mark.parametrize("spread", [0.0, 1e-5])
def test_long_runs(tc, n, runs, spread):
    rng = np.random.default_rng(n)
    even = rng.random((n, 3)).astype(np.float32)
    p = _cloud(n, runs, spread, n + len(runs))
    m = rng.uniform(0.5, 2.0, n).astype(np.float32)
    ctx = _ctx(tc)
    ctx.build(_dev(even), _dev(m), 8)  # the depth that the next sort counts on
    ctx.build(_dev(p), _dev(m), 8)
    _compare_tree(ctx, oracle.Tree(p, m, 8))
    # inside a step, on the even cloud's depth again: the drift makes the runs
    ctx.build(_dev(even), _dev(m), 8)
    ctx.forces(0.6, 0.01)
    dt = 2.0**-10
    ctx.set_velocity(_dev(((p.astype(np.float64) - even) / dt).astype(np.float32)))
    ctx.forces(0.6, 1e3, 0.0)
    ctx.step(dt)
    x, _ = ctx.get_state()
    _compare_tree(ctx, oracle.Tree(x, m, 8))


def test_long_runs_of_systems(tc):
    """System bits above the key's, runs that end at a system's last body."""
    sizes = [200, 1, 65, 64, 1500, 40]
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])
    rng = np.random.default_rng(3)
    even = rng.random((n, 3)).astype(np.float32)
    p = even.copy()
    for s in (0, 2, 3, 4):
        p[off[s] + 1:off[s + 1]] = 0.5 + 1e-6 * rng.random((sizes[s] - 1, 3))
    m = np.ones(n, np.float32)
    ctx = tc.Context()
    for x in (even, p):
        ctx.build_batch(_dev(x), _dev(m), off, 8)
    tr = ctx.tree()
    for s in range(len(sizes)):
        t = oracle.Tree(p[off[s]:off[s + 1]], m[off[s]:off[s + 1]], 8)
        assert np.array_equal(tr["perm"][off[s]:off[s + 1]], t.perm + off[s])
        assert np.array_equal(tr["keys"][off[s]:off[s + 1]], t.keys)
