"""Leaves longer than the steps their end is looked for one by one: coincident
bodies around that length, each run followed by the next, and root leaves of a
batch, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import _compare_tree, _ctx, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 8, 33, 4096])
@pytest.mark.parametrize("level_launches", [False, True])
def test_coincident_runs(tc, leaf, level_launches):
    rng = np.random.default_rng(leaf)
    runs = [1, 31, 32, 33, 34, 35, 64, 65, 1000, 3000, 1]
    spots = rng.random((len(runs), 3))
    near = spots + 2.0**-20 * rng.integers(0, 2, spots.shape)  # neighbours of a spot, a few grid steps off
    p = np.vstack([np.repeat(spots, runs, 0), np.repeat(near, runs[::-1], 0)])
    if level_launches:  # past 2^19 bodies the internal cells follow by level
        p = np.vstack([p, rng.random(((1 << 19) + 1 - len(p), 3))])
    p = rng.permutation(p).astype(np.float32)
    m = rng.uniform(0.5, 2.0, len(p)).astype(np.float32)
    ctx = _ctx(tc)
    t = oracle.Tree(p, m, leaf)
    for _ in range(2):
        ctx.build(_dev(p), _dev(m), leaf)
        _compare_tree(ctx, t, 64)


def test_root_leaves_of_a_batch():
    from paper_1211_2293_gb300 import tc

    sizes = [1, 32, 33, 34, 100, 4096, 2, 33]
    off = np.concatenate([[0], np.cumsum(sizes)])
    rng = np.random.default_rng(5)
    p = rng.random((off[-1], 3)).astype(np.float32)
    p[off[4]:off[5]] = 0.25
    m = rng.uniform(0.5, 2.0, off[-1]).astype(np.float32)
    ctx = tc.Context()
    ctx.build_batch(p, m, off, 4096)
    tr = ctx.tree()
    assert len(tr["count"]) == len(sizes)
    assert np.array_equal(tr["first"], off[:-1]) and np.array_equal(tr["count"], sizes)
    for s in range(len(sizes)):
        M = m[off[s]:off[s + 1]].astype(np.float64).sum()
        assert abs(tr["mass"][s] - M) <= 1e-12 * M
