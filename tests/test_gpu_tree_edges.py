"""The tree at the edges of its kernels' blocks: 1024 bodies a counting block and
a small sort tile, 4096 a scan tile and the sort of one block, leaf thresholds
on both sides of the staged window (256), and body counts on both sides of the
one (2^19) that sums internal cells in the leaves' launch and sorts in small
tiles, all bit for bit against the oracle; built twice, the second time with
the first one's depth (the sort of the top digits and its completion)."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import _bodies, _compare_tree, _ctx, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1023, 1024, 1025, 4095, 4096, 4097, 8193])
@pytest.mark.parametrize("leaf", [1, 255, 256, 257])
def test_block_edges(n, leaf):
    from paper_1211_2293_gb300 import tc

    p, _, m = _bodies("plummer", n, n + leaf)
    ctx = _ctx(tc)
    t = oracle.Tree(p, m, leaf)
    for _ in range(2):
        ctx.build(_dev(p), _dev(m), leaf)
        _compare_tree(ctx, t, 64)


@pytest.mark.parametrize("n", [(1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("kind", ["plummer", "masses"])
def test_moments_in_one_launch_or_by_level(kind, n):
    from paper_1211_2293_gb300 import tc

    p, _, m = _bodies(kind, n, 11)
    ctx = _ctx(tc)
    t = oracle.Tree(p, m, 16)
    for _ in range(2):
        ctx.build(_dev(p), _dev(m), 16)
        _compare_tree(ctx, t, 64)


@pytest.mark.parametrize("nsys,size", [(2, 40), (40, 100), (41, 100), (300, 17), (257, 2100)])
def test_digits_shared_by_key_and_system(nsys, size):
    """Sorts whose topmost digits hold key and system bits together: every
    system's bodies in the order of the system built alone."""
    from paper_1211_2293_gb300 import tc

    n = nsys * size
    p, _, m = _bodies("random", n, nsys)
    off = np.arange(nsys + 1) * size
    ctx = tc.Context()
    for _ in range(2):
        ctx.build_batch(_dev(p), _dev(m), off, 4)
        tr = ctx.tree()
        for s in {0, 1, nsys // 2, nsys - 1}:
            t = oracle.Tree(p[off[s]:off[s + 1]], m[off[s]:off[s + 1]], 4)
            assert np.array_equal(tr["perm"][off[s]:off[s + 1]], t.perm + off[s])
            assert np.array_equal(tr["keys"][off[s]:off[s + 1]], t.keys)
