"""The tree at the edges of its kernels' blocks: 1024 bodies a counting block,
4096 a scan tile, leaf thresholds on both sides of the staged window (256), and
body counts on both sides of the one that sums internal cells in the leaves'
launch, all bit for bit against the oracle."""
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
    ctx.build(_dev(p), _dev(m), leaf)
    _compare_tree(ctx, oracle.Tree(p, m, leaf), 64)


@pytest.mark.parametrize("n", [(1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("kind", ["plummer", "masses"])
def test_moments_in_one_launch_or_by_level(kind, n):
    from paper_1211_2293_gb300 import tc

    p, _, m = _bodies(kind, n, 11)
    ctx = _ctx(tc)
    ctx.build(_dev(p), _dev(m), 16)
    _compare_tree(ctx, oracle.Tree(p, m, 16), 64)
