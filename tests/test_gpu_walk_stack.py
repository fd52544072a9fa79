"""The walk stack of the learned split walk is the one asked for: a tree that
needs more than the default overflows there (reported) and is walked with a
larger setting."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NP = 13 * 64 + 64 + 64 * 64 + 64 + 64 * 3 + 3


def _nested(levels=16):
    """Bodies whose tree keeps the stack growing: of each cube [-s, 0]^3 the
    seven children away from the origin hold eight cells of two bodies each,
    the eighth is the next cube.  At theta = 0 a walk that opens the newest
    cells first comes to hold 895 opened cells (leaf_max 1)."""
    out = []
    for lev in range(levels):
        h = 2.0 ** -lev / 2
        for c in range(7):
            corner = np.array([-2 * h + h * ((c >> b) & 1) for b in (2, 1, 0)])
            for k in range(8):
                o = corner + [h / 2 * ((k >> b) & 1) for b in (2, 1, 0)]
                out += [o + h / 8, o + 3 * h / 8]
    p = np.array(out)
    p[0] = -1 + 2.0 ** -22  # the root cube is [-1, 0]^3
    return np.vstack([p, np.full(3, -2.0 ** -19)]).astype(np.float32)


@pytest.mark.parametrize("tile", [64, 128, 256])
@pytest.mark.parametrize("warps", [1, 4])
def test_learned_walk_takes_the_stack_asked_for(tile, warps):
    from paper_1211_2293_gb300 import tc

    p = _nested()
    n = len(p)
    m = np.full(n, 1.0 / n, np.float32)
    rng = np.random.default_rng(11)
    model = np.ones(tc.MLP_NMODEL, np.float32)
    model[:NP] = 0.2 * rng.standard_normal(NP)

    def walk(split, stack):
        # (a group per body: with that many groups each is walked whole)
        ctx = tc.Context(quad=1, gmax=1, split=split, stack=stack, tile=tile, warps=warps, verify=1)
        ctx.mlp_set(model, 0.5)
        ctx.set_config(learned=1)
        ctx.build(p, m, 1)
        ctx.forces(0.0, 0.05)
        return ctx.get_acc(), ctx.lists()

    if warps == 4:
        with pytest.raises(tc.TcError) as e:
            walk(1, 600)
        assert e.value.code == tc.TC_EDEVICE and "stack" in str(e.value)
    a0, l0 = walk(0, 4096)
    for stack in (2048, 8192):
        a1, l1 = walk(1, stack)
        for k in l0:
            assert np.array_equal(l0[k], l1[k]), k
        # all pairs: both sums within 32 roundings of the terms' magnitudes,
        # which are at most 1 / EPS^2 in all (unit mass)
        assert np.abs(a1 - a0).max() <= 2 * 32 * 2.0 ** -24 / 0.05 ** 2 + 4e-5 * np.abs(a0).max()
