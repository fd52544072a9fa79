"""The split walk's parts per group (chosen by the number of groups), at the
sizes where their number changes, against the one-warp walk: the same lists,
and sums that agree to the float32 rounding of both."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

# groups (0.7 gmax bodies) x parts <= 20 per SM: 8 parts up to 17024 bodies on
# 152 SMs, 4 up to 34048, 2 up to 68096; groups ordered from 6810 on
EPS = 0.05
SIZES = [1, 2, 63, 65, 300, 6800, 6820, 17020, 17030, 34040, 34060, 68090, 68100]


def _both(make, forces):
    out = []
    for split in (0, 1):
        ctx = make(split)
        forces(ctx)
        acc = ctx.get_acc(with_pot=True)
        out.append((ctx.lists(), *acc))
        forces(ctx)  # again on the same tree
        assert np.array_equal(ctx.get_acc(), acc[0])
        ctx.close()
    return out


def _compare(out, m):
    (l0, a0, p0), (l1, a1, p1) = out
    for k in l0:
        assert np.array_equal(l0[k], l1[k]), k
    # each walk's sums: 2e-5 of the result and 32 roundings of the terms'
    # magnitudes, and a term is at most its potential / EPS
    lim = 2e-5 * np.linalg.norm(a0, axis=1) + 32 * 2.0**-24 * np.abs(p0) / EPS
    assert np.all(np.linalg.norm(a1 - a0, axis=1) <= 2 * lim)
    assert np.all(np.abs(p1 - p0) <= 4e-5 * (np.abs(p0) + m / EPS))


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("theta", [0.0, 0.6])
def test_parts_list_alike(n, theta):
    from paper_1211_2293_gb300 import tc

    if theta == 0.0 and n > 7000:
        pytest.skip("all pairs")
    p, _, m = inputs.plummer(max(n, 2), seed=n, with_velocity=False)
    p, m = p[:n], m[:n]

    def make(split):
        ctx = tc.Context(want_pot=1, verify=1, split=split)
        ctx.build(p, m, 8)
        return ctx

    _compare(_both(make, lambda ctx: ctx.forces(theta, EPS)), m)


def test_parts_of_systems():
    """Systems of one leaf, of one body and of many groups in one batch."""
    from paper_1211_2293_gb300 import tc

    sizes = [1, 3, 8, 9, 64, 65, 500, 4000, 1, 200]
    off = np.concatenate([[0], np.cumsum(sizes)])
    p, _, m = inputs.plummer(int(off[-1]), seed=3, with_velocity=False)

    def make(split):
        ctx = tc.Context(want_pot=1, verify=1, split=split)
        ctx.build_batch(p, m, off, 8)
        return ctx

    _compare(_both(make, lambda ctx: ctx.forces(0.5, EPS)), m)


def test_parts_without_their_scratch(monkeypatch):
    """Where the parts' sums find no memory the groups are walked whole."""
    from paper_1211_2293_gb300 import tc

    p, _, m = inputs.plummer(5000, seed=4, with_velocity=False)
    free = tc.Context()
    free.build(p, m, 8)
    free.forces(0.6, EPS)
    a0 = free.get_acc()
    for cap in range(1, 64):  # the smallest cap (in 100 kB) that lets the build through
        monkeypatch.setenv("TC_ALLOC_CAP_BYTES", str(100000 * cap))
        ctx = tc.Context()
        try:
            ctx.build(p, m, 8)
        except tc.TcError:
            ctx.close()
            continue
        for _ in range(2):
            ctx.forces(0.6, EPS)
            a1 = ctx.get_acc()
            assert np.all(np.linalg.norm(a1 - a0, axis=1) <= 4e-5 * np.linalg.norm(a0, axis=1).mean())
        break
    else:
        pytest.fail("no cap let the build through")
