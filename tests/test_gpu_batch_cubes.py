"""Root cubes of batches on either side of the number of systems from which a
launch of their own forms them: those of the systems built alone, in a
synchronised build and inside a step, and bad input still reported."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys", [511, 512, 513, 3000])
def test_cubes_of_many_systems(nsys):
    from paper_1211_2293_gb300 import tc

    rng = np.random.default_rng(nsys)
    size = rng.integers(1, 9, nsys)
    size[[0, nsys // 2, nsys - 1]] = [1, 2500, 1100]  # one body; several chunks
    off = np.concatenate([[0], np.cumsum(size)])
    n = int(off[-1])
    scale = np.repeat(10.0 ** rng.uniform(-4, 3, nsys), size)[:, None]
    p = (rng.standard_normal((n, 3)) * scale).astype(np.float32)
    v = (rng.standard_normal((n, 3)) * scale).astype(np.float32)
    m = np.full(n, 1e-9, np.float32)
    check = np.concatenate([[0, nsys // 2, nsys - 1], rng.choice(nsys, 20)])

    def alone(x):
        out = []
        for s in check:
            c = tc.Context()
            c.build(x[off[s]:off[s + 1]], m[off[s]:off[s + 1]], 8)
            out.append(c.cube())
            c.close()
        return np.array(out)

    ctx = tc.Context()
    ctx.build_batch(p, m, off, 8)
    assert np.array_equal(ctx.systems()[1][check], alone(p))
    ctx.set_velocity(v)
    ctx.forces(0.6, 1.0)
    ctx.step(0.5)
    x, _ = ctx.get_state()
    assert not np.array_equal(x, p)
    assert np.array_equal(ctx.systems()[1][check], alone(x))
    bad = p.copy()
    bad[off[nsys // 2] + 2000, 2] = np.inf
    with pytest.raises(tc.TcError) as e:
        ctx.build_batch(bad, m, off, 8)
    assert e.value.code == tc.TC_EINVAL
