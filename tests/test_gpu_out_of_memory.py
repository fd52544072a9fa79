"""A call that finds no memory (TC_ALLOC_CAP_BYTES) leaves the context usable,
wherever among its buffers that happened: what was there and went with them is
refused, and the next call that finds memory gives what a fresh context does."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu


def _starved(tc, monkeypatch, call, after, step):
    """call under caps that grow by `step` bytes until it goes through; after
    every refusal after() without a cap.  Returns the refusals."""
    for k in range(400):
        monkeypatch.setenv("TC_ALLOC_CAP_BYTES", str(1 + k * step))
        try:
            call()
            return k
        except tc.TcError as e:
            assert e.code == tc.TC_ENOMEM
        finally:
            monkeypatch.delenv("TC_ALLOC_CAP_BYTES")
        after()
    pytest.fail("no cap let the call through")


def _evaluate(ctx, p, m):
    ctx.build(p, m, 8)
    ctx.forces(0.6, 0.01)
    return ctx.get_acc(), ctx.get_state()[1]


@pytest.mark.parametrize("big", ["one", "batch"])
def test_larger_build_refused(monkeypatch, big):
    from paper_1211_2293_gb300 import tc

    p, v, m = inputs.plummer(2000, 3)
    q, _, w = inputs.plummer(20000, 4)
    want, _ = _evaluate(tc.Context(), p, m)
    ctx = tc.Context()
    _evaluate(ctx, p, m)
    off = np.concatenate([[0], np.sort(np.random.default_rng(5).permutation(19998)[:3000] + 1), [20000]])

    def call():
        ctx.build(q, w, 8) if big == "one" else ctx.build_batch(q, w, off, 8)

    def after():
        for refused in (lambda: ctx.forces(0.6, 0.01), lambda: ctx.step(1e-3), ctx.get_acc, ctx.get_state, ctx.tree,
                        lambda: ctx.fmm(0.5, 0.01), lambda: ctx.set_velocity(v)):
            with pytest.raises(tc.TcError) as e:
                refused()
            assert e.value.code == tc.TC_ESTATE
        acc, vel = _evaluate(ctx, p, m)
        assert np.array_equal(acc, want) and not vel.any()
        ctx.set_velocity(v)
        ctx.step(1e-3)
        ctx.sync()

    assert _starved(tc, monkeypatch, call, after, 200000) > 5
    fresh = tc.Context()
    fresh.build(q, w, 8) if big == "one" else fresh.build_batch(q, w, off, 8)
    for c in (ctx, fresh):
        c.forces(0.6, 0.01)
    assert np.array_equal(ctx.get_acc(), fresh.get_acc())


def test_fmm_refused_after_a_larger_build(monkeypatch):
    from paper_1211_2293_gb300 import tc

    p, _, m = inputs.plummer(3000, 6)
    fresh = tc.Context()
    fresh.build(p, m, 8)
    fresh.fmm(0.5, 0.01)
    want = fresh.get_acc()
    for again in range(3):  # refused at the start, and further on
        ctx = tc.Context()
        ctx.build(p[:500], m[:500], 8)
        ctx.fmm(0.5, 0.01)
        ctx.build(p, m, 8)
        ctx.forces(0.6, 0.01)
        acc = ctx.get_acc()
        # (the treecode's accelerations are kept by a refused pass)
        assert _starved(tc, monkeypatch, lambda: ctx.fmm(0.5, 0.01), lambda: np.testing.assert_array_equal(ctx.get_acc(), acc),
                        300000 + 70000 * again) > 3
        assert np.array_equal(ctx.get_acc(), want)
        ctx.close()


@pytest.mark.parametrize("what", ["train", "forward", "pairs", "direct", "list", "learned"])
def test_other_scratch_refused(monkeypatch, what):
    """A small call, the larger one refused, the small one again: what it gives
    is what it gave."""
    from paper_1211_2293_gb300 import tc

    rng = np.random.default_rng(7)
    p, _, m = inputs.plummer(6000, 8)
    X = rng.standard_normal((20000, 13)).astype(np.float32)
    T = (0.3 * X[:, :3]).astype(np.float32)
    model = (0.1 * rng.standard_normal(tc.MLP_NMODEL)).astype(np.float32)
    idx = np.arange(6000, dtype=np.int64)
    quad = what in ("pairs", "learned")
    ctx = tc.Context(quad=int(quad))
    ctx.build(p, m, 8)
    if what in ("forward", "learned"):
        ctx.mlp_set(model, 0.5)

    def run(small):
        n = 200 if small else 20000
        if what == "train":
            return ctx.mlp_train(X[:n], T[:n], epochs=2, batch=128 if small else 8192)
        if what == "forward":
            return ctx.mlp_forward(X[:n])
        if what == "pairs":
            return ctx.mlp_pairs(0.6, 0.01, 0.5, 0.001 if small else 0.05, 9, 3000 if small else 60000)[0]
        if what == "direct":
            return ctx.direct(idx[:100] if small else idx, 0.01)[0]
        if what == "list":
            return ctx.group_list(1, 0.9 if small else 0.1)[0]
        ctx.set_config(learned=1, split=1 if small else 2)
        ctx.forces(0.7, 0.01)
        return ctx.get_acc()

    if what != "train":  # (a first call of everything is refused part-way too)
        run(True)
    first = None if what == "train" else run(True)

    def after():
        got = run(True)
        assert first is None or np.array_equal(got, first)

    _starved(tc, monkeypatch, lambda: run(False), after, 100000)
    # (the network run after the walk adds its cells to a group's sum by atomics, in no fixed order)
    last = what == "learned"
    got = run(last)
    used, ctx = ctx, tc.Context(quad=int(quad))
    ctx.build(p, m, 8)
    if what in ("forward", "learned"):
        ctx.mlp_set(model, 0.5)
    assert np.array_equal(run(last), got)
    used.close()


def test_training_memory_does_not_grow_with_the_passes(monkeypatch):
    """Thousands of passes run in the memory that one takes (and 32 kB), and a
    refused training leaves the model that was there."""
    from paper_1211_2293_gb300 import tc

    rng = np.random.default_rng(12)
    X = rng.standard_normal((64, 13)).astype(np.float32)
    T = (0.3 * X[:, :3]).astype(np.float32)
    free = tc.Context()
    want = free.mlp_train(X, T, epochs=8000, batch=16)
    ctx = tc.Context()
    k = _starved(tc, monkeypatch, lambda: ctx.mlp_train(X, T, epochs=1, batch=16), lambda: None, 4096)
    model = ctx.mlp_get()[0]
    monkeypatch.setenv("TC_ALLOC_CAP_BYTES", str(1 + k * 4096 + 32768))
    with pytest.raises(tc.TcError) as e:
        ctx.mlp_train(rng.standard_normal((5000, 13)).astype(np.float32), rng.standard_normal((5000, 3)).astype(np.float32))
    assert e.value.code == tc.TC_ENOMEM and np.array_equal(ctx.mlp_get()[0], model)
    assert np.array_equal(ctx.mlp_train(X, T, epochs=8000, batch=16), want)
    assert np.array_equal(ctx.mlp_get()[0], free.mlp_get()[0])


@pytest.mark.parametrize("systems", [1, 3])
def test_direct_sum_without_its_scratch(monkeypatch, systems):
    """Where the slices' sums find no memory fewer slices, or one, do: the same
    tiles' sums, added in FP64 in another grouping."""
    from paper_1211_2293_gb300 import tc

    n = 20000
    p, _, m = inputs.plummer(n, 13)
    off = np.array([0, n]) if systems == 1 else np.array([0, 400, 9000, n])
    idx = np.random.default_rng(14).permutation(n)[:300].astype(np.int64)
    free = tc.Context()
    free.build_batch(p, m, off, 8)
    want = free.direct(idx, 0.01)

    def build():
        build.ctx = tc.Context()
        build.ctx.build_batch(p, m, off, 8)

    k = _starved(tc, monkeypatch, build, lambda: build.ctx.close(), 100000)
    # room for the indices and results (14 kB) alone, for some slices, for all
    for more in (32768, 200000, 400000, 1 << 20):
        monkeypatch.setenv("TC_ALLOC_CAP_BYTES", str(1 + k * 100000 + more))
        got = build.ctx.direct(idx, 0.01)
        for a, b in zip(got, want):
            # 80 tiles' sums: each addition rounds at 2^-53 of what is added so far
            assert np.all(np.abs(a - b) <= 160 * 2.0**-53 * n * m[0] / 0.01**2)
        acc = np.zeros((300, 3))
        ctx = build.ctx
        ctx._c(ctx._lib.tc_direct(ctx._h, idx.ctypes.data, 300, 0.01, 1.0, acc.ctypes.data, None))
        assert np.array_equal(acc, got[0])
