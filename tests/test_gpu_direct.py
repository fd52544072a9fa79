"""tc_direct at the edges of its blocks (256 targets), tiles (256 sources) and
source slices, one system and several, against an FP64 direct sum."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu


def _direct64(p, m, off, idx, eps):
    acc, pot, mag = np.zeros((len(idx), 3)), np.zeros(len(idx)), np.zeros(len(idx))
    x, w, e2 = p.astype(np.float64), m.astype(np.float64), float(np.float32(eps)) ** 2
    for k, i in enumerate(idx):
        s = np.searchsorted(off, i, side="right") - 1
        a, b = off[s], off[s + 1]
        d = x[a:b] - x[i]
        ri = 1.0 / np.sqrt((d * d).sum(1) + e2)
        t = d * (w[a:b] * ri**3)[:, None]
        acc[k], mag[k] = t.sum(0), np.linalg.norm(t, axis=1).sum()
        pot[k] = w[i] * ri[i - a] - (w[a:b] * ri).sum()
    return acc, pot, mag


@pytest.mark.parametrize("sizes,ns", [([1], 1), ([255], 3), ([256], 256), ([257], 257), ([5000], 1), ([5000], 255),
                                      ([5000], 513), ([70001], 700), ([1, 2, 300, 255, 513], 257),
                                      ([4000, 4096, 7], 1024)])
def test_direct_edges(sizes, ns):
    from paper_1211_2293_gb300 import tc

    n, eps = sum(sizes), 0.01
    p, _, m = inputs.plummer(n, seed=n + ns, with_velocity=False)
    off = np.concatenate([[0], np.cumsum(sizes)])
    idx = inputs.sample_indices(n, min(n, ns), seed=5)
    ctx = tc.Context()
    ctx.build_batch(p, m, off, 16)
    acc, pot = ctx.direct(idx, eps)
    ea, ep, mag = _direct64(p, m, off, idx, eps)
    # each term a few float32 roundings, each tile a chain of 256 of them
    assert np.all(np.linalg.norm(acc - ea, axis=1) <= 1e-5 * np.linalg.norm(ea, axis=1) + 32 * 2.0**-24 * mag)
    assert np.all(np.abs(pot - ep) <= 4e-6 * np.abs(ep) + 1e-6 * m[idx] / eps)
