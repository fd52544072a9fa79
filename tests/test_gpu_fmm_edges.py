"""The FMM's walk and radii where they can go wrong: cells that don't fill a
block's run of eight, cells that accept more than the 320 that wait together,
leaves of two equal bodies (both are the farthest), a cluster far smaller than
its cell's rounding unit; against the oracle, with the bounds of
test_gpu_fmm.py."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs
from tests.test_gpu_fmm import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf,theta", [(9, 1, 0.6), (65, 1, 0.6), (513, 4, 0.5), (6000, 2, 0.35), (3000, 3, 0.8)])
def test_fmm_small_trees_and_full_queues(tc, n, leaf, theta):
    p, _, m = inputs.plummer(n, 40 + n)
    _compare(tc, p, m, leaf, theta, 0.01, 1.0, f"{n} {leaf}")


def test_fmm_cluster_below_its_cells_rounding(tc):
    p, _, m = inputs.plummer(2000, 31)
    q, _, w = inputs.uniform_cube(500, 32)
    p = np.concatenate([np.float32(0.7) + p * np.float32(1e-4), q]).astype(np.float32)
    m = np.concatenate([m, w])
    _compare(tc, p, m, 8, 0.6, 0.01, 1.0, "cluster")
