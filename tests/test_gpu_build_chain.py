"""Builds whose kernels overlap their predecessors' ends: two inputs of
different trees built and walked in turn, without a wait in between, give the
same bits every time, up to and past the size that overlaps."""
import numpy as np
import pytest

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 5000, 20000, 300000, (1 << 19), (1 << 19) + 1])
def test_builds_in_turn(n):
    import torch

    from paper_1211_2293_gb300 import tc

    sets = []
    for make, seed in ((inputs.plummer, 1), (inputs.uniform_cube, 2)):
        p, _, m = make(n, seed)
        sets.append((torch.from_numpy(np.ascontiguousarray(p)).cuda(), torch.from_numpy(np.ascontiguousarray(m)).cuda()))
    ctx = tc.Context()
    ref = []
    for p, m in sets:
        ctx.build(p, m, 16)
        ctx.forces(0.7, 0.05)
        ref.append((ctx.get_acc(), ctx.tree()["prefix"]))
    for k in range(12):
        p, m = sets[k % 2]
        ctx.build(p, m, 16)
        ctx.forces(0.7, 0.05)
        acc, prefix = ref[k % 2]
        if k % 4 > 1:
            assert np.array_equal(ctx.get_acc(), acc)
            assert np.array_equal(ctx.tree()["prefix"], prefix)
