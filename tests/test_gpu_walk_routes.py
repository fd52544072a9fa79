"""split = 1 takes the one-warp walk where that is the faster one: there its bits
are those of split = 0, elsewhere the lists are and the sums agree to rounding;
and a replayed step takes the walk that a direct call takes."""
import numpy as np
import pytest
import torch

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu

EPS = 0.05
NP = 13 * 64 + 64 + 64 * 64 + 64 + 64 * 3 + 3
QUAD = dict(quad=1, quadrupole=1)
LEARN = dict(quad=1, learned=1)
# systems, bodies of each, configuration, theta, band, the one-warp walk is taken
# (on 152 SMs: 12 / 20 / 40 groups of 45 bodies an SM are 81700 / 136200 / 272400 bodies)
CASES = [
    (9100, 15, {}, 0.6, 0, True), (9000, 15, {}, 0.6, 0, True), (3000, 15, {}, 0.6, 0, False), (17000, 8, {}, 0.6, 0, False),
    (460, 300, {}, 0.6, 0, True), (460, 301, {}, 0.6, 0, False), (1, 140000, {}, 0.6, 0, False),
    (140, 600, QUAD, 0.6, 0, True), (140, 601, QUAD, 0.6, 0, False), (130, 600, QUAD, 0.6, 0, False),
    (1, 271000, QUAD, 0.9, 0, False), (1, 274000, QUAD, 0.9, 0, True), (1, 274000, QUAD, 0.8, 0, False),
    (1, 274000, dict(QUAD, want_pot=1), 0.65, 0, True), (1, 274000, dict(QUAD, want_pot=1), 0.62, 0, False),
    (1, 82000, dict(QUAD, warps=1), 0.7, 0, True), (1, 81000, dict(QUAD, warps=1), 0.7, 0, False),
    (1, 82000, dict(QUAD, stack=2048), 0.7, 0, True),
    (28, 3000, LEARN, 0.67, 0.55, True), (28, 3010, LEARN, 0.67, 0.55, False), (27, 3000, LEARN, 0.67, 0.55, False),
    (1, 274000, LEARN, 0.67, 0.55, False), (1, 274000, LEARN, 0.67, 0.5, True), (1, 274000, LEARN, 0.75, 0.7, True),
    (1, 271000, LEARN, 0.9, 0.5, False), (1, 274000, dict(LEARN, gmax=128), 0.9, 0.5, False),
    (1, 82000, dict(LEARN, gmax=32), 0.67, 0.55, True), (1, 81000, dict(LEARN, gmax=32), 0.67, 0.55, False),
    (1500, 1000, dict(LEARN, gmax=128), 0.67, 0.55, True), (1, 140000, dict(LEARN, gmax=128, warps=1), 0.67, 0.55, False),
    (1, 82000, dict(LEARN, tile=256), 0.67, 0.55, True), (1, 82000, dict(LEARN, tile=64), 0.67, 0.55, False),
]


@pytest.mark.parametrize("nsys,k,cfg,theta,band,one_warp", CASES)
def test_route(nsys, k, cfg, theta, band, one_warp):
    from paper_1211_2293_gb300 import tc

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are those of 152 SMs")
    n = nsys * k
    off = np.arange(nsys + 1) * k
    p, v, m = inputs.plummer(n, seed=nsys)
    dp, dv, dm = (torch.from_numpy(x).cuda() for x in (p, v, m))
    model = np.ones(tc.MLP_NMODEL, np.float32)
    model[:NP] = 0.2 * np.random.default_rng(11).standard_normal(NP)

    def context(**more):
        c = dict(cfg, **more)
        learned = c.pop("learned", 0)
        ctx = tc.Context(**c)
        if learned:
            ctx.mlp_set(model, band)
            ctx.set_config(learned=1)
        ctx.build_batch(dp, dm, off, 8)
        return ctx

    out = []
    for split in (0, 1):
        ctx = context(split=split, verify=1)
        ctx.forces(theta, EPS)
        out.append((ctx.lists(), ctx.get_acc()))
    (l0, a0), (l1, a1) = out
    for key in l0:
        assert np.array_equal(l0[key], l1[key]), key
    assert np.array_equal(a0, a1) == one_warp
    # both walks' sums, and corrections of some 4 times their cells' terms at most
    assert np.abs(a1 - a0).max() <= 2 * 256 * 2.0**-24 * m.sum() / EPS**2
    if n > 100000 and nsys == 1:
        return
    steps = []
    for graph in (0, 1):
        ctx = context(graph=graph)
        ctx.set_velocity(dv)
        ctx.forces(theta, EPS)
        ctx.step(1e-4)
        steps.append((*ctx.get_state(), ctx.get_acc()))
    for a, b in zip(*steps):
        assert np.array_equal(a, b)
