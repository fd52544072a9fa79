"""tc_get_acc leaves the caller's buffers as they are when it reports a device
error, and fills them whatever memory and alignment they have."""
import numpy as np
import pytest
import torch

from paper_1211_2293_gb300 import inputs

pytestmark = pytest.mark.gpu


def _buffer(kind, n):
    """n floats, their first `off` floats into an allocation."""
    off = 1 if kind.endswith("odd") else 0
    if kind.startswith("device"):
        return torch.full((n + 4,), 7.0, device="cuda")[off:off + n]
    if kind.startswith("pinned"):
        return torch.full((n + 4,), 7.0).pin_memory()[off:off + n]
    return np.full(n + 4, 7.0, np.float32)[off:off + n]


def _host(x):
    return x.cpu().numpy() if isinstance(x, torch.Tensor) else x


@pytest.mark.parametrize("n", [1, 5, 4096, 100003])
@pytest.mark.parametrize("acc_in,pot_in", [("device", "device"), ("device_odd", "device_odd"), ("host", "host"),
                                           ("pinned", "pinned"), ("device", "host"), ("host_odd", "device_odd")])
def test_buffers_of_a_failed_phase(n, acc_in, pot_in):
    from paper_1211_2293_gb300 import tc

    p, _, m = inputs.plummer(max(n, 2), seed=3, with_velocity=False)
    p, m = p[:n], m[:n]
    ctx = tc.Context(want_pot=1)
    ctx.build(p, m, 4)
    ctx.forces(0.6, 0.01)
    want_acc, want_pot = ctx.get_acc(with_pot=True)
    acc, pot = _buffer(acc_in, 3 * n), _buffer(pot_in, n)
    ctx.get_acc(acc=acc, pot=pot)
    assert np.array_equal(_host(acc), want_acc.ravel()) and np.array_equal(_host(pot), want_pot)
    if n != 4096:
        return
    # a stack too small for theta = 0: what the buffers hold stays
    acc, pot = _buffer(acc_in, 3 * n), _buffer(pot_in, n)
    ctx.set_config(stack=64)
    ctx.forces(0.0, 0.01)
    with pytest.raises(tc.TcError) as e:
        ctx._c(ctx._lib.tc_get_acc(ctx._h, tc._ptr(acc), tc._ptr(pot)))
    assert e.value.code == tc.TC_EDEVICE
    assert np.all(_host(acc) == 7.0) and np.all(_host(pot) == 7.0)
