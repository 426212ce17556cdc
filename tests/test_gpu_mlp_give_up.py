"""A training pass whose tensor-core waits gave up (marked so from the host, as the kernel does it) takes no Adam
step: weights, moments and step count stay as they were, the error is reported once by the next call that synchronises,
and the run goes on as if the lost steps had not been asked for."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import _lib, sgs  # noqa: E402

pytestmark = pytest.mark.gpu


def _data(seed, P=1000):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((10, P), generator=g, device="cuda"), torch.randn((6, P), generator=g, device="cuda")


def _give_up(net):
    _lib.check(_lib.lib().dns_mlp_debug_give_up(net._h), "dns_mlp_debug_give_up")


@pytest.mark.parametrize("report", ["get_params", "train_step", "loss_grad"])
def test_no_step_on_sums_that_are_not_valid(report):
    X, T = _data(1)
    net, ref = sgs.MLP(seed=2), sgs.MLP(seed=2)
    for n in (net, ref):
        for _ in range(3):
            n.train_step(X, T, 1e-2, want_loss=False)
    before = net.get_params()
    _give_up(net)
    for _ in range(2):
        net.train_step(X, T, 1e-2, want_loss=False)
    with pytest.raises(RuntimeError, match="TIMEOUT"):
        if report == "get_params":
            net.get_params()
        elif report == "train_step":
            net.train_step(X, T, 1e-2)
        else:
            net.loss_grad(X, T)
    assert np.array_equal(net.get_params(), before)
    X, T = _data(3)
    assert net.train_step(X, T, 1e-2) == ref.train_step(X, T, 1e-2)
    assert np.array_equal(net.get_params(), ref.get_params())
    net.close()
    ref.close()


def test_new_parameters_end_it():
    X, T = _data(4)
    net, ref = sgs.MLP(seed=5), sgs.MLP(seed=6)
    _give_up(net)
    net.train_step(X, T, 1e-2, want_loss=False)
    net.set_params(sgs.init_params(6))
    for n in (net, ref):
        n.train_step(X, T, 1e-2, want_loss=False)
    with pytest.raises(RuntimeError, match="TIMEOUT"):  # still to be reported
        net.get_params()
    assert np.array_equal(net.get_params(), ref.get_params())
    assert _lib.lib().dns_mlp_debug_give_up(ctypes.c_void_p()) == _lib.DNS_ERR_ARG
    net.close()
    ref.close()
