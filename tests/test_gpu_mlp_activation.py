"""The activation of the network kernels over its whole range: SiLU and its slope vanish for strongly negative
arguments of any size, and follow the reference elsewhere. One path z -> SiLU -> times a power of two that
brings it to order one -> SiLU -> output; three BF16 roundings (2^-9 relative each) are left between the kernel and the
reference with the same roundings: held to 2^-6."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sgs_mlp as sg  # noqa: E402
from paper_1602_03638_gb300 import sgs  # noqa: E402

pytestmark = pytest.mark.gpu


def _net(z, w2):
    v = np.zeros(5286, dtype=np.float32)
    v[10:20] = 1
    v[660:724] = z
    v[724] = w2  # W2[0][0]
    v[4884:4890] = 1  # W3[0][:]
    v[5274:5280] = 1
    return v


@pytest.mark.parametrize("z", [-41.0, -30.0, -5.0, -0.5, 0.5, 5.0, 40.0, 80.0, 1e4, 1e20])
def test_one_path(z):
    a = z / (1 + np.exp(-z))
    v = _net(z, 2.0 ** -np.round(np.log2(abs(a))))
    X = np.zeros((130, 10), dtype=np.float32)
    net = sgs.MLP(v)
    y = net.forward(torch.from_numpy(X.T.copy()).cuda()).cpu().numpy().T
    net.close()
    ref = sg.forward(sg.unflatten(v.astype(np.float64)), X.astype(np.float64), round_bf16=True)
    want = ref["tau"] if "tau" in ref else ref["y"]
    assert np.abs(y - want).max() <= 2.0 ** -6 * np.abs(want).max()


@pytest.mark.parametrize("z", [-60.0, -1e3, -1e10, -1e20, -1e38])
def test_vanishes_below(z):
    v = _net(z, 1.0)
    v[724:4820] = 1  # all of W2
    v[4820:4884] = 0.5  # b2
    X = torch.ones((10, 300), device="cuda")
    T = torch.zeros((6, 300), device="cuda")
    net = sgs.MLP(v)
    y = net.forward(X).cpu().numpy()
    assert np.abs(y - 0.5 / (1 + np.exp(-0.5))).max() <= 2.0 ** -8
    _, g = net.loss_grad(X, T)
    assert np.abs(g[20:724]).max() <= 1e-15  # W1, b1: no slope
    net.close()


@pytest.mark.parametrize("z", [float("nan"), float("-inf"), float("inf")])
def test_non_finite_arguments_show(z):
    net = sgs.MLP(_net(z, 1.0))
    y = net.forward(torch.zeros((10, 5), device="cuda"))
    assert not torch.isfinite(y).any()
    net.close()
