"""Loss and gradient of the training kernel (tcgen05, tiles of 128 points, blocks that walk several
tiles, partial sums added in order) at the edges of its tiles and grid, against the reference with
the same BF16 roundings. Tolerance: the longest chain of products takes four BF16 roundings
(2^-9 relative each) that fall differently where FP32 sums differ in the last bit; 2e-2 of a
gradient's norm is twice that sum for a single point."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sgs_mlp as sg  # noqa: E402
from paper_1602_03638_gb300 import sgs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 2, 127, 128, 129, 38912, 38913, 80001])
def test_gradient_at_tile_and_grid_edges(P):
    rng = np.random.default_rng(P)
    X = rng.normal(size=(P, 10)).astype(np.float32)
    T = rng.normal(size=(P, 6)).astype(np.float32)
    v = sgs.init_params(3)
    v[660:724] = 0.1 * rng.normal(size=64)
    v[5274:5280] = rng.uniform(0.5, 2.0, size=6)
    net = sgs.MLP(v)
    Xd, Td = (torch.from_numpy(a.T.copy()).cuda() for a in (X, T))
    loss, g = net.loss_grad(Xd, Td)
    lref, gref = sg.loss_and_grads(sg.unflatten(v.astype(np.float64)), X.astype(np.float64), T.astype(np.float64),
                                   round_bf16=True)
    assert abs(loss - lref) < 1e-3 * lref
    gv = sg.unflatten(g.astype(np.float64))
    for name in ("W1", "b1", "W2", "b2", "W3", "b3"):
        assert np.linalg.norm(gv[name] - gref[name]) < 2e-2 * np.linalg.norm(gref[name]), name
    for name in ("in_shift", "in_scale", "out_scale", "out_shift"):
        assert not gv[name].any()
    again = net.loss_grad(Xd, Td)
    assert again[0] == loss and np.array_equal(again[1], g)
    net.close()
