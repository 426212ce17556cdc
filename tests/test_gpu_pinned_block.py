"""Solvers and networks share one block of pinned memory for their read-backs: each keeps its own piece, whatever
the order in which they come and go, past what the block holds, and from several threads."""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver, sgs  # noqa: E402

pytestmark = pytest.mark.gpu


def _check_solver(s, inside):
    uh = np.zeros(s.spec_shape, dtype=np.complex64)
    uh[0, 0, 1, 1] = 1
    if not inside:
        uh[0, 0, 3, 0] = 1  # outside the 2/3 box of 8 points
    s.set_state_spectral(uh)
    assert s.get_option("rows_vanish") == float(inside)


def _check_net(net, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X, T = torch.randn((10, 200), generator=g, device="cuda"), torch.randn((6, 200), generator=g, device="cuda")
    a = net.loss_grad(X, T)
    b = net.loss_grad(X, T)
    assert a[0] == b[0] > 0 and np.array_equal(a[1], b[1]) and a[1].any()


def _some(seed, nets, solvers):
    rng = np.random.default_rng(seed)
    alive = []
    for i in rng.permutation(nets + solvers):
        alive.append(sgs.MLP(seed=int(i)) if i < nets else Solver(8, 0.01, 0.01, "f32"))
        for k in rng.permutation(len(alive))[:3]:
            o = alive[k]
            if isinstance(o, Solver):
                _check_solver(o, bool(rng.integers(2)))
            else:
                _check_net(o, int(k))
        if len(alive) > 12 and rng.random() < 0.5:
            alive.pop(int(rng.integers(len(alive)))).close()
    for k in rng.permutation(len(alive)):
        alive[k].close()


def test_pieces_come_and_go():
    _some(0, 12, 20)
    _some(1, 3, 3)


def test_from_several_threads():
    errors = []

    def work(seed):
        try:
            _some(seed, 3, 8)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
