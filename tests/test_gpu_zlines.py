"""The FP32 z-pass, small grids and 256- to 1024-point lines, inside the right-hand side, against u x omega, its projection
and the viscous term in plain FP64 transforms, with states inside and outside the 2/3 box (planes read as zeros, and
all planes). Tolerance: three FP32 inverse and three forward passes keep 1e-6 relative L2 (the bound of the y-pass
test, for three); six and a product whose projection halves it at most: 4e-6."""

import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver  # noqa: E402

pytestmark = pytest.mark.gpu


def _k(shape):
    f = [torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64) for n in shape]
    f[2] = torch.arange(shape[2] // 2 + 1, device="cuda", dtype=torch.float64)
    return f[0][:, None, None], f[1][None, :, None], f[2][None, None, :]


@pytest.mark.parametrize("shape", [(n, n, n) for n in (8, 12, 16, 24, 32, 48, 64, 96, 128)] + [(256, 256, 256), (512, 512, 512), (1024, 512, 256), (1024, 1024, 1024)])
@pytest.mark.parametrize("full", [True, False])
def test_right_hand_side(shape, full):
    nu = 1e-6  # the viscous term small beside the products
    k = _k(shape)
    kept = [3 * q.abs() < n for q, n in zip(k, shape)]
    box = kept[0] & kept[1] & kept[2]
    g = torch.Generator(device="cuda").manual_seed(sum(shape) + full)
    uh = torch.empty((3, *shape[:2], shape[2] // 2 + 1), dtype=torch.complex64, device="cuda")
    for c in range(3):
        z = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda"))
        if not full:
            z *= box
        for q, n in zip(k, shape):  # no coefficients at the half-sampling frequency
            z *= q.abs() < n / 2
        uh[c] = z
    with Solver(shape, nu, 1e-3, "f32") as s:
        s.set_state_spectral(uh)
        assert s.get_option("rows_vanish") == (0.0 if full else 1.0)
        out = torch.empty_like(uh)
        s.rhs(out)
        torch.cuda.synchronize()
    torch.cuda.empty_cache()
    phys = lambda z: torch.fft.irfftn(z, s=shape)
    u = [phys(uh[c].to(torch.complex128)) for c in range(3)]
    kp = lambda i, c: 1j * k[i] * uh[c].to(torch.complex128)
    w = [phys(kp(1, 2) - kp(2, 1)), phys(kp(2, 0) - kp(0, 2)), phys(kp(0, 1) - kp(1, 0))]
    n = []
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        n.append(torch.fft.rfftn(u[a] * w[b] - u[b] * w[a]) * box)
    del u, w
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    p = (k[0] * n[0] + k[1] * n[1] + k[2] * n[2]) / k2.clamp(min=1)
    for c in range(3):
        ref = n[c] - k[c] * p - nu * k2 * uh[c]
        assert (out[c] - ref).norm() <= 4e-6 * ref.norm()
