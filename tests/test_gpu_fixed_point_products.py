"""u x omega and u_i u_j of the FP64 form keep FP64's accuracy in every component: a weak third
component beside strong ones, and broad spectra (whose L1 norm is many times the values) on long lines.

Tolerance per component: u, omega and the transform back each within 3 x 2^-53 (the bound of the
transforms' own test), the products one rounding; as much again for the plain FP64 transforms of the
reference: 20 x 2^-53. The filtered products against the separate calls, which round
the same products in FP64: 8 last bits of each product's own largest coefficient."""

import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver, _lib, sgs  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 20 * 2.0 ** -53


def _k(n):
    f = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    return f[:, None, None], f[None, :, None], torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)[None, None, :]


def _solenoidal(u, n):
    """Coefficients of the mesh field u without the half-sampling frequency and the divergence."""
    k = _k(n)
    uh = torch.stack([torch.fft.rfftn(c) for c in u])
    for q in k:
        uh *= q.abs() < n / 2
    k2 = (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).clamp(min=1)
    d = (k[0] * uh[0] + k[1] * uh[1] + k[2] * uh[2]) / k2
    for c in range(3):
        uh[c] -= k[c] * d
    return uh


def _plane(n, weak):
    """Two strong velocities in the plane and a third of size `weak`, all constant along z."""
    g = torch.Generator(device="cuda").manual_seed(n)
    u = torch.randn((3, n, n), generator=g, device="cuda", dtype=torch.float64)[..., None].expand(3, n, n, n).clone()
    u[2] *= weak
    uh = _solenoidal(u, n)
    uh[..., 1:] = 0
    return uh


def _errors(uh, n):
    """Per component, the right-hand side against u x omega, masked and projected, in plain FP64."""
    with Solver(n, 1e-30, 1e-3, "f64") as s:
        s.set_state_spectral(uh)
        out = torch.empty_like(uh)
        s.rhs(out)
        torch.cuda.synchronize()
    k = _k(n)
    box = (3 * k[0].abs() < n) & (3 * k[1].abs() < n) & (3 * k[2] < n)
    phys = lambda z: torch.fft.irfftn(z, s=(n, n, n))
    u = [phys(uh[c]) for c in range(3)]
    w = [phys(1j * (k[(c + 1) % 3] * uh[(c + 2) % 3] - k[(c + 2) % 3] * uh[(c + 1) % 3])) for c in range(3)]
    ref = torch.stack([torch.fft.rfftn(u[(c + 1) % 3] * w[(c + 2) % 3] - u[(c + 2) % 3] * w[(c + 1) % 3]) * box for c in range(3)])
    del u, w
    p = (k[0] * ref[0] + k[1] * ref[1] + k[2] * ref[2]) / (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).clamp(min=1)
    for c in range(3):
        ref[c] -= k[c] * p
    return [float((out[c] - ref[c]).norm() / ref[c].norm()) for c in range(3)]


@pytest.mark.parametrize("weak", [1e-3, 1e-6, 1e-12, 1e-20, 1e-60])
@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 256])
def test_a_weak_component_keeps_its_bits(n, weak):
    assert max(_errors(_plane(n, weak), n)) <= TOL


@pytest.mark.parametrize("n", [16, 48, 64, 256, 512])
def test_every_mode_occupied(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    u = torch.randn((3, n, n, n), generator=g, device="cuda", dtype=torch.float64)
    uh = _solenoidal(u, n)
    del u
    assert max(_errors(uh, n)) <= TOL


@pytest.mark.parametrize("weak", [1e-6, 1e-20])
@pytest.mark.parametrize("n,nc", [(12, 12), (16, 6), (48, 24), (128, 64), (256, 62)])
def test_filtered_products_of_a_weak_component(n, nc, weak):
    with Solver(n, 0.01, 0.01, "f64") as s:
        sgs.on_torch_stream(s)
        s.set_state_spectral(_plane(n, weak))
        u = torch.empty(s.phys_shape, dtype=torch.float64, device="cuda")
        s.get_state(u)
        ph = sgs.r2c(s, sgs.pointwise_products(u, "f64"))
        ref = torch.cat([sgs.spectral_filter(ph[i:i + 3].contiguous(), nc, "f64") for i in (0, 3)])
        bar, p = torch.empty((3,) + ref.shape[1:], dtype=ref.dtype, device="cuda"), torch.empty_like(ref)
        _lib.check(_lib.lib().dns_filtered_products(s.handle, nc, sgs._p(bar), sgs._p(p)), "dns_filtered_products")
        torch.cuda.synchronize()
    for c in range(6):
        assert (p[c] - ref[c]).abs().max() <= 8 * 2.0 ** -52 * ref[c].abs().max(), c


@pytest.mark.parametrize("n", [8, 12, 16, 48, 64, 128])
def test_a_product_with_a_zero_line_takes_no_bits(n):
    """u = (0, e cos x, A sin x + e sin y): the third component of u x omega is u_x omega_y - u_y omega_x = 0 A - e^2
    cos x cos y, which stays whatever A is (at kz = 0 the projection leaves that component alone)."""
    A, e = 1e150, 1e-100
    uh = torch.zeros((3, n, n, n // 2 + 1), dtype=torch.complex128, device="cuda")
    uh[1, 1, 0, 0] = uh[1, -1, 0, 0] = 0.5 * n ** 3 * e
    uh[2, 1, 0, 0], uh[2, -1, 0, 0] = -0.5j * n ** 3 * A, 0.5j * n ** 3 * A
    uh[2, 0, 1, 0], uh[2, 0, -1, 0] = -0.5j * n ** 3 * e, 0.5j * n ** 3 * e
    with Solver(n, 1e-300, 1e-3, "f64") as s:
        s.set_state_spectral(uh)
        out = torch.empty_like(uh)
        s.rhs(out)
        torch.cuda.synchronize()
    want = -0.25 * n ** 3 * e * e
    for x, y in ((1, 1), (1, -1), (-1, 1), (-1, -1)):
        assert abs(out[2, x, y, 0].item() - want) <= TOL * abs(want), (x, y)
