"""1 / |k|^2 of the FP64 projection (Newton's iteration from the hardware's approximation) equals the rounded
quotient on every wavenumber of the box, over box lengths that spread |k|^2 from 2^-60 to 2^60. At rest and with
a force f the right-hand side is f - k (k . f) / |k|^2: with f = (1, 0, 0) and k_x = 1 its second component is -k_y / |k|^2,
formed from the reciprocal by one product. Box lengths are powers of two, so |k|^2 is exact.

Why the iteration rounds correctly: from an approximation of 20 bits, one step leaves 2^-40, so that the last, r + r (1 - x r) with
1 - x r by a fused product, is the exact quotient but for 2^-80 before its one rounding."""

import math

import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ey,ez", [(0, 0), (-3, 2), (9, 0), (0, -9), (-30, -30), (22, 22)])
@pytest.mark.parametrize("N", [16, 96, 256])
def test_reciprocal_is_the_rounded_quotient(N, ey, ez):
    lengths = (2 * math.pi, 2 * math.pi * 2.0 ** -ey, 2 * math.pi * 2.0 ** -ez)
    with Solver(N, 1e-300, 1e-3, "f64", lengths=lengths) as s:
        f = torch.zeros(s.spec_shape, dtype=torch.complex128, device="cuda")
        s.set_state_spectral(f)
        f[0] = 1
        s.set_forcing(f)
        out = torch.empty_like(f)
        s.rhs(out)
        torch.cuda.synchronize()
    kc = (N + 2) // 3
    ky = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)[:, None]
    kz = torch.arange(kc, device="cuda", dtype=torch.float64)[None, :]
    kept = 3 * ky[:, 0].abs() < N
    ky, kz = ky[kept] * 2.0 ** ey, kz * 2.0 ** ez
    k2 = 1.0 + ky * ky + kz * kz
    assert torch.equal(out[1, 1, kept][:, :kc].real, -ky * (1.0 / k2))
    assert not out[1, 1, kept][:, :kc].imag.any()
