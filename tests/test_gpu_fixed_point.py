"""The FP64 form's line transforms run on 64-bit fixed point with one scale per line: their accuracy
against extended precision, their range, and what non-finite values and zeros become.

Tolerance of the 3D transforms: each of the three passes rounds its result to 53 bits and adds the
fixed-point part, together below 2^-53 of the line's norm, so 3 x 2^-53 relative L2 (a 1024-point
line would still keep this)."""

import numpy as np
import pytest
import scipy.fft as sf

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver  # noqa: E402
from paper_1602_03638_gb300._lib import DNS_ERR_NONFINITE  # noqa: E402,F401

pytestmark = pytest.mark.gpu

LD = np.longdouble
TOL = 3 * 2.0 ** -53


def _bits16(x):
    m, e = np.frexp(x)
    return np.ldexp(np.round(m * 2.0 ** 16), e - 16)


def _factors(N, kind, rng):
    """Hermitian 1D spectra of 16-bit numbers: products of three are exact in FP64."""
    out = []
    for _ in range(3):
        k = np.fft.fftfreq(N, 1.0 / N)
        env = {"white": 1.0, "gauss": np.exp(-(k / 3.0) ** 2), "power": (1.0 + np.abs(k)) ** -1.7}[kind]
        z = (rng.standard_normal(N) + 1j * rng.standard_normal(N)) * env
        z = _bits16(z.real) + 1j * _bits16(z.imag)
        z = np.where(np.arange(N) <= N // 2, z, np.conj(z[(-np.arange(N)) % N]))
        z[0] = z[0].real
        z[N // 2] = 0
        out.append(z)
    return out


def _ld(z):
    return z.real.astype(LD) + 1j * z.imag.astype(LD)


def _outer(a, b, c):
    return a[:, None, None] * b[None, :, None] * c[None, None, :]


@pytest.mark.parametrize("kind", ["white", "gauss", "power"])
@pytest.mark.parametrize("N", [8, 12, 16, 24, 48, 64, 96, 128])
def test_transforms_against_extended_precision(N, kind):
    rng = np.random.default_rng(N)
    h = N // 2 + 1
    f = [_factors(N, kind, rng) for _ in range(3)]
    with Solver(N, 0.01, 0.01, "f64") as s:
        spec = torch.from_numpy(np.stack([_outer(a, b, c[:h]) for a, b, c in f])).cuda()
        phys = torch.empty(s.phys_shape, dtype=torch.float64, device="cuda")
        s.transform_c2r(spec, phys)
        torch.cuda.synchronize()
        ref = np.stack([_outer(*[sf.ifft(_ld(v)).real for v in c]) for c in f])
        got = phys.cpu().numpy().astype(LD)
        assert float(np.sqrt(((got - ref) ** 2).sum() / (ref ** 2).sum())) <= TOL
        mesh = [[_bits16(np.fft.ifft(v).real) for v in c] for c in f]
        s.transform_r2c(torch.from_numpy(np.stack([_outer(*c) for c in mesh])).cuda(), spec)
        torch.cuda.synchronize()
        lines = [[sf.fft(v.astype(LD)) for v in c] for c in mesh]
        for c in lines:
            for v in c:
                v[N // 2] = 0
        ref = np.stack([_outer(a, b, c[:h]) for a, b, c in lines])
        got = _ld(spec.cpu().numpy())
        # a Gaussian's sums cancel: its error is one of the mesh values' norm (Parseval: N^(3/2) times)
        norm = np.sqrt(N ** 3 * sum((_outer(*c) ** 2).sum() for c in mesh) / 2)
        assert float(np.sqrt((np.abs(got - ref) ** 2).sum()) / norm) <= TOL


@pytest.mark.parametrize("N", [16, 48, 128])
def test_power_of_two_scales_every_bit(N):
    g = torch.Generator(device="cuda").manual_seed(1)
    with Solver(N, 0.01, 0.01, "f64") as s:
        u = torch.randn(s.phys_shape, generator=g, dtype=torch.float64, device="cuda")
        out = []
        for e in (0, 600, -600):
            spec = torch.empty(s.spec_shape, dtype=torch.complex128, device="cuda")
            back = torch.empty_like(u)
            s.transform_r2c(u * 2.0 ** e, spec)
            s.transform_c2r(spec, back)
            torch.cuda.synchronize()
            out.append((spec * 2.0 ** -e, back * 2.0 ** -e))
        for spec, back in out[1:]:
            assert torch.equal(torch.view_as_real(spec), torch.view_as_real(out[0][0])) and torch.equal(back, out[0][1])


@pytest.mark.parametrize("N", [12, 64])
def test_zeros_stay_zero_and_non_finite_values_spread(N):
    with Solver(N, 0.01, 0.01, "f64") as s:
        u = torch.zeros(s.phys_shape, dtype=torch.float64, device="cuda")
        spec = torch.empty(s.spec_shape, dtype=torch.complex128, device="cuda")
        s.transform_r2c(u, spec)
        torch.cuda.synchronize()
        assert not torch.view_as_real(spec).any()
        for bad in (float("nan"), float("inf")):
            u.zero_()
            u[1, 2, 3, 1] = bad
            s.transform_r2c(u, spec)
            torch.cuda.synchronize()
            assert torch.isnan(spec[1].real).any() and not torch.view_as_real(spec[0]).any()
            s.set_state(u)
            s.step(1)
            with pytest.raises(RuntimeError):
                s.diagnostics()
