"""The FP64 form keeps the range of a double: scaling the input by a power of two scales every bit of
the transforms and of u x omega, down to where results become subnormal and up to where they overflow;
below that they underflow gradually and above they are not finite. (Subnormal results: half of 2^-1074
from the scaling of the reference and from the result each, per pass.)"""

import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver  # noqa: E402

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -1074


def _p2(x, e):
    return x * 2.0 ** (e // 2) * 2.0 ** (e - e // 2)


@pytest.mark.parametrize("N", [8, 12, 16, 48, 64, 128, 512])
def test_transforms_over_the_whole_range(N):
    _transforms((N,) * 3)


def test_long_rows_over_the_whole_range():
    _transforms((1024, 512, 256))  # lines of 1024 points are read twice


def _transforms(shape):
    nx, ny, _ = shape
    g = torch.Generator(device="cuda").manual_seed(nx)
    with Solver(shape, 0.01, 0.01, "f64") as s:
        u = torch.rand(s.phys_shape, generator=g, dtype=torch.float64, device="cuda") + 0.5
        spec = torch.empty(s.spec_shape, dtype=torch.complex128, device="cuda")
        back = torch.empty_like(u)
        s.transform_r2c(u, spec)
        s.transform_c2r(spec, back)
        torch.cuda.synchronize()
        top = int(torch.view_as_real(spec).abs().max().log2().floor())
        small = torch.view_as_real(spec).abs()
        small = int(small[small > 0].min().log2().floor())
        out, phys = torch.empty_like(spec), torch.empty_like(u)
        # to the largest results, and to where the least ones (of the passes between too, smaller by up to N each)
        # are normal yet
        for e in (-1021 - small + nx.bit_length() + ny.bit_length() + 8, -900, 940, 1021 - top):
            s.transform_r2c(_p2(u, e), out)
            assert torch.equal(_p2(torch.view_as_real(out), -e), torch.view_as_real(spec)), e
            s.transform_c2r(out, phys)
            if e > -960:
                assert torch.equal(_p2(phys, -e), back), e
        for e in (-1040, -1070):  # subnormal values on the mesh
            v = _p2(u, e)
            s.transform_r2c(v, out)
            w = _p2(v, 1000)  # the same numbers, normal
            s.transform_r2c(w, spec)
            torch.cuda.synchronize()
            d = _p2(torch.view_as_real(out), 1000) - torch.view_as_real(spec)
            # three passes; a pass adds up N roundings at most
            assert d.abs().max() <= _p2(torch.tensor(TINY, dtype=torch.float64, device="cuda"), 1000) * (1 + nx + nx * ny)
            assert torch.view_as_real(out).abs().max() > 0
        s.transform_r2c(_p2(u, 1023 - top + 3), out)
        assert not torch.isfinite(torch.view_as_real(out)).all()


@pytest.mark.parametrize("N", [8, 12, 16, 48, 64, 128])
def test_products_over_the_whole_range(N):
    g = torch.Generator(device="cuda").manual_seed(N)
    k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64).abs() < N / 2
    uh = torch.stack([torch.fft.rfftn(torch.randn((N,) * 3, generator=g, dtype=torch.float64, device="cuda")) for _ in range(3)])
    uh *= k[:, None, None] & k[None, :, None]
    uh[..., N // 2] = 0
    with Solver(N, 1e-300, 0.01, "f64") as s:
        out = []
        for e in (0, -495, -490, -300, 300, 480):
            s.set_state_spectral(_p2(uh, e))
            r = torch.empty_like(uh)
            s.rhs(r)
            torch.cuda.synchronize()
            out.append(_p2(torch.view_as_real(r), -2 * e))
    for r in out[1:]:
        assert (r - out[0]).norm() <= 1e-15 * out[0].norm()
