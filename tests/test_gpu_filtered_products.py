"""dns_filtered_products (products formed inside the z-pass, only the modes of the coarse grid carried
on) against the separate calls it replaces: read the state back, multiply on the mesh, transform,
filter. The transforms are the same passes, so both agree to the rounding of the working
precision: a last bit of the largest coefficient per pass, held to 8 of them."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1602_03638_gb300 import Solver, inputs, sgs  # noqa: E402
from paper_1602_03638_gb300 import _lib  # noqa: E402

pytestmark = pytest.mark.gpu

CDT = {"f32": torch.complex64, "f64": torch.complex128}
RDT = {"f32": torch.float32, "f64": torch.float64}
EPS = {"f32": 2.0 ** -23, "f64": 2.0 ** -52}


def _separate(s, Nc):
    uh = torch.empty(s.spec_shape, dtype=CDT[s.dtype], device="cuda")
    s.get_state_spectral(uh)
    u = torch.empty(s.phys_shape, dtype=RDT[s.dtype], device="cuda")
    s.get_state(u)
    p = sgs.pointwise_products(u, s.dtype)
    ph = sgs.r2c(s, p)
    return sgs.spectral_filter(uh, Nc, s.dtype), torch.cat([sgs.spectral_filter(ph[i:i + 3].contiguous(), Nc, s.dtype) for i in (0, 3)])


@pytest.mark.parametrize("full", [False, True])  # inside the 2/3 box (skipped rows), and every mode occupied
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,Nc", [(8, 2), (12, 12), (16, 6), (48, 24), (64, 64), (96, 34), (128, 64), (256, 62)])
def test_equals_the_separate_calls(N, Nc, dtype, full):
    with Solver(N, 0.01, 0.01, dtype) as s:
        sgs.on_torch_stream(s)
        if full:
            g = torch.Generator(device="cuda").manual_seed(N)
            s.set_state(torch.randn(s.phys_shape, generator=g, device="cuda", dtype=RDT[dtype]))
        else:
            s.set_state_spectral(inputs.isotropic_spectral(N, seed=3, k0=max(1.0, N / 8), device="cuda").to(CDT[dtype]))
        before = s.get_state_spectral()
        ref_u, ref_p = _separate(s, Nc)
        u = torch.empty_like(ref_u)
        p = torch.empty_like(ref_p)
        _lib.check(_lib.lib().dns_filtered_products(s.handle, Nc, sgs._p(u), sgs._p(p)), "dns_filtered_products")
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(u), torch.view_as_real(ref_u))
        assert (p - ref_p).abs().max() <= 8 * EPS[dtype] * ref_p.abs().max()
        assert np.array_equal(s.get_state_spectral(), before)
        s.step(1)  # the work buffers are primed again
        stepped = s.get_state_spectral()
        s.set_state_spectral(before)
        s.step(1)
        assert np.array_equal(s.get_state_spectral(), stepped)


def test_arguments_are_checked():
    buf = torch.empty(4096, dtype=torch.complex64, device="cuda")
    L = _lib.lib()
    with Solver(16, 0.01, 0.01, "f32") as s:
        for Nc in (0, 3, 18):
            assert L.dns_filtered_products(s.handle, Nc, sgs._p(buf), sgs._p(buf)) == _lib.DNS_ERR_ARG
        assert L.dns_filtered_products(s.handle, 8, None, sgs._p(buf)) == _lib.DNS_ERR_ARG
    with Solver((32, 16, 24), 0.01, 0.01, "f32") as s:
        assert L.dns_filtered_products(s.handle, 8, sgs._p(buf), sgs._p(buf)) == _lib.DNS_ERR_UNSUPPORTED
