"""The vector updates and bilinear forms of the shifted solve, one iteration:
x = (r.r / r.(H - z) r) r for r = b, formed in 64 bits from the library's own
(H - z) b.  Odd and even state counts, and right-hand sides of 1e-30 and 1e18
(parts outside the range the FP32/FP64 bit conversions take).  complex64 rounds
H b (1e-7 of its largest value) and x: 1e-5 of the largest value, as the sums
r.(H - z) r of the seeded noise cancel to no less than a hundredth."""
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.complex64, 1e-5), (torch.complex128, 1e-12)])
@pytest.mark.parametrize("S", [1, 2, 3, 8])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e18])
def test_one_iteration(dtype, tol, S, scale):
    m = rsg.Mesh(rsg.BOX, (23, 17, 19), spacing=0.3)
    H = rsg.Hamiltonian(m, dtype)
    H.set_potential(torch.linspace(-1, 1, m.P, dtype=torch.float64).cuda())
    g = torch.Generator(device="cuda").manual_seed(S)
    b = torch.randn((m.P, rsg.padded_ld(S, dtype)), dtype=dtype, device="cuda", generator=g)
    b.imag *= 0.2     # r.r is then far from zero
    b *= scale
    z = complex(-1.5, 0.7)
    hb = H.apply(b, S=S).to(torch.complex128)
    x = torch.zeros_like(b)
    H.shifted_solve(b, x, z, max_iter=1, tol=1e-14, S=S)
    r = b[:, :S].to(torch.complex128) / scale
    q = hb[:, :S] / scale - z * r
    ref = ((r * r).sum(0) / (r * q).sum(0)) * r
    got = x[:, :S].to(torch.complex128) / scale
    assert ((got - ref).abs().amax(0) / ref.abs().amax(0)).max().item() < tol
