"""complex64 Cholesky-QR of states that are correlated over thousands of runs of
the Gram sums, at scales whose squares and sums over many points pass the
largest FP32 number (at 4e18 after three runs of 8 points), and far below one,
against a 64-bit Cholesky-QR.  The common part gives the block a condition
number below 20, so FP32 rounding of the block and the update leaves at most 20
u sqrt(S) = 1e-5; the bound is the library's 2e-5."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e18, 4e18, 1e-15])
@pytest.mark.parametrize("S", [2, 8, 24, 70])
def test_correlated_states(S, scale):
    h = 0.3
    m = rsg.Mesh(rsg.BOX, (45, 43, 41), spacing=h)
    H = rsg.Hamiltonian(m, torch.complex64)
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64, device="cuda", generator=g)
    c = torch.randn((m.P, 1), dtype=torch.complex64, device="cuda", generator=g)
    x = (0.5 * x + c / c.abs()) * scale
    y = x[:, :S].to(torch.complex128) / scale
    G = y.conj().T @ y * h ** 3
    want = torch.linalg.solve_triangular(torch.linalg.cholesky(G).conj(), y.T, upper=False).T
    n2 = H.orthonormalize(x, S=S)
    assert np.abs(n2 / (G.diagonal().real.cpu().numpy() * scale ** 2) - 1).max() < 1e-12
    got = x[:, :S].to(torch.complex128)
    err = ((got - want).abs().amax(0) / want.abs().amax(0)).max().item()
    assert err < 2e-5, err
