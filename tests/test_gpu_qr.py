"""Cholesky-QR, norms and the FP64 Gram sums at the edges of their tiles.

State counts around the column tiles (8, 16, 32, 64, 128 columns), point
counts that leave remainders, against a 64-bit Cholesky-QR in torch.  The
blocks are noise on at least four points per state, whose Gram matrix has a
condition number below 40, so rounding of relative size u in the block leaves
at most about 40 u sqrt(S) in the result: 1e-12 in complex128 and the
library's 2e-5 in complex64.
"""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _reference(x, h):
    G = x.conj().T @ x * h ** 3
    L = torch.linalg.cholesky(G)
    return torch.linalg.solve_triangular(L.conj(), x.T, upper=False).T, G.diagonal().real.cpu().numpy()


@pytest.mark.parametrize("dtype,tol", [(torch.complex64, 2e-5), (torch.complex128, 1e-12)])
@pytest.mark.parametrize("n,S", [((9, 9, 9), 1), ((7, 11, 5), 2), ((13, 5, 3), 3), ((13, 11, 9), 8), ((13, 11, 9), 9),
                                 ((13, 11, 9), 15), ((13, 11, 9), 16), ((17, 13, 9), 17), ((17, 13, 9), 31),
                                 ((17, 13, 9), 32), ((17, 13, 9), 33), ((19, 17, 13), 63), ((19, 17, 13), 64),
                                 ((19, 17, 13), 65), ((23, 19, 17), 127), ((23, 19, 17), 128), ((23, 19, 17), 129),
                                 ((23, 19, 17), 170), ((23, 23, 19), 257), ((25, 23, 19), 353)])
def test_orthonormalize_edges(dtype, tol, n, S):
    h = 0.3
    m = rsg.Mesh(rsg.BOX, n, spacing=h)
    H = rsg.Hamiltonian(m, dtype)
    g = torch.Generator(device="cuda").manual_seed(7 * S + n[0])
    x = torch.randn((m.P, rsg.padded_ld(S, dtype)), dtype=dtype, device="cuda", generator=g)
    ref, n2 = _reference(x[:, :S].to(torch.complex128), h)
    got = H.orthonormalize(x, S=S)
    assert np.abs(got / n2 - 1).max() < 1e-12
    y = x[:, :S].to(torch.complex128)
    err = ((y - ref).abs().amax(0) / ref.abs().amax(0)).max().item()
    assert err < tol, err


@pytest.mark.parametrize("S", [1, 3, 64, 70])
def test_norms_outside_single_precision_squares(S):
    """Squares that FP32 cannot hold (1e-25, 1e25) and zero states."""
    m = rsg.Mesh(rsg.BOX, (31, 13, 11), spacing=0.3)
    H = rsg.Hamiltonian(m, torch.complex64)
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64, device="cuda", generator=g)
    x *= torch.tensor([1.0, 1e-25, 1e25, 0.0, 1e-12], device="cuda")[torch.arange(x.shape[1], device="cuda") % 5]
    x[: m.P // 3] *= 1e-9
    ref = (x[:, :S].to(torch.complex128).abs() ** 2).sum(0).cpu().numpy() * m.h ** 3
    got = H.norms(x, S=S)
    assert np.all(np.abs(got - ref) <= 1e-12 * ref)
