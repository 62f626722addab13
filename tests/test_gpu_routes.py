"""Which stencil ran, and its result against FP64: the complex64 choice by size
(kernel and planes per segment asserted) against the complex128 staged kernel on
the same rounded inputs, to the library's 2e-5; the complex128 integer sums with
1, 5 and 32 planes per block forced on thin, wide and small meshes against the
staged FP64 kernel (another summation order), to 1e-12 of the largest value."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _hams(shape, n, atoms, scaled, seed, dtypes):
    m = rsg.Mesh(rsg.SPHERE, radius=n, spacing=0.2) if shape == "sphere" else rsg.Mesh(rsg.BOX, n, spacing=0.2)
    r = np.random.default_rng(seed)
    V = r.uniform(-2, 1, m.P).astype(np.float32).astype(np.float64)
    half = 0.5 * np.ptp(m.xyz, axis=0)
    at = (r.uniform(-0.6, 0.6, (atoms, 3)) * half, np.full(atoms, 1.1), np.full(atoms, 1, np.int32), np.full(atoms, 0.3),
          [np.diag(r.uniform(-1, 1, 4)) for _ in range(atoms)])
    out = []
    for dt in dtypes:
        H = rsg.Hamiltonian(m, dt)
        if scaled:
            H.set_complex_scaling(0.3, V.astype(np.complex128))
        else:
            H.set_potential(V)
            H.set_field(0.02, (0.6, -0.3, 0.7))
            if atoms:
                H.set_projectors(*at)
        out.append(H)
    return m, out


def _close(got, ref, tol):
    err = ((got.to(torch.complex128) - ref).abs().amax(0) / ref.abs().amax(0)).max().item()
    assert err < tol, err


@pytest.mark.parametrize("shape,n,S,atoms,scaled,kernel,zseg", [
    ("box", (24, 24, 24), 16, 3, False, 1, 0), ("box", (200, 7, 5), 40, 0, False, 1, 0), ("sphere", 9.0, 2, 3, False, 1, 0),
    ("box", (97, 95, 60), 1, 0, False, 1, 0), ("box", (24, 24, 24), 16, 0, True, 6, 0),
    ("box", (48, 47, 49), 16, 3, False, 7, 12), ("box", (33, 31, 32), 64, 0, False, 7, 16),
    ("box", (131, 29, 57), 10, 3, False, 7, 24), ("sphere", 7.0, 13, 3, False, 7, 24), ("box", (48, 47, 49), 16, 0, True, 7, 12),
    ("box", (96, 33, 96), 4, 0, False, 5, 12), ("box", (140, 33, 96), 6, 3, False, 5, 24),
    ("sphere", 10.0, 5, 3, False, 5, 32), ("box", (70, 70, 200), 8, 0, False, 5, 48), ("box", (97, 95, 60), 1, 0, True, 5, 12)])
def test_complex64_choice(shape, n, S, atoms, scaled, kernel, zseg):
    m, (H, D) = _hams(shape, n, atoms, scaled, S, (torch.complex64, torch.complex128))
    if not scaled:
        D.set_option("kernel", 0)
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64, device="cuda", generator=g)
    d = x[:, :S].to(torch.complex128).contiguous()
    for got, ref in ((H.apply(x, S=S), D.apply(d)), (H.taylor(x, 0.004, S=S), D.taylor(d, 0.004))):
        assert (H.get_option("last_kernel"), H.get_option("last_zseg")) == (kernel, zseg)
        assert D.get_option("last_kernel") == (6 if scaled else 0)
        _close(got[:, :S], ref, 2e-5)


@pytest.mark.parametrize("planes", [1, 5, 32])
@pytest.mark.parametrize("shape,n,S,atoms", [("box", (17, 16, 9), 200, 2), ("box", (300, 5, 3), 130, 0), ("box", (24, 24, 24), 1, 1),
                                             ("box", (33, 20, 70), 3, 2), ("box", (1, 1, 90), 17, 0), ("sphere", 4.0, 5, 2)])
def test_integer_sums(shape, n, S, atoms, planes):
    m, (H,) = _hams(shape, n, atoms, False, S, (torch.complex128,))
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, S), dtype=torch.complex128, device="cuda", generator=g)
    H.set_option("sum_planes", planes)
    got = H.apply(x), H.taylor(x, 0.004)
    assert (H.get_option("last_kernel"), H.get_option("last_sum_planes")) == (1, planes)
    H.set_option("kernel", 0)
    for a, b in zip(got, (H.apply(x), H.taylor(x, 0.004))):
        assert H.get_option("last_kernel") == 0
        _close(a, b, 1e-12)


def test_default_integer_sums():
    """By size: FP64 sums on the smallest meshes, integer sums on larger ones;
    image walls add in FP64."""
    for n, S, want in ((9, 1, False), (16, 1, False), (61, 8, True), (64, 1, True)):
        m, (H,) = _hams("box", (n,) * 3, 0, False, 0, (torch.complex128,))
        x = torch.zeros((m.P, S), dtype=torch.complex128, device="cuda")
        H.apply(x)
        assert (H.get_option("last_sum_planes") > 0) == want, (n, S)
    m.set_boundary(rsg.BC_ODD)
    H.apply(x)
    assert H.get_option("last_sum_planes") == 0
