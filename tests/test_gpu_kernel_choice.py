"""The complex64 kernel choice: on meshes where the default configuration takes
short column segments, narrow chunks or the plain kernel, the result equals
that of the plain kernel to the library's complex64 tolerance (2e-5 of the
largest value per state), with projectors, a field and complex scaling."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _ham(shape, n, scaled, atoms, seed):
    m = rsg.Mesh(rsg.SPHERE, radius=n, spacing=0.2) if shape == "sphere" else rsg.Mesh(rsg.BOX, n, spacing=0.2)
    H = rsg.Hamiltonian(m, torch.complex64)
    r = np.random.default_rng(seed)
    V = r.uniform(-2, 1, m.P)
    if scaled:
        H.set_complex_scaling(0.3, V.astype(np.complex128))
        return m, H
    H.set_potential(V)
    if atoms:
        half = 0.5 * np.ptp(m.xyz, axis=0)
        H.set_projectors(r.uniform(-0.6, 0.6, (atoms, 3)) * half, np.full(atoms, 1.1), np.full(atoms, 1, np.int32),
                         np.full(atoms, 0.3), [np.diag(r.uniform(-1, 1, 4)) for _ in range(atoms)])
    H.set_field(0.02, (0.6, -0.3, 0.7))
    return m, H


@pytest.mark.parametrize("scaled,atoms", [(False, 0), (False, 3), (True, 0)])
@pytest.mark.parametrize("shape,n,S", [("box", (24, 24, 24), 16), ("box", (48, 47, 49), 16), ("box", (96, 33, 96), 4),
                                       ("box", (33, 31, 32), 64), ("box", (131, 29, 57), 10), ("sphere", 7.0, 13),
                                       ("sphere", 9.0, 2), ("box", (200, 7, 5), 40)])
def test_default_choice_matches_plain_kernel(scaled, atoms, shape, n, S):
    m, H = _ham(shape, n, scaled, atoms, S)
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64, device="cuda", generator=g)
    y = H.apply(x, S=S)
    t = H.taylor(x, 0.004, S=S)
    H.set_option("kernel", 1)
    for got, ref in ((y, H.apply(x, S=S)), (t, H.taylor(x, 0.004, S=S))):
        err = ((got - ref)[:, :S].abs().amax(0) / ref[:, :S].abs().amax(0)).max().item()
        assert err < 2e-5, err
