"""The complex128 integer neighbour sums are odd: H(-u) = -H(u) in every bit,
whatever the range of the values, and neighbours of opposite signs cancel
exactly (a field that is odd about a point gives zero there)."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _ham(n):
    m = rsg.Mesh(rsg.BOX, n, spacing=0.2)
    H = rsg.Hamiltonian(m, torch.complex128)
    r = np.random.default_rng(5)
    H.set_potential(r.uniform(-2, 1, m.P))
    H.set_option("sum_planes", 8)
    return m, H, r


@pytest.mark.parametrize("spread", [0.0, 3.0, 20.0, 60.0, 900.0])
@pytest.mark.parametrize("S", [1, 4])
def test_odd(S, spread):
    m, H, r = _ham((34, 21, 27))
    u = (r.standard_normal((m.P, S)) + 1j * r.standard_normal((m.P, S))) * np.exp2(r.uniform(-spread, spread, (m.P, S)))
    x = torch.from_numpy(u).cuda()
    a, b = H.apply(x), H.apply(-x)
    assert H.get_option("last_sum_planes") == 8
    assert torch.isfinite(torch.view_as_real(a)).all() and torch.equal(a, -b)


def test_opposite_neighbours_cancel():
    m, H, r = _ham((45, 36, 27))
    u = np.zeros((27, 36, 45), complex)
    centres = [(z, y, x) for z in (4, 13, 22) for y in (4, 13, 22, 31) for x in (4, 13, 22, 31, 40)]
    for z, y, x in centres:   # stars that do not meet, each with its own magnitudes along x, y and z
        for k in range(1, 5):
            a, b, c = (r.standard_normal(3) + 1j * r.standard_normal(3)) * np.exp2(r.uniform(-70, 70, 3))
            u[z, y, x - k], u[z, y, x + k] = a, -a
            u[z, y - k, x], u[z, y + k, x] = -b, b
            u[z - k, y, x], u[z + k, y, x] = c, -c
    got = H.apply(torch.from_numpy(u.reshape(-1, 1)).cuda()).cpu().numpy().reshape(27, 36, 45)
    assert H.get_option("last_sum_planes") == 8
    assert all(got[c] == 0 for c in centres)
