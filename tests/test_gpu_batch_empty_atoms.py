"""Batches whose systems hold atoms without a mesh point in their sphere (first,
last, between others, all of them): the step equals single-system propagation
(the library's 2e-5 for batches with projectors)."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu

OUT = (40.0, 0.0, 0.0)   # outside every mesh here
IN = [(0.3, -0.2, 0.1), (-0.4, 0.3, -0.2)]


def _system(n, S, centres, lmax, seed):
    m = rsg.Mesh(rsg.CUBE, n, spacing=0.25)
    H = rsg.Hamiltonian(m, torch.complex64)
    r = np.random.default_rng(seed)
    H.set_potential(r.uniform(-2, 1, m.P))
    na, k = len(centres), (lmax + 1) ** 2
    H.set_projectors(np.array(centres), np.full(na, 1.0), np.full(na, lmax, np.int32), np.full(na, 0.3),
                     [np.diag(r.uniform(-1, 1, k)) for _ in range(na)])
    x = torch.zeros((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64)
    x[:, :S] = torch.from_numpy(r.standard_normal((m.P, S)) + 1j * r.standard_normal((m.P, S)))
    return H, S, x.cuda()


@pytest.mark.parametrize("persistent", [1, 0])
def test_atoms_without_points(persistent):
    lists = [[OUT, IN[0]], [IN[0], OUT], [OUT], [OUT, OUT], [IN[0], OUT, IN[1]], [OUT, IN[1], OUT, IN[0], OUT]]
    sy = [_system(9 + 2 * i, 1 + 2 * i, c, 1, i) for i, c in enumerate(lists)]
    batch = rsg.Batch([H for H, _, _ in sy], [S for _, S, _ in sy])
    batch.set_option("persistent", persistent)
    xs = [x.clone() for _, _, x in sy]
    batch.propagate(xs, 2, 0.01, scheme=rsg.ETRS)
    assert batch.get_option("batched") == 1
    for (H, S, x), got in zip(sy, xs):
        H.propagate(x, 2, 0.01, scheme=rsg.ETRS, S=S)
        d, ref = (got - x)[:, :S], x[:, :S]
        assert (d.abs().amax(0) / ref.abs().amax(0)).max().item() < 2e-5
