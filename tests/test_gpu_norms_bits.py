"""complex64 state norms keep FP64 accuracy.  The squares of FP32 values are exact
in FP64 and math.fsum adds them exactly.  An unbiased FP64 sum of this block
structure (at most 300 groups a lane, 256 lanes, a few blocks) stays within 2.5e-16
of that (rms over states), a sum that keeps 48 bits is off by 7e-16 whatever the
size: the bound lies between."""
import math

import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("packet", [False, True])
@pytest.mark.parametrize("n,S", [((5, 5, 5), 24), ((12, 12, 12), 8), ((23, 19, 17), 33), ((31, 32, 30), 16), ((31, 32, 30), 64)])
def test_norms_keep_fp64_bits(n, S, packet):
    h = 0.5   # a power of two: h^3 rounds nothing
    m = rsg.Mesh(rsg.BOX, n, spacing=h)
    H = rsg.Hamiltonian(m, torch.complex64)
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((m.P, rsg.padded_ld(S, torch.complex64)), dtype=torch.complex64, device="cuda", generator=g)
    if packet:
        x *= torch.exp(-torch.linspace(-4, 4, m.P, device="cuda") ** 2)[:, None]
    v = torch.view_as_real(x[:, :S]).double().cpu().numpy()
    want = np.array([math.fsum((v[:, s] ** 2).ravel()) for s in range(S)]) * h ** 3
    err = np.sqrt(np.mean((H.norms(x, S=S) / want - 1) ** 2))
    assert err < 4e-16, err
