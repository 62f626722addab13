"""The complex64 choice by size belongs to the mesh: every Hamiltonian on it
takes the same one, and an application that failed half way leaves none behind."""
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _ham(m):
    H = rsg.Hamiltonian(m, torch.complex64)
    H.set_potential(torch.zeros(m.P, dtype=torch.float64))
    x = torch.randn((m.P, 16), dtype=torch.complex64, device="cuda")
    H.orthonormalize(x.clone())   # the status word exists from here on
    return H, x


def test_failed_table_allocation_leaves_no_choice():
    m = rsg.Mesh(rsg.BOX, (48, 47, 49), spacing=0.2)
    H, x = _ham(m)
    want = H.apply(x)
    choice = H.get_option("last_kernel"), H.get_option("last_zseg")
    assert choice == (7, 12)
    m = rsg.Mesh(rsg.BOX, (48, 47, 49), spacing=0.2)
    D = rsg.Hamiltonian(m, torch.complex128)
    D.set_potential(torch.zeros(m.P, dtype=torch.float64))
    D.apply(x.to(torch.complex128))   # the row table exists from here on
    H, _ = _ham(m)
    rsg.rsg.load().rsg_debug_fail_allocations(1)
    try:
        with pytest.raises(rsg.RSGError, match="tile upload"):
            H.apply(x)
    finally:
        rsg.rsg.load().rsg_debug_fail_allocations(0)
    for h in (H, _ham(m)[0]):
        got = h.apply(x)
        assert (h.get_option("last_kernel"), h.get_option("last_zseg")) == choice
        assert torch.equal(got, want)
