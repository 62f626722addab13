"""The complex64 choice by size belongs to the mesh: every Hamiltonian on it
takes the same one, and an application that failed half way leaves none behind."""
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _ham(m, S=16):
    H = rsg.Hamiltonian(m, torch.complex64)
    H.set_potential(torch.zeros(m.P, dtype=torch.float64))
    x = torch.randn((m.P, S), dtype=torch.complex64, device="cuda")
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


@pytest.mark.parametrize("key,value", [("zseg", 190), ("zseg", 120), ("stages", 3), ("wide_ty", 6)])
def test_a_shape_set_by_the_caller_is_kept(key, value):
    """Also where it is the default's: the choice by size steps back."""
    m = rsg.Mesh(rsg.BOX, (96, 96, 96), spacing=0.2)
    H, x = _ham(m, 32)
    H.apply(x)
    assert H.get_option("last_zseg") < 120   # cut by size
    H.set_option(key, value)
    H.apply(x)
    assert (H.get_option("last_kernel"), H.get_option("last_zseg")) == (7, value if key == "zseg" else 190)
