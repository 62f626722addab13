"""Applications and steps on a non-blocking stream straight after the tables they
read were made, and inside a stream capture: the same bits as on the default
stream."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu

CASES = [(torch.complex64, (61, 47, 45), 16, 3), (torch.complex64, (33, 31, 32), 2, 2), (torch.complex64, (70, 52, 66), 32, 0),
         (torch.complex128, (40, 41, 42), 4, 3), (torch.complex128, (12, 13, 11), 1, 2)]


def _ham(dtype, n, S, atoms):
    m = rsg.Mesh(rsg.BOX, n, spacing=0.2)
    H = rsg.Hamiltonian(m, dtype)
    r = np.random.default_rng(S)
    H.set_potential(r.uniform(-2, 1, m.P))
    if atoms:
        half = 0.5 * np.ptp(m.xyz, axis=0)
        H.set_projectors(r.uniform(-0.6, 0.6, (atoms, 3)) * half, np.full(atoms, 1.1), np.full(atoms, 1, np.int32),
                         np.full(atoms, 0.3), [np.diag(r.uniform(-1, 1, 4)) for _ in range(atoms)])
    g = torch.Generator(device="cuda").manual_seed(S)
    return H, torch.randn((m.P, rsg.padded_ld(S, dtype)), dtype=dtype, device="cuda", generator=g)


@pytest.mark.parametrize("dtype,n,S,atoms", CASES)
def test_non_blocking_stream_after_uploads(dtype, n, S, atoms):
    H, x = _ham(dtype, n, S, atoms)
    want = H.taylor(x, 0.004, S=S)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(8):
        H, x = _ham(dtype, n, S, atoms)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            got = H.taylor(x, 0.004, S=S)   # first application: row and tile tables are made here
        st.synchronize()
        assert torch.equal(got, want)


@pytest.mark.parametrize("dtype,n,S,atoms", CASES)
def test_step_in_a_captured_graph(dtype, n, S, atoms):
    H, x = _ham(dtype, n, S, atoms)
    want = x.clone()
    H.propagate(want, 4, 0.004, S=S, want_drift=False)
    a = x.clone()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        H.propagate(a, 1, 0.004, S=S, want_drift=False)   # buffers and tables exist from here on
    st.synchronize()
    a.copy_(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        H.propagate(a, 2, 0.004, S=S, want_drift=False)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(a, want)


def test_batch_on_a_non_blocking_stream():
    sy = [_ham(torch.complex64, (9 + 4 * i,) * 3, 1 + 3 * i, 2) for i in range(4)]
    S = [1 + 3 * i for i in range(4)]
    want = [x.clone() for _, x in sy]
    rsg.Batch([H for H, _ in sy], S).propagate(want, 3, 0.01)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(8):
        xs = [x.clone() for _, x in sy]
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            rsg.Batch([H for H, _ in sy], S).propagate(xs, 3, 0.01)
        st.synchronize()
        for got, w in zip(xs, want):
            assert torch.equal(got, w)
