"""Hamiltonians on one mesh, each used by its own host thread and stream: the
mesh's tables are made on first use by whichever thread comes first, and every
result has the bits of a run by itself."""
import threading

import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 5, 8, 13, 16, 24]


def _ham(m, dtype, S):
    H = rsg.Hamiltonian(m, dtype)
    r = np.random.default_rng(S)
    H.set_potential(r.uniform(-2, 1, m.P))
    g = torch.Generator(device="cuda").manual_seed(S)
    return H, torch.randn((m.P, rsg.padded_ld(S, dtype)), dtype=dtype, device="cuda", generator=g)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_one_mesh_many_threads(dtype):
    def mesh(k):
        return rsg.Mesh(rsg.BOX, (29 + k, 41, 33 + 2 * k), spacing=0.2)

    for k in range(6):
        m = mesh(k)
        want = []
        for S in SIZES:
            H, x = _ham(m, dtype, S)
            want.append(H.apply(x, S=S)[:, :S])
        m = mesh(k)   # no tables yet
        hams = [_ham(m, dtype, S) for S in SIZES]
        torch.cuda.synchronize()
        got, errors, gate = [None] * len(SIZES), [], threading.Barrier(len(SIZES))

        def work(i):
            try:
                st = torch.cuda.Stream()
                gate.wait()
                with torch.cuda.stream(st):
                    got[i] = hams[i][0].apply(hams[i][1], S=SIZES[i])[:, :SIZES[i]]
                st.synchronize()
            except Exception as e:
                errors.append(e)

        ts = [threading.Thread(target=work, args=(i,)) for i in range(len(SIZES))]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errors, errors
        for S, a, b in zip(SIZES, got, want):
            assert torch.equal(a, b), S
