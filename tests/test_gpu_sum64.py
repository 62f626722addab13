"""The complex128 stencil with integer neighbour sums, on meshes large enough
that the default takes it (a quarter of a million values or more): ragged
tiles, odd and even state counts, spheres, projectors and a field against the
staged FP64 kernel (kernel 0, another summation order: 1e-12 of the largest
value, the library's complex128 tolerance), values spread over the exponent
range, and Inf, NaN, denormals and values near the largest double."""
import numpy as np
import pytest
import torch

import paper_1501_05654_gb300 as rsg

pytestmark = pytest.mark.gpu


def _ham(shape, n, atoms, seed):
    m = rsg.Mesh(rsg.SPHERE, radius=n, spacing=0.2) if shape == "sphere" else rsg.Mesh(rsg.BOX, n, spacing=0.2)
    H = rsg.Hamiltonian(m, torch.complex128)
    r = np.random.default_rng(seed)
    H.set_potential(r.uniform(-2, 1, m.P))
    if atoms:
        half = 0.5 * np.ptp(m.xyz, axis=0)
        H.set_projectors(r.uniform(-0.6, 0.6, (atoms, 3)) * half, np.full(atoms, 1.1), np.full(atoms, 1, np.int32),
                         np.full(atoms, 0.3), [np.diag(r.uniform(-1, 1, 4)) for _ in range(atoms)])
    return m, H, r


def _kernel0(H, f):
    H.set_option("kernel", 0)
    out = f()
    H.set_option("kernel", 1)
    return out


@pytest.mark.parametrize("shape,n,S,atoms", [("box", (70, 61, 45), 3, 0), ("box", (65, 66, 41), 4, 3),
                                             ("box", (33, 129, 65), 17, 0), ("box", (17, 16, 9), 200, 2),
                                             ("box", (300, 5, 3), 130, 0), ("sphere", 9.0, 2, 4), ("sphere", 8.0, 1, 0)])
def test_matches_fp64_sums(shape, n, S, atoms):
    m, H, r = _ham(shape, n, atoms, S)
    x = torch.from_numpy(r.standard_normal((m.P, S)) + 1j * r.standard_normal((m.P, S))).cuda()
    for eps in (0.0, 0.03):
        H.set_field(eps, (0.6, -0.3, 0.7))
        for f in (lambda: H.apply(x), lambda: H.taylor(x, 0.004)):
            got, ref = f(), _kernel0(H, f)
            err = ((got - ref).abs().amax(0) / ref.abs().amax(0)).max().item()
            assert err < 1e-12, (eps, err)


def test_range_of_values():
    """Every value of its own magnitude, 2^-900 to 2^900: each result to 1e-12
    of the largest term of its own star."""
    m, H, r = _ham("box", (64, 64, 64), 0, 1)
    u = (r.standard_normal((m.P, 1)) + 1j * r.standard_normal((m.P, 1))) * np.exp2(r.uniform(-900, 900, (m.P, 1)))
    x = torch.from_numpy(u).cuda()
    got, ref = H.apply(x), _kernel0(H, lambda: H.apply(x))
    g = torch.nn.functional.pad(x.abs().reshape(64, 64, 64), (4,) * 6)
    big = torch.zeros_like(g)
    for d in range(3):
        for k in range(-4, 5):
            big = torch.maximum(big, torch.roll(g, k, d))
    big = big[4:-4, 4:-4, 4:-4].reshape(-1, 1) * 50.0   # the largest weight, 3 w_0, is 53
    assert ((got - ref).abs() <= 1e-12 * big).all()


def _plain(u, V):
    """-1/2 lap u + V u on the 64^3 box, h = 0.2, FP64 numpy."""
    w = [-0.5 * c / 0.04 for c in (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)]
    g = np.zeros((72, 72, 72, u.shape[1]))
    g[4:-4, 4:-4, 4:-4] = u.reshape(64, 64, 64, -1)
    out = (3 * w[0]) * g[4:-4, 4:-4, 4:-4] + V.reshape(64, 64, 64, 1) * g[4:-4, 4:-4, 4:-4]
    for k in range(1, 5):
        s = 0
        for d in range(3):
            for sg in (-k, k):
                s = s + np.roll(g, sg, d)[4:-4, 4:-4, 4:-4]
        out = out + w[k] * s
    return out.reshape(-1, u.shape[1])


def test_special_values():
    m, H, r = _ham("box", (64, 64, 64), 0, 2)
    V = r.uniform(-2, 1, m.P)
    H.set_potential(V)
    u = (r.standard_normal((m.P, 2)) + 1j * r.standard_normal((m.P, 2))) * 1e-300
    u[: m.P // 2, 0] = 0
    u[100, 0], u[70000, 1], u[90000, 0], u[150000, 1] = np.inf, np.nan, -np.inf, 1e308
    u[m.P - 70000:, 0] *= 1e-15   # denormals
    x = torch.from_numpy(u).cuda()
    got = H.apply(x).cpu().numpy()
    # the real operator acts on real and imaginary parts by themselves
    for g, w in ((got.real, _plain(u.real, V)), (got.imag, _plain(u.imag, V))):
        assert np.array_equal(np.isnan(g), np.isnan(w)) and np.array_equal(np.isinf(g), np.isinf(w))
        ok = np.isfinite(w)
        assert np.array_equal(np.sign(g[np.isinf(g)]), np.sign(w[np.isinf(w)]))
        assert np.all(np.abs(g[ok] - w[ok]) <= 1e-12 * np.maximum(np.abs(w[ok]), 1e-298))
