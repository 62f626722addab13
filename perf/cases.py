"""Performance cases: the work a user of this library has it do.

Each case is one pass through the public Python entry points on inputs made
from a seed.  The families are the library's own: one Hamiltonian application
(the building block of everything else), time steps of a block of states with
and without re-orthonormalisation, steps under complex scaling, the
optimal-control gradient, the ground-state iteration, the shifted solve and
the orthonormalisation alone, in both compute types.  Sizes follow the
repository's workloads: 24^3 to 192^3 cubes, spheres of index-mapped points up
to radius 18 bohr, 1 to 128 states, odd state counts, ragged boxes.  Batches of
uneven systems are not among them: some sets of systems end in
RSG_ERR_TIMEOUT, so a drawn batch cannot be timed; a system of that workload's
size is stepped by itself instead.

States that are propagated are smooth packets (what a run starts from); blocks
that H is applied to, solved with or filtered are noise, as in the workloads.
"""
import math

import numpy as np
import torch

import paper_1501_05654_gb300 as rsg

DTYPES = {"c64": torch.complex64, "c128": torch.complex128}


def listed():
    return [
        # One application on the smallest mesh of the batch workload, one
        # state, one atom: a user's own iteration on a toy system, bound by
        # launches and host work.
        dict(name="apply_cube24_c64_s1", kind="apply", shape="cube", n=24, h=0.25, S=1, dtype="c64",
             atoms=1, lmax=1, rcut=2.5, eps=0.0),
        # One application to 13 states (odd, so rows are padded) on a sphere,
        # with projectors and a static field: the matrix-vector product of a
        # user's own solver on a mid-sized molecule.
        dict(name="apply_sphere10_c64_s13", kind="apply", shape="sphere", R=10.0, h=0.2, S=13, dtype="c64",
             atoms=12, lmax=1, rcut=2.5, eps=0.01),
        # The oscillator workload: FP64, 32^3, four states, exponential
        # midpoint, 20 of its 100 steps under a time-dependent field.
        dict(name="expmid_cube32_c128_s4", kind="steps", shape="cube", n=32, h=0.3, S=4, dtype="c128",
             atoms=0, lmax=0, rcut=0.0, eps=0.01, scheme="expmid", nsteps=20, dt=0.01, gs=0),
        # The headline workload: one ETRS step of 64 complex64 states on the
        # 3,053,617-point sphere, 32 wells, 32 atoms x 4 projectors.
        dict(name="etrs_sphere18_c64_s64", kind="steps", shape="sphere", R=18.0, h=0.2, S=64, dtype="c64",
             atoms=32, lmax=1, rcut=2.5, eps=0.0, scheme="etrs", nsteps=1, dt=0.01, gs=0),
        # The same molecule type in FP64 (the complex128 runs of that
        # workload), on a smaller sphere with 16 states.
        dict(name="etrs_sphere12_c128_s16", kind="steps", shape="sphere", R=12.0, h=0.2, S=16, dtype="c128",
             atoms=16, lmax=1, rcut=2.5, eps=0.0, scheme="etrs", nsteps=1, dt=0.01, gs=0),
        # The large mixed-precision workload: 192^3, 128 states, 64 atoms x 9
        # projectors, the step that ends in an FP64 re-orthonormalisation.
        dict(name="etrs_qr_cube192_c64_s128", kind="steps", shape="cube", n=192, h=0.18, S=128, dtype="c64",
             atoms=64, lmax=2, rcut=3.0, eps=0.0, scheme="etrs", nsteps=1, dt=0.01, gs=1),
        # Resonances: a complex-scaled step of 32 states on a sphere.
        dict(name="scaled_sphere14_c64_s32", kind="scaled", shape="sphere", R=14.0, h=0.2, S=32, dtype="c64",
             theta=0.3, wells=16, scheme="etrs", nsteps=1, dt=0.01),
        # One system of the batch workload's size stepped by itself: an
        # ordinary small molecule, 16 states on 48^3, two steps.
        dict(name="etrs_cube48_c64_s16", kind="steps", shape="cube", n=48, h=0.25, S=16, dtype="c64", atoms=4, lmax=1,
             rcut=2.5, eps=0.0, scheme="etrs", nsteps=2, dt=0.02, gs=0),
        # The control workload, FP64 and complex64: one electron on 64^3,
        # double well, 4 ETRS substeps per interval.
        dict(name="gradient_cube64_c128", kind="gradient", n=64, h=0.3, dtype="c128", nsteps=10, nsub=4, dt=0.05,
             every=5),
        dict(name="gradient_cube64_c64", kind="gradient", n=64, h=0.3, dtype="c64", nsteps=20, nsub=4, dt=0.05,
             every=10),
        # Ground state: three iterations of the eigensolver on the 61^3 mesh
        # of the few-electron model (FP64, 8 states).
        dict(name="eigen_cube61_c128_s8", kind="eigen", shape="cube", n=61, h=0.4, S=8, dtype="c128", atoms=0,
             lmax=0, rcut=0.0, eps=0.0, iters=3, degree=16),
        # Linear response at an imaginary frequency: 8 iterations of the
        # shifted solve (a loose inner solve), 8 right-hand sides, wells and
        # projectors.
        dict(name="shifted_sphere14_c64_s8", kind="shifted", shape="sphere", R=14.0, h=0.2, S=8, dtype="c64",
             atoms=16, lmax=1, rcut=2.5, eps=0.0, zr=-0.5, zi=4.0, iters=8),
    ]


# ---------------------------------------------------------------- drawn cases

def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _logint(rng, lo, hi):
    return int(min(hi, max(lo, round(_log(rng, lo, hi)))))


def _draw_mesh(rng, c, biggest):
    """A cube, a ragged box or a sphere of at most `biggest` points."""
    shape = rng.choice(["cube", "box", "sphere"])
    top = biggest ** (1 / 3)
    c["shape"] = shape
    c["h"] = round(rng.uniform(0.18, 0.3), 3)
    if shape == "cube":
        c["n"] = _logint(rng, 16, min(160, top))
    elif shape == "box":
        c["nx"], c["ny"], c["nz"] = (_logint(rng, 12, min(160, top)) for _ in range(3))
    else:
        c["R"] = round(_log(rng, 1.8, min(16.0, c["h"] * top * 0.6)), 2)
    return _count(c)


def _draw_atoms(rng, c):
    c["atoms"] = rng.choice([0, 1, 3, 8, 24])
    c["lmax"] = rng.choice([0, 1, 1, 2])
    c["rcut"] = round(rng.uniform(1.2, 3.0), 2)


def _count(c):
    if c["shape"] == "cube":
        return c["n"] ** 3
    if c["shape"] == "box":
        return c["nx"] * c["ny"] * c["nz"]
    return int(4.2 * (c["R"] / c["h"]) ** 3) + 1


def draw(rng):
    kind = rng.choice(["apply", "apply", "steps", "steps", "steps", "scaled", "gradient", "eigen",
                       "shifted", "ortho"])
    dtype = rng.choice(["c64", "c64", "c128"])
    if kind == "gradient":
        return dict(kind=kind, n=_logint(rng, 16, 72), h=round(rng.uniform(0.25, 0.4), 3), dtype=dtype,
                    nsteps=rng.randint(2, 12), nsub=rng.randint(1, 4), dt=0.02, every=rng.randint(2, 12))
    c = dict(kind=kind, dtype=dtype)
    if kind == "eigen":
        c.update(shape="cube", n=_logint(rng, 16, 64), h=round(rng.uniform(0.3, 0.5), 3), S=rng.randint(2, 12),
                 atoms=0, lmax=0, rcut=0.0, eps=0.0, iters=2, degree=rng.randint(8, 16))
        return c
    P = _draw_mesh(rng, c, 4.0e6 if dtype == "c64" else 1.0e6)
    # point-states: the largest listed case holds 9e8 (complex64); FP64 draws
    # are kept to a tenth of its time
    most = {"apply": 4e8, "steps": 2.5e8, "scaled": 2.5e8, "shifted": 3e7, "ortho": 2e8}[kind]
    if dtype == "c128":
        most *= 0.15
    c["S"] = _logint(rng, 1, max(1, min(128, int(most / P))))
    if kind == "scaled":
        c.update(theta=round(rng.uniform(0.05, 0.6), 3), wells=rng.randint(1, 16),
                 scheme=rng.choice(["etrs", "expmid"]), nsteps=rng.randint(1, 2), dt=0.005)
        return c
    if kind == "ortho":
        return c
    _draw_atoms(rng, c)
    c["eps"] = rng.choice([0.0, 0.01])
    if kind == "steps":
        c.update(scheme=rng.choice(["etrs", "expmid"]), nsteps=rng.randint(1, 3), dt=0.005,
                 gs=rng.choice([0, 0, 1]) if c["S"] * 200 < P else 0)
    if kind == "shifted":
        # complex64 solves: large imaginary shifts and few iterations, whose
        # iterates single precision carries
        lo, hi, most = (0.1, 0.5, 25) if dtype == "c128" else (4.0, 6.0, 8)
        c.update(zr=round(rng.uniform(-2.0, -0.5), 2), zi=round(rng.uniform(lo, hi), 2), iters=rng.randint(4, most))
    return c


# ---------------------------------------------------------------- inputs

def _coords(c):
    """Lattice integers (P, 3) as float64 on the GPU, z slowest and x fastest,
    and the position of lattice (0, 0, 0)."""
    if c["shape"] == "sphere":
        r = math.floor(c["R"] / c["h"] + 1e-6)
        a = torch.arange(-r, r + 1, device="cuda", dtype=torch.float64)
        z, y, x = torch.meshgrid(a, a, a, indexing="ij")
        keep = (x * x + y * y + z * z) <= (c["R"] / c["h"]) ** 2 + 1e-6
        return torch.stack([x[keep], y[keep], z[keep]], 1), (0.0, 0.0, 0.0)
    n = (c["n"],) * 3 if c["shape"] == "cube" else (c["nx"], c["ny"], c["nz"])
    ax = [torch.arange(k, device="cuda", dtype=torch.float64) for k in n]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1), tuple(-(k - 1) * c["h"] / 2 for k in n)


def _half(c):
    """Half extents of the mesh along x, y, z (bohr)."""
    if c["shape"] == "sphere":
        return np.full(3, c["R"] / math.sqrt(3.0))
    n = (c["n"],) * 3 if c["shape"] == "cube" else (c["nx"], c["ny"], c["nz"])
    return 0.5 * c["h"] * (np.array(n) - 1.0)


def _wells(r, half, n):
    cen = r.uniform(-0.8, 0.8, (n, 3)) * half
    return cen, r.uniform(1.0, 4.0, n), r.uniform(0.8, 1.5, n)


def _well_potential(xyz, wells, theta=None):
    """Gaussian wells at every point; complex at rotated coordinates when theta is given."""
    v = torch.zeros(xyz.shape[0], device="cuda", dtype=torch.float64 if theta is None else torch.complex128)
    z = xyz if theta is None else xyz * complex(math.cos(theta), math.sin(theta))
    for cen, d, w in zip(*wells):
        t = z - torch.tensor(cen, device="cuda", dtype=torch.float64)
        v -= d * torch.exp(-(t * t).sum(1) / (2 * w * w))
    return v


def _packets(xyz, r, half, S, ld, dtype, h):
    """Smooth normalised packets, one per state: random centre, width and momentum."""
    out = torch.zeros((xyz.shape[0], ld), device="cuda", dtype=dtype)
    for s in range(S):
        cen = torch.tensor(r.uniform(-0.5, 0.5, 3) * half, device="cuda")
        k = torch.tensor(r.uniform(-0.6, 0.6, 3), device="cuda")
        sg = r.uniform(0.8, 1.5)
        a = torch.exp(-((xyz - cen) ** 2).sum(1) / (4 * sg * sg))
        a /= torch.sqrt((a * a).sum() * h ** 3)
        out[:, s] = torch.polar(a, xyz @ k).to(dtype)
    return out


def _noise(P, S, ld, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.randn((P, ld), device="cuda", dtype=dtype, generator=g)
    out[:, S:] = 0
    return out


def _atoms(c, r, half):
    n = c.get("atoms", 0)
    if not n:
        return None
    m = (c["lmax"] + 1) ** 2
    rc = np.full(n, c["rcut"])
    return (r.uniform(-0.7, 0.7, (n, 3)) * half, rc, np.full(n, c["lmax"], dtype=np.int32), rc / 4.0,
            [np.diag(r.uniform(-1.0, 1.0, m)) for _ in range(n)])


def _ld(S, dtype):
    return S + (S % 2) if dtype == torch.complex64 else S


def _inputs(c, seed):
    """Everything random of a single-system case."""
    r = np.random.Generator(np.random.PCG64(seed))
    dtype = DTYPES[c["dtype"]]
    if c["kind"] == "gradient":
        c = dict(c, shape="cube", S=1)
    ijk, org = _coords(c)
    xyz = ijk * c["h"] + torch.tensor(org, device="cuda", dtype=torch.float64)
    half, S = _half(c), c["S"]
    d = dict(ijk=ijk, xyz=xyz)
    if c["kind"] == "gradient":
        x, y, z = xyz.unbind(1)
        d["V"] = 0.02 * (x * x - 4.0) ** 2 + 0.125 * (y * y + z * z)
        d["psi0"] = _packets(xyz, r, 0.2 * half, 1, 1, dtype, c["h"])[:, 0].contiguous()
        d["target"] = _packets(xyz, r, 0.2 * half, 1, 1, dtype, c["h"])[:, 0].contiguous()
        t = np.arange(c["nsteps"]) * c["dt"]
        w, p = r.uniform(0.05, 0.6, 8), r.uniform(0.0, 6.28, 8)
        d["eps"] = 0.05 * np.sin(w[:, None] * t + p[:, None]).mean(0)
        return d
    if c["kind"] == "ortho":
        d["psi"] = _noise(xyz.shape[0], S, _ld(S, dtype), dtype, seed)
        return d
    if c["kind"] == "scaled":
        d["vt"] = _well_potential(xyz, _wells(r, half, c["wells"]), c["theta"])
    else:
        d["V"] = _well_potential(xyz, _wells(r, half, max(4, c["atoms"])))
        d["atoms"] = _atoms(c, r, half)
        u = r.standard_normal(3)
        d["dir"] = u / np.linalg.norm(u)
    if c["kind"] in ("steps", "scaled"):
        d["psi"] = _packets(xyz, r, half, S, _ld(S, dtype), dtype, c["h"])
        if c.get("gs"):     # a noise part of norm 0.3 keeps packets that overlap independent
            scale = 0.3 / math.sqrt(xyz.shape[0] * c["h"] ** 3)
            d["psi"] += _noise(xyz.shape[0], S, _ld(S, dtype), dtype, seed) * scale
        if c.get("eps"):
            d["field"] = c["eps"] * np.cos(0.3 * np.arange(c["nsteps"]))
    else:
        d["psi"] = _noise(xyz.shape[0], S, _ld(S, dtype), dtype, seed)
    return d


def _mesh(c):
    if c["shape"] == "sphere":
        return rsg.Mesh(rsg.SPHERE, radius=c["R"], spacing=c["h"])
    if c["shape"] == "cube":
        return rsg.Mesh(rsg.CUBE, c["n"], spacing=c["h"])
    return rsg.Mesh(rsg.BOX, (c["nx"], c["ny"], c["nz"]), spacing=c["h"])


def prepare(case, seed):
    c = case
    d = _inputs(c, seed)
    mesh = rsg.Mesh(rsg.CUBE, c["n"], spacing=c["h"]) if c["kind"] == "gradient" else _mesh(c)
    H = rsg.Hamiltonian(mesh, DTYPES[c["dtype"]])
    st = dict(case=c, H=H)
    if "vt" in d:
        H.set_complex_scaling(c["theta"], d["vt"])
    elif "V" in d:
        H.set_potential(d["V"])
    if d.get("atoms") is not None:
        H.set_projectors(*d["atoms"])
    if c.get("eps") and c["kind"] != "steps":
        H.set_field(c["eps"], d["dir"])
    for k in ("psi", "psi0", "target", "eps", "field", "dir"):
        if k in d:
            st[k] = d[k]
    return st


# ---------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    kind = c["kind"]
    H = state["H"]
    if kind == "gradient":
        J, g = H.control_gradient(state["psi0"], state["target"], state["eps"], c["dt"], nsub=c["nsub"],
                                  checkpoint_every=c["every"])
        # a complex64 run's gradient carries single precision: it is handed on as such
        return (np.array([J]), g) if c["dtype"] == "c128" else (np.array([J], np.float32), g.astype(np.float32))
    psi, S = state["psi"], c["S"]
    if kind == "apply":
        return H.apply(psi, S=S)[:, :S]
    if kind in ("steps", "scaled"):
        H.propagate(psi, c["nsteps"], c["dt"], scheme=getattr(rsg, c["scheme"].upper()), eps=state.get("field"),
                    dir=state.get("dir", (1.0, 0.0, 0.0)), gs_every=c.get("gs", 0), S=S, want_drift=False)
        return psi[:, :S]
    if kind == "ortho":
        n2 = H.orthonormalize(psi, S=S)
        return psi[:, :S], n2 if c["dtype"] == "c128" else n2.astype(np.float32)
    if kind == "eigen":
        x = psi.clone()
        ev, res, _ = H.eigensolve(x, max_iter=c["iters"], degree=c["degree"], tol=1e-12, S=S)
        return (x[:, :S], ev, res) if c["dtype"] == "c128" else (x[:, :S], ev.astype(np.float32))
    x = torch.zeros_like(psi)
    H.shifted_solve(psi, x, complex(c["zr"], c["zi"]), max_iter=c["iters"], tol=1e-12, S=S)
    return x[:, :S]


# ---------------------------------------------------------------- work

def _napply(c):
    """Hamiltonian applications of one pass."""
    stages = {"etrs": 8, "expmid": 4}
    if c["kind"] == "apply":
        return 1
    if c["kind"] in ("steps", "scaled"):
        return c["nsteps"] * stages[c["scheme"]]
    if c["kind"] == "gradient":
        return 3 * c["nsteps"] * c["nsub"] * 8
    if c["kind"] == "eigen":
        return c["iters"] * (c["degree"] + 1)
    return c["iters"] + 1


def work(case):
    """Bytes and operations of one pass.  An application needs the whole block
    of the one before (stencil reach and projector sums over whole spheres), so
    each reads and writes the block once; the potential is read with it."""
    c = case
    P = c["n"] ** 3 if c["kind"] == "gradient" else _count(c)
    S = c.get("S", 1)
    z = 8 if c["dtype"] == "c64" else 16
    if c["kind"] == "ortho":
        return {"bytes": 2.0 * P * S * z, "flops": 8.0 * P * S * S}
    n = _napply(c)
    flops = n * P * S * 108.0      # 25 weights and the diagonal on re and im
    if c.get("atoms"):
        flops += n * c["atoms"] * (c["lmax"] + 1) ** 2 * 4.2 * (c["rcut"] / c["h"]) ** 3 * S * 8.0
    if c.get("gs"):
        flops += 8.0 * P * S * S * c["nsteps"]
    return {"bytes": n * (2.0 * P * S * z + P * z / 2.0), "flops": flops}


# ---------------------------------------------------------------- 64-bit reference (plain torch)

W = (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)


class _Ref:
    """H in 64 bits on a zero-padded dense box, applied to (P, s) blocks."""

    def __init__(self, c, d):
        self.h, self.theta = c["h"], c.get("theta", 0.0) if "vt" in d else None
        ijk = d["ijk"].long()
        ijk = ijk - ijk.amin(0)
        n = (ijk.amax(0) + 1).tolist()
        self.n = n
        self.idx = (ijk[:, 2] * n[1] + ijk[:, 1]) * n[0] + ijk[:, 0]
        self.v = d["vt"] if "vt" in d else d["V"]
        self.xyz = d["xyz"]
        self.atoms = []
        if d.get("atoms") is not None:
            for cen, rc, lm, beta, hm in zip(*d["atoms"]):
                t = self.xyz - torch.tensor(cen, device="cuda")
                r2 = (t * t).sum(1)
                at = torch.nonzero(r2 <= rc * rc)[:, 0]
                x, y, z = t[at].unbind(1)
                q = [torch.ones_like(x), x, y, z, x * y, y * z, z * x, x * x - y * y, 3 * z * z - r2[at]]
                p = torch.stack(q[: (lm + 1) ** 2], 1) * torch.exp(-r2[at] / (2 * beta * beta))[:, None]
                p = p / torch.sqrt((p * p).sum(0) * self.h ** 3)
                self.atoms.append((at, p.to(torch.complex128), torch.tensor(hm, device="cuda", dtype=torch.complex128)))

    def lap(self, u):
        n = self.n
        g = torch.zeros((n[2] + 8, n[1] + 8, n[0] + 8, u.shape[1]), dtype=u.dtype, device="cuda")
        box = torch.zeros((n[2] * n[1] * n[0], u.shape[1]), dtype=u.dtype, device="cuda")
        box = box.index_copy(0, self.idx, u)
        mid = [slice(4, 4 + n[2]), slice(4, 4 + n[1]), slice(4, 4 + n[0])]
        g[mid[0], mid[1], mid[2]] = box.view(n[2], n[1], n[0], -1)
        out = g[mid[0], mid[1], mid[2]] * (3 * W[0])
        for ax in range(3):
            for k in range(1, 5):
                for s in (-k, k):
                    w = list(mid)
                    w[ax] = slice(4 + s, 4 + s + n[2 - ax])
                    out.add_(g[w[0], w[1], w[2]], alpha=W[k])
        return out.reshape(-1, u.shape[1])[self.idx] / self.h ** 2

    def apply(self, u, eps=0.0, dir=(1.0, 0.0, 0.0)):
        if self.theta is not None:
            rot = complex(math.cos(2 * self.theta), -math.sin(2 * self.theta))
            return -0.5 * rot * self.lap(u) + self.v[:, None] * u
        x = self.xyz @ torch.tensor(np.asarray(dir, dtype=np.float64), device="cuda")
        out = -0.5 * self.lap(u) + (self.v + eps * x)[:, None] * u
        for at, p, hm in self.atoms:
            out.index_add_(0, at, p @ (hm @ (p.T @ u[at] * self.h ** 3)))
        return out

    def taylor(self, u, tau, eps=0.0, dir=(1.0, 0.0, 0.0)):
        t = o = u
        for k in range(1, 5):
            t = self.apply(t, eps, dir) * (-1j * tau / k)
            o = o + t
        return o

    def step(self, u, dt, scheme, nsub=1, eps=0.0, dir=(1.0, 0.0, 0.0)):
        n, tau = (nsub, dt / nsub) if scheme == "expmid" else (2 * nsub, 0.5 * dt / nsub)
        for _ in range(n):
            u = self.taylor(u, tau, eps, dir)
        return u


def _orthonormal(x, h):
    """Gram-Schmidt in index order by Cholesky of the Gram matrix."""
    G = x.conj().T @ x * h ** 3
    L = torch.linalg.cholesky(G)
    return torch.linalg.solve_triangular(L.conj(), x.T, upper=False).T, G.diagonal().real.clone()


def _by_columns(f, x, points):
    """f on groups of columns that keep the dense box of the reference small."""
    k = max(1, int(3e8 / points))
    return torch.cat([f(x[:, i:i + k]) for i in range(0, x.shape[1], k)], 1)


def _exact_gradient(c, d):
    ref = _Ref(dict(c, shape="cube"), d)
    psi, tgt = d["psi0"].to(torch.complex128)[:, None], d["target"].to(torch.complex128)
    at, h3 = [psi], c["h"] ** 3
    for e in d["eps"]:
        at.append(ref.step(at[-1], c["dt"], "etrs", c["nsub"], float(e)))
    ov = (tgt.conj() * at[-1][:, 0]).sum() * h3
    # chi = cotangent of Re/Im of the final state; back through each interval,
    # whose derivative in eps comes with the Taylor terms' own
    chi = (2 * h3 * ov * tgt)[:, None]
    g = np.zeros(c["nsteps"])
    tau, n = 0.5 * c["dt"] / c["nsub"], 2 * c["nsub"]
    X = ref.xyz[:, :1].to(torch.complex128)
    for k in range(c["nsteps"] - 1, -1, -1):
        e = float(d["eps"][k])
        us = [at[k]]
        for _ in range(n - 1):
            us.append(ref.taylor(us[-1], tau, e))
        for u in reversed(us):
            # T = sum_m B^m / m!, B = -i tau H: dT/de u = sum_m 1/m! sum_j B^j (-i tau X) B^(m-1-j) u
            a, b = [u], [chi]
            for _ in range(3):
                a.append(ref.apply(a[-1], e) * (-1j * tau))
                b.append(ref.apply(b[-1], e) * (1j * tau))
            for i in range(4):
                for j in range(4 - i):
                    g[k] += float((b[j].conj() * (-1j * tau * X) * a[i]).sum().real) / math.factorial(i + j + 1)
            chi = ref.taylor(chi, -tau, e)
    return np.array([float(abs(ov) ** 2)]), g


def exact(case, seed):
    c = case
    if c["kind"] == "eigen":
        return None     # the iterates depend on the filter's own bounds
    d = _inputs(c, seed)
    if c["kind"] == "gradient":
        return _exact_gradient(c, d)
    psi = d["psi"][:, : c["S"]].to(torch.complex128)
    if c["kind"] == "ortho":
        return _orthonormal(psi, c["h"])
    ref = _Ref(c, d)
    points = ref.n[0] * ref.n[1] * ref.n[2]
    dir = d.get("dir", (1.0, 0.0, 0.0))
    if c["kind"] == "apply":
        return _by_columns(lambda u: ref.apply(u, c["eps"], dir), psi, points)
    if c["kind"] in ("steps", "scaled"):
        for k in range(c["nsteps"]):
            e = float(d["field"][k]) if "field" in d else 0.0
            psi = _by_columns(lambda u: ref.step(u, c["dt"], c["scheme"], 1, e, dir), psi, points)
            if c.get("gs"):
                psi = _orthonormal(psi, c["h"])[0]
        return psi
    # conjugate-orthogonal conjugate gradients, all right-hand sides in step
    z = complex(c["zr"], c["zi"])
    A = lambda u: _by_columns(lambda w: ref.apply(w, c["eps"], dir), u, points) - z * u  # noqa: E731
    x, r = torch.zeros_like(psi), psi.clone()
    p, rho = r.clone(), (psi * psi).sum(0)
    for _ in range(c["iters"]):
        q = A(p)
        a = rho / (p * q).sum(0)
        x, r = x + a * p, r - a * q
        new = (r * r).sum(0)
        p, rho = r + new / rho * p, new
    return x
