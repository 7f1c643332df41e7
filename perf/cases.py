"""The measured workloads: what a program that uses the Hubbard projector has it do, through the public
entry points of `paper_1711_08935_gb300.dftu`, from one isolated shell to gigabytes of states.

Kinds of pass
  scf        project -> occupations -> U/J -> H psi += V_U psi -> n, U, J, E_U read back (one iteration)
  rt         several real-time Taylor steps in place, then U, J, E_U read back
  laser      a real-time iteration under a vector potential: phases, projection, potential, current, apply
  forces     the potential of the states, then the Hubbard forces from their gradients
  molecules  one pass over a batch of small isolated systems, applied in place
  setup      the spheres, orbitals and Coulomb integrals of a cell, as at the start of a run and after every
             change of the atoms or their radial functions
  noalloc    the handle-free projection of a caller that brings its own sphere tables

Results of complex64 states are accurate to single precision and are handed on in it.
"""
import ctypes as C
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1711_08935_gb300 import dftu

DEV = torch.device("cuda:0")
SPIN = {"unpolarised": dftu.UNPOLARIZED, "collinear": dftu.COLLINEAR, "noncollinear": dftu.NONCOLLINEAR}
DT = 0.01          # real-time step, atomic units
DR, RMAX = 0.005, 12.0


# ---------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------
def listed():
    return [
        # one d shell in an isolated box, the smallest call: launches and latency (an atom, a quantum dot)
        dict(name="shell_scf", kind="scf", family="shell", n=32, L=9.6, nbands=21, nk=1, dtype="complex128"),
        # a small cell whose spheres cross the faces, odd band count: an ordinary SCF iteration
        dict(name="small_oxide_scf", kind="scf", family="oxide2", n=40, L=12.0, nbands=23, nk=2, dtype="complex128"),
        # the transition-metal oxide supercell in double precision: the production iteration
        dict(name="oxide_scf_c128", kind="scf", family="oxide", n=96, L=24.0, nbands=256, nk=1, dtype="complex128"),
        # the same in single precision
        dict(name="oxide_scf_c64", kind="scf", family="oxide", n=96, L=24.0, nbands=256, nk=1, dtype="complex64"),
        # spinor states (spin-orbit), p shells anywhere in the cell, odd band count
        dict(name="spinor_scf", kind="scf", family="spinor", n=96, L=24.0, natoms=10, nbands=127, nk=2, dtype="complex128"),
        # real-time propagation, 64 atoms of three species, single precision
        dict(name="rt_c64", kind="rt", family="lattice", n=128, L=38.4, nbands=256, nk=1, steps=4, dtype="complex64"),
        # the same propagation in double precision on a coarser grid
        dict(name="rt_c128", kind="rt", family="lattice", n=96, L=38.4, nbands=96, nk=1, steps=4, dtype="complex128"),
        # real time under a laser pulse: the gauge-invariant operator and the current of every step
        dict(name="laser", kind="laser", family="oxide", n=81, L=24.0, nbands=96, nk=1, dtype="complex128"),
        # relaxation: forces on the atoms of a cell
        dict(name="forces", kind="forces", family="oxide", n=72, L=24.0, nbands=65, nk=1, dtype="complex128"),
        # many uneven molecules in one batch
        dict(name="molecules", kind="molecules", family="molecules", count=16, edge=72, bands=160, dtype="complex64"),
        # the start of a run: spheres, orbitals and Coulomb integrals of the supercell
        dict(name="setup", kind="setup", family="oxide", n=96, L=24.0, nbands=64, nk=1, dtype="complex128"),
        # one atom's projections without a handle
        dict(name="noalloc", kind="noalloc", family="oxide", n=96, L=24.0, nbands=128, nk=1, dtype="complex128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scf"] * 5 + ["rt", "rt", "laser", "forces", "molecules", "setup", "noalloc"])
    dtype = rng.choice(["complex128", "complex64"])
    if kind == "scf":
        family = rng.choice(["shell", "oxide2", "oxide", "spinor"])
        if family == "shell":
            n = rng.randint(24, 44)
            return dict(kind=kind, family=family, n=n, L=0.3 * n, nbands=_log_int(rng, 5, 64), nk=1, dtype=dtype)
        if family == "oxide2":
            return dict(kind=kind, family=family, n=rng.randint(34, 48), L=12.0, nbands=_log_int(rng, 6, 96), nk=rng.randint(1, 3), dtype=dtype)
        if family == "oxide":
            nk = rng.randint(1, 2)
            return dict(kind=kind, family=family, n=rng.randint(60, 96), L=24.0, nbands=_log_int(rng, 16, 256 // nk), nk=nk, dtype=dtype)
        nk = rng.randint(1, 2)
        return dict(kind=kind, family=family, n=rng.randint(60, 96), L=24.0, natoms=rng.randint(3, 10), nbands=_log_int(rng, 12, 127), nk=nk, dtype=dtype)
    if kind == "rt":
        top = 224 if dtype == "complex64" else 96
        return dict(kind=kind, family="lattice", n=rng.randint(64, 112 if dtype == "complex64" else 96), L=38.4, nbands=_log_int(rng, 8, top), nk=1,
                    steps=rng.randint(1, 4), dtype=dtype)
    if kind in ("laser", "forces"):
        return dict(kind=kind, family="oxide", n=rng.randint(56, 84), L=24.0, nbands=_log_int(rng, 8, 96), nk=1, dtype=dtype)
    if kind == "molecules":
        return dict(kind=kind, family="molecules", count=rng.randint(3, 16), edge=rng.randint(52, 72), bands=rng.randint(30, 160), dtype=dtype)
    if kind == "setup":
        family = rng.choice(["oxide2", "oxide"])
        n = rng.randint(34, 48) if family == "oxide2" else rng.randint(60, 96)
        return dict(kind=kind, family=family, n=n, L=12.0 if family == "oxide2" else 24.0, nbands=_log_int(rng, 8, 64), nk=rng.randint(1, 2), dtype=dtype)
    return dict(kind=kind, family="oxide", n=rng.randint(60, 96), L=24.0, nbands=_log_int(rng, 8, 128), nk=1, dtype=dtype)


# ---------------------------------------------------------------------------------------------------------
# geometries, states, occupations
# ---------------------------------------------------------------------------------------------------------
def _radial(n, l, Z):
    """Nodeless hydrogen-like radial function (n = l + 1) on r_i = i DR, normalised."""
    r = np.arange(int(round(RMAX / DR)) + 1) * DR
    R = r ** l * np.exp(-Z * r / n)
    return SimpleNamespace(dr=DR, R=R / math.sqrt(float(np.sum(R * R * r * r) * DR)))


def _atom(pos, species, l, radius):
    return SimpleNamespace(pos=tuple(float(x) for x in pos), species=species, l=l, radius=float(radius))


def _system(n, L, atoms, radials, kpts, spin, periodic=True):
    h = L / n
    grid = SimpleNamespace(n=(n, n, n), h=(h, h, h), origin=(0.0, 0.0, 0.0), periodic=periodic, dV=h ** 3, L=(n * h,) * 3)
    kpts = np.asarray(kpts, dtype=np.float64).reshape(-1, 3)
    return SimpleNamespace(grid=grid, atoms=atoms, radials=radials, kpts=kpts, wk=np.full(len(kpts), 1.0 / len(kpts)),
                           spin=spin, ns=1 if spin == "unpolarised" else 2)


def _kpoints(L, nk):
    ks = [(a, b, c) for a in (-1, 1) for b in (-1, 1) for c in (-1, 1)]
    return [[0.25 * 2 * math.pi / L * x for x in ks[i % 8]] for i in range(nk)]


def _geometry(case):
    """The systems of a case (one, or a list for a batch)."""
    fam, d3, p2 = case["family"], _radial(3, 2, 4.0), _radial(2, 1, 4.55)
    if fam == "shell":        # a d shell on the central grid point of an isolated box
        n, L = case["n"], case["L"]
        return _system(n, L, [_atom([(n // 2) * (L / n)] * 3, 0, 2, 4.0)], [d3], [[0.0] * 3], "unpolarised", periodic=False)
    if fam == "oxide2":       # 2 metal d shells and 2 oxygen p shells
        L = case["L"]
        at = [_atom((0, 0, 0), 0, 2, 4.5), _atom((L / 2, L / 2, 0), 0, 2, 4.5), _atom((L / 4, L / 4, L / 4), 1, 1, 3.5),
              _atom((3 * L / 4, 3 * L / 4, L / 4), 1, 1, 3.5)]
        return _system(case["n"], L, at, [d3, p2], _kpoints(L, case["nk"]), "collinear")
    if fam == "oxide":        # rocksalt-like: 8 metal d shells and 8 oxygen p shells
        L = case["L"]
        c = [(i, j, k) for k in range(2) for j in range(2) for i in range(2)]
        at = [_atom([x * L / 2 for x in q], 0, 2, 4.5) for q in c] + [_atom([x * L / 2 + L / 4 for x in q], 1, 1, 3.5) for q in c]
        return _system(case["n"], L, at, [d3, p2], _kpoints(L, case["nk"]), "collinear")
    if fam == "spinor":       # p shells at random places
        rng = np.random.default_rng(3)
        at = [_atom(rng.uniform(0, case["L"], 3), 0, 1, 4.5) for _ in range(case["natoms"])]
        return _system(case["n"], case["L"], at, [_radial(2, 1, 2.0)], _kpoints(case["L"], case["nk"]), "noncollinear")
    if fam == "lattice":      # 64 atoms of three species; the larger spheres overlap across the cell faces
        L, at = case["L"], []
        for i in range(64):
            s = i % 3
            pos = [(i % 4) * L / 4 + 0.1, (i // 4 % 4) * L / 4 + 0.2, (i // 16) * L / 4 + 0.3]
            at.append(_atom(pos, s, (1, 2, 2)[s], (3.5, 4.5, 5.0)[s]))
        k = [[(q + 0.5) / case["nk"] * math.pi / L] * 3 for q in range(case["nk"])]
        return _system(case["n"], L, at, [_radial(2, 1, 3.0), d3, _radial(3, 2, 3.2)], k, "unpolarised")
    out = []                  # molecules: uneven boxes, 1-8 d shells, uneven band counts
    rng = np.random.default_rng(5)
    for _ in range(case["count"]):
        n = int(rng.integers(48, case["edge"] + 1))
        L, at = 0.3 * n, []
        for _ in range(int(rng.integers(1, 9))):
            R = float(rng.uniform(4.0, 5.0))
            at.append(_atom(rng.uniform(R, max(R, L - R), 3), 0, 2, R))
        s = _system(n, L, at, [d3], [[0.0] * 3], "collinear", periodic=False)
        s.nbands = int(rng.integers(20, case["bands"] + 1))
        out.append(s)
    return out


def _axis(sys_, a, X, k, alpha, p):
    """[n] values of (x - X)^p exp(-alpha (x - X)^2) along axis a, Bloch-summed over three images."""
    g = sys_.grid
    x = torch.arange(g.n[a], dtype=torch.float64, device=DEV) * g.h[a]
    out = torch.zeros(g.n[a], dtype=torch.complex128, device=DEV)
    for T in ((-1, 0, 1) if g.periodic else (0,)):
        d = x - (X + T * g.L[a])
        out += complex(math.cos(k * T * g.L[a]), math.sin(k * T * g.L[a])) * d ** p * torch.exp(-alpha * d * d)
    return out.to(torch.complex64)


def _basis(sys_, k):
    """[9 natoms][npts] smooth functions around the atoms: s, p and d polynomials times Gaussians."""
    rows = []
    for at in sys_.atoms:
        alpha = (0.6, 0.9, 0.5)[at.species]
        ax = [[_axis(sys_, a, at.pos[a], float(k[a]), alpha, p) for p in range(3)] for a in range(3)]

        def f(px, py, pz):
            return (ax[2][pz][:, None, None] * ax[1][py][None, :, None] * ax[0][px][None, None, :]).reshape(-1)

        xx, yy, zz = f(2, 0, 0), f(0, 2, 0), f(0, 0, 2)
        for b in (f(0, 0, 0), f(1, 0, 0), f(0, 1, 0), f(0, 0, 1), f(1, 1, 0), f(0, 1, 1), f(1, 0, 1), xx - yy, 2 * zz - xx - yy):
            rows.append(b / torch.linalg.vector_norm(b))
    return torch.stack(rows)


def _states(sys_, nbands, seed, dtype):
    """Normalised states: random combinations of smooth functions around the atoms with 5 % noise, an
    antiferromagnetic weighting of the metal atoms between the spin channels.  Collinear and unpolarised
    [k][spin][band][point], spinors [k][band][component][point]."""
    g = sys_.grid
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    npts, nk, ns = g.n[0] * g.n[1] * g.n[2], len(sys_.kpts), sys_.ns
    nc = sys_.spin == "noncollinear"
    out = torch.empty((nk, nbands, 2, npts) if nc else (nk, ns, nbands, npts), dtype=dtype, device=DEV)
    for ik in range(nk):
        B = _basis(sys_, sys_.kpts[ik])
        for s in range(ns):
            w = torch.ones(len(sys_.atoms), device=DEV)
            if sys_.spin == "collinear":
                for i, at in enumerate(sys_.atoms):
                    if at.l == 2:
                        w[i] = 0.85 if (i.bit_count() + s) % 2 == 0 else 0.15
            cf = torch.randn(nbands, B.shape[0], 2, generator=gen, device=DEV)
            cf = torch.view_as_complex(cf) * w.repeat_interleave(9)[None, :]
            for b0 in range(0, nbands, 32):
                x = cf[b0:b0 + 32] @ B
                z = torch.view_as_complex(torch.randn(x.shape[0], npts, 2, generator=gen, device=DEV))
                x = x + z * (0.05 / math.sqrt(npts) * torch.linalg.vector_norm(x, dim=1, keepdim=True) / math.sqrt(2.0))
                nrm = torch.linalg.vector_norm(x, dim=1, keepdim=True).to(torch.float64) * math.sqrt(g.dV * (2.0 if nc else 1.0))
                x = (x.to(torch.complex128) / nrm).to(dtype) if dtype == torch.complex128 else x / nrm.to(torch.float32)
                if nc:
                    out[ik, b0:b0 + 32, s] = x
                else:
                    out[ik, s, b0:b0 + 32] = x
        del B
    return out


def _occupations(sys_, nbands):
    """Fermi occupations, half filling: [k][spin][band] (spinors [k][band]), per spin."""
    e = (torch.arange(nbands, dtype=torch.float64, device=DEV) + 0.5) / nbands - 0.5
    f = 1.0 / (1.0 + torch.exp(e / 0.05))
    shape = (len(sys_.kpts), nbands) if sys_.spin == "noncollinear" else (len(sys_.kpts), sys_.ns, nbands)
    return f.expand(shape).contiguous()


def _vector_potential(seed):
    r = np.random.default_rng(seed)
    return r.uniform(-0.3, 0.3, 3)


def _gradient(sys_, psi, a):
    """Central differences of the states along axis a (x fastest)."""
    n = sys_.grid.n
    x = psi.view(*psi.shape[:-1], n[2], n[1], n[0])
    return ((torch.roll(x, -1, -1 - a) - torch.roll(x, 1, -1 - a)) / (2 * sys_.grid.h[a])).reshape(psi.shape).contiguous()


def _dtype(case):
    return torch.complex128 if case["dtype"] == "complex128" else torch.complex64


def _inputs(case, seed):
    """Everything that a pass reads, from the seed alone."""
    s = _geometry(case)
    x = SimpleNamespace(case=case, system=s)
    if case["kind"] == "molecules":
        x.psi = [_states(m, m.nbands, seed * 1000 + i, _dtype(case)) for i, m in enumerate(s)]
        x.f = [_occupations(m, m.nbands) for m in s]
        return x
    if case["kind"] == "setup":
        # other radial functions for every seed
        rng = np.random.default_rng(seed)
        s.radials = [_radial(l + 1, l, Z * rng.uniform(0.9, 1.1)) for l, Z in ((2, 4.0), (1, 4.55))]
        return x
    x.psi = _states(s, case["nbands"], seed, _dtype(case))
    x.f = _occupations(s, case["nbands"])
    if case["kind"] == "laser":
        x.A = _vector_potential(seed)
    if case["kind"] in ("scf", "laser"):
        x.hpsi = x.psi * 0.5            # the other terms of H psi are in the buffer already
    if case["kind"] == "forces":
        x.dpsi = [_gradient(s, x.psi, a) for a in range(3)]
    if case["kind"] == "noalloc":
        m = _sphere(s, s.atoms[0])
        x.rows = x.psi[0, 0].contiguous()
        x.idx = torch.from_numpy(m.idx.astype(np.int32)).to(DEV)
        x.phase = torch.from_numpy(np.exp(1j * ((m.T * np.array(s.grid.L)) @ s.kpts[0]))).to(DEV)
        x.phi = torch.from_numpy(m.phi).to(DEV)
    return x


# ---------------------------------------------------------------------------------------------------------
# what a program has in hand before the call, and the call
# ---------------------------------------------------------------------------------------------------------
def _handle(s, max_bands):
    h = dftu.Handle(s.grid, s.kpts, s.wk, SPIN[s.spin], max_bands)
    h.setup_atoms(s.atoms, s.radials)
    for sp in range(len(s.radials)):
        h.coulomb_integrals(sp)
    return h


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "molecules":
        x.handles = [_handle(m, m.nbands) for m in x.system]
        x.batch = dftu.Batch(x.handles)
        x.batch.bind(x.psi, x.f)
        x.coef = torch.tensor([-1j * DT], dtype=torch.complex128, device=DEV)   # a first-order real-time step
    elif kind == "noalloc":
        x.lib = dftu.load()
        x.out = torch.empty(case["nbands"], x.phi.shape[1], dtype=torch.complex128, device=DEV)
    elif kind != "setup":
        x.h = _handle(x.system, case["nbands"])
        if kind == "laser":
            x.A = torch.from_numpy(x.A).to(DEV)
    return x


def _single(case, v):
    """Results of complex64 states in single precision."""
    if case["dtype"] == "complex128":
        return v
    if isinstance(v, (list, tuple)):
        return [_single(case, y) for y in v]
    v = np.asarray(v)
    return v.astype(np.complex64 if v.dtype.kind == "c" else np.float32)


def run(x):
    case, kind = x.case, x.case["kind"]
    if kind == "scf":
        h = x.h
        h.project(x.psi)
        h.occupations(x.f)
        h.acbn0_uj()
        h.apply(x.hpsi)
        r = h.results()
        return dict(hpsi=x.hpsi, n=_single(case, r["n"]), U=_single(case, r["U"]), J=_single(case, r["J"]),
                    EU_atom=_single(case, r["EU_atom"]), EU=_single(case, r["EU"]))
    if kind == "rt":
        x.h.taylor_steps(x.psi, x.f, DT, case["steps"])
        r = x.h.results()
        return dict(psi=x.psi, U=_single(case, r["U"]), J=_single(case, r["J"]), EU=_single(case, r["EU"]))
    if kind == "laser":
        h = x.h
        h.set_vector_potential(x.A)
        h.project(x.psi)
        h.occupations(x.f)
        h.acbn0_uj()
        cur = h.hubbard_current(x.psi, x.f)
        h.apply(x.hpsi)
        return dict(hpsi=x.hpsi, current=_single(case, cur))
    if kind == "forces":
        h = x.h
        h.project(x.psi)
        h.occupations(x.f)
        h.acbn0_uj()
        return dict(forces=_single(case, h.forces(x.dpsi, x.f)))
    if kind == "molecules":
        b = x.batch
        b.project()
        b.occupations()
        b.acbn0_uj()
        b.apply(x.coef)
        return dict(psi=x.psi, EU=_single(case, [m.results()["EU"] for m in x.handles]))
    if kind == "setup":
        s = x.system
        h = dftu.Handle(s.grid, s.kpts, s.wk, SPIN[s.spin], case["nbands"])
        npts = h.setup_atoms(s.atoms, s.radials)
        V = [h.coulomb_integrals(sp) for sp in range(len(s.radials))]
        first = [next(i for i, a in enumerate(s.atoms) if a.species == sp) for sp in range(len(s.radials))]
        maps = [h.get_sphere(i) for i in first]
        h.close()
        return dict(npts=npts, V=V, idx=[m[0] for m in maps], image=[m[1] for m in maps], phi=[m[2] for m in maps])
    p = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    st = x.lib.dftu_project_sphere_noalloc(p(x.rows), dftu.C128 if x.rows.dtype == torch.complex128 else dftu.C64, x.rows.shape[0],
                                           x.rows.shape[1], p(x.idx), p(x.phase), p(x.phi), x.idx.numel(), x.phi.shape[1],
                                           x.system.grid.dV, p(x.out), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    if st != dftu.DFTU_OK:
        raise RuntimeError("projection refused: %d" % st)
    return dict(p=x.out)


# ---------------------------------------------------------------------------------------------------------
# the work that a pass cannot do without
# ---------------------------------------------------------------------------------------------------------
def _count(s, at):
    """Points of an atom's sphere, by volume."""
    return 4.0 / 3.0 * math.pi * at.radius ** 3 / s.grid.dV


def _state_work(s, nbands, size, reads, writes, products):
    """Bytes and floating-point operations of `reads` gathers and `writes` scatters of every sphere point,
    with `products` complex-times-real products per point and orbital."""
    rows = len(s.kpts) * s.ns * nbands
    b = f = 0.0
    for at in s.atoms:
        n = _count(s, at)
        b += n * rows * size * (reads + writes) + n * (2 * at.l + 1) * 8
        f += n * rows * (2 * at.l + 1) * 4 * products
    return b, f


def _fft_work(s):
    """Coulomb integrals of every species: the pair densities' Poisson solves on the padded box."""
    b = f = 0.0
    for sp in range(len(s.radials)):
        at = next(a for a in s.atoms if a.species == sp)
        M = 2 * at.l + 1
        P = M * (M + 1) // 2
        nb = [_smooth(int(math.ceil((4 * at.radius + 2 * max(s.grid.h)) / s.grid.h[a]))) for a in range(3)]
        N = nb[0] * nb[1] * nb[2]
        f += P * (2 * 2.5 * N * math.log2(N) + 2 * N) + 2 * P * P * _count(s, at)
        b += P * (N + _count(s, at)) * 8
    return b, f


def work(case):
    size = 16 if case["dtype"] == "complex128" else 8
    kind, s = case["kind"], _geometry(case)
    if kind == "molecules":
        w = [_state_work(m, m.nbands, size, 2, 1, 2) for m in s]
        b, f = sum(x[0] for x in w), sum(x[1] for x in w)
    elif kind == "scf":
        b, f = _state_work(s, case["nbands"], size, 2, 1, 2)
    elif kind == "rt":        # one gather before the first step, then every step reads and writes every point
        b, f = _state_work(s, case["nbands"], size, 1 + case["steps"], case["steps"], 2 * case["steps"] + 1)
    elif kind == "laser":     # the projection and the current read the same states
        b, f = _state_work(s, case["nbands"], size, 2, 1, 5)
    elif kind == "forces":
        b, f = _state_work(s, case["nbands"], size, 4, 0, 4)
    elif kind == "setup":
        b, f = _fft_work(s)
        for at in s.atoms:    # the maps, orbitals, their splits and the displaced tables
            b += _count(s, at) * (4 + 12 + 1 + (2 * at.l + 1) * 16 * 4)
            f += _count(s, at) * (60 + 4 * (2 * at.l + 1) ** 2)
    else:
        one = SimpleNamespace(**{**vars(s), "atoms": s.atoms[:1], "kpts": s.kpts[:1], "ns": 1})
        b, f = _state_work(one, case["nbands"], size, 1, 0, 1)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------------------
# the same results in 64 bits, from the equations
# ---------------------------------------------------------------------------------------------------------
def _lagrange(rad, r):
    t = r / rad.dr
    i = np.floor(t).astype(np.int64)
    a = np.clip(i - 1, 0, len(rad.R) - 4)
    x = t - a
    w = (-(x - 1) * (x - 2) * (x - 3) / 6, x * (x - 2) * (x - 3) / 2, -x * (x - 1) * (x - 3) / 2, x * (x - 1) * (x - 2) / 6)
    return np.where(i < len(rad.R) - 1, sum(w[q] * rad.R[a + q] for q in range(4)), 0.0)


def _ylm(l, d, r):
    x, y, z = d.T
    with np.errstate(divide="ignore", invalid="ignore"):
        if l == 1:
            Y = math.sqrt(3 / (4 * math.pi)) * np.stack([y, z, x], 1) / r[:, None]
        else:
            c1, c2, c3 = math.sqrt(15 / (4 * math.pi)), math.sqrt(5 / (16 * math.pi)), math.sqrt(15 / (16 * math.pi))
            Y = np.stack([c1 * x * y, c1 * y * z, c2 * (3 * z * z - r * r), c1 * x * z, c3 * (x * x - y * y)], 1) / (r * r)[:, None]
    Y[r == 0] = 0.0
    return Y


def _sphere(s, at):
    """Points of an atom's sphere (z outer, x inner), their lattice images and orthonormal orbitals."""
    g = s.grid
    lo = [math.floor((at.pos[a] - at.radius) / g.h[a]) - 1 for a in range(3)]
    hi = [math.ceil((at.pos[a] + at.radius) / g.h[a]) + 1 for a in range(3)]
    u = np.stack([v.reshape(-1) for v in np.meshgrid(*[np.arange(lo[a], hi[a] + 1) for a in (2, 1, 0)], indexing="ij")][::-1], 1)
    d = u * np.array(g.h) - np.array(at.pos)
    d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
    keep = d2 <= at.radius * at.radius
    if not g.periodic:
        keep &= np.all((u >= 0) & (u < np.array(g.n)), axis=1)
    u, d, r = u[keep], d[keep], np.sqrt(d2[keep])
    T = np.floor_divide(u, np.array(g.n))
    w = u - T * np.array(g.n)
    raw = _lagrange(s.radials[at.species], r)[:, None] * _ylm(at.l, d, r)
    lam, W = np.linalg.eigh(g.dV * raw.T @ raw)
    return SimpleNamespace(idx=w[:, 0] + g.n[0] * (w[:, 1] + g.n[1] * w[:, 2]), T=T, u=u, d=d, phi=raw @ (W * lam ** -0.5) @ W.T)


def _smooth(n):
    while True:
        k = n
        for p in (2, 3, 5):
            while k % p == 0:
                k //= p
        if k == 1:
            return n
        n += 1


def _coulomb(s, at, m):
    """(ab|cd) of one shell by the truncated-kernel Poisson solve on a padded box."""
    g, M = s.grid, m.phi.shape[1]
    Rc = 2 * at.radius + 2 * max(g.h)
    nb = [_smooth(int(math.ceil((2 * at.radius + Rc) / g.h[a]))) for a in range(3)]
    G = [2 * math.pi * torch.fft.fftfreq(nb[a], d=g.h[a], dtype=torch.float64, device=DEV) for a in range(3)]
    G2 = G[0][:, None, None] ** 2 + G[1][None, :, None] ** 2 + G[2][None, None, :] ** 2
    K = 4 * math.pi * (1 - torch.cos(torch.sqrt(G2) * Rc)) / torch.where(G2 == 0, 1.0, G2)
    K[0, 0, 0] = 2 * math.pi * Rc * Rc
    u = torch.from_numpy(m.u - m.u.min(0)).to(DEV)
    phi = torch.from_numpy(m.phi).to(DEV)
    pairs = [(a, b) for a in range(M) for b in range(a, M)]
    dens = torch.stack([phi[:, a] * phi[:, b] for a, b in pairs])
    W = torch.empty(len(pairs), len(pairs), dtype=torch.float64)
    for j in range(len(pairs)):
        box = torch.zeros(*nb, dtype=torch.float64, device=DEV)
        box[u[:, 0], u[:, 1], u[:, 2]] = dens[j]
        v = torch.fft.ifftn(K * torch.fft.fftn(box)).real
        W[:, j] = (g.dV * (dens @ v[u[:, 0], u[:, 1], u[:, 2]])).cpu()
    at_ = {p: i for i, p in enumerate(pairs)}
    ix = np.array([[at_[min(a, b), max(a, b)] for b in range(M)] for a in range(M)])
    return W.numpy()[ix[:, :, None, None], ix[None, None, :, :]]


class _Exact:
    """One system's operator in 64 bits: rows are the (k, spin or component) blocks of the states."""

    def __init__(self, s, A=None, coulomb=True):
        self.s, self.maps, cache = s, [_sphere(s, a) for a in s.atoms], {}
        self.V4 = []
        for at, m in zip(s.atoms, self.maps):
            if coulomb and at.species not in cache:
                cache[at.species] = _coulomb(s, at, m)
            self.V4.append(cache.get(at.species))
        self.idx = [torch.from_numpy(m.idx.astype(np.int64)).to(DEV) for m in self.maps]
        self.G = []            # [k][atom] points x M: phi exp(i k T) exp(i A d)
        for k in s.kpts:
            row = []
            for m in self.maps:
                th = (m.T * np.array(s.grid.L)) @ k + (m.d @ A if A is not None else 0.0)
                row.append(torch.from_numpy(np.exp(1j * th)[:, None] * m.phi).to(DEV))
            self.G.append(row)

    def rows(self, psi):
        """(k, spin, view [band][point]) of every block of states."""
        nc = self.s.spin == "noncollinear"
        return [(k, c, psi[k, :, c] if nc else psi[k, c]) for k in range(len(self.s.kpts)) for c in range(self.s.ns)]

    def project(self, psi, weight=None):
        """p[atom][k][spin][band][m]; weight: a factor of every point of an atom."""
        out = []
        for I, idx in enumerate(self.idx):
            w = torch.from_numpy(weight(self.maps[I])).to(DEV)[:, None] if weight else 1.0
            p = [self.s.grid.dV * (x.index_select(1, idx).to(torch.complex128) @ (self.G[k][I] * w)) for k, c, x in self.rows(psi)]
            out.append(torch.stack(p).reshape(len(self.s.kpts), self.s.ns, p[0].shape[0], -1))
        return out

    def potential(self, p, f):
        """n, U, J, E per atom and V per atom (acting on the combined index (spin, m) of a spinor)."""
        s, nc = self.s, self.s.spin == "noncollinear"
        wk = torch.from_numpy(s.wk).to(DEV)
        wf = wk[:, None] * f if nc else wk[:, None, None] * f
        nbar = {}
        for I, at in enumerate(s.atoms):
            t = p[I].abs().square().sum(-1)
            t = t.sum(1) if nc else t
            nbar[at.species] = nbar[at.species] + t if at.species in nbar else t
        res = SimpleNamespace(n=[], U=[], J=[], E=[], V=[])
        for I, at in enumerate(s.atoms):
            M, q = p[I].shape[-1], p[I]
            if nc:
                q = q.permute(0, 2, 1, 3).reshape(q.shape[0], q.shape[2], 2 * M)
                rho = [torch.einsum("kb,kbx,kby->xy", (wf * y).to(q.dtype), q, q.conj())[None].cpu().numpy() for y in (1.0, nbar[at.species])]
            else:
                rho = [torch.einsum("ksb,ksbx,ksby->sxy", (wf * y).to(q.dtype), q, q.conj()).cpu().numpy() for y in (1.0, nbar[at.species])]
            n, P, V4 = rho[0].swapaxes(1, 2), rho[1].swapaxes(1, 2), self.V4[I]
            if nc:
                blk = lambda a: a[0].reshape(2, M, 2, M).transpose(0, 2, 1, 3)  # noqa: E731
            else:
                def blk(a):
                    b = np.zeros((2, 2, M, M), dtype=complex)
                    b[0, 0], b[1, 1] = a[0], a[-1]
                    return b
            nb, Pb = blk(n), blk(P)
            D = np.einsum("stmm->stm", nb)
            tot = Pb[0, 0] + Pb[1, 1]
            numU = np.einsum("ab,cd,abcd->", tot, tot, V4)
            numJ = sum(np.einsum("ab,cd,adcb->", Pb[x, y], Pb[y, x], V4) for x in range(2) for y in range(2))
            same = sum(D[x, x].sum() ** 2 - (D[x, x] ** 2).sum() for x in range(2))
            flip = sum((D[x, 1 - x] * D[1 - x, x]).sum() for x in range(2))
            opp = 2 * D[0, 0].sum() * D[1, 1].sum()
            cross = sum(D[x, 1 - x].sum() * D[1 - x, x].sum() for x in range(2)) - flip
            U, J = float((numU / (same + opp - flip)).real), float((numJ / (same + cross)).real)
            e = sum(float((np.trace(b) - np.einsum("xy,yx->", b, b)).real) for b in n) * (2 if s.spin == "unpolarised" else 1)
            res.n.append(n)
            res.U.append(U)
            res.J.append(J)
            res.E.append(0.5 * (U - J) * e)
            res.V.append(torch.from_numpy((U - J) * (0.5 * np.eye(rho[0].shape[-1]) - rho[0])).to(DEV))
        return res

    def times(self, V, p):
        """V p, laid out like p."""
        out = []
        for Vi, pi in zip(V, p):
            if self.s.spin == "noncollinear":
                nk, _, nb, M = pi.shape
                q = pi.permute(0, 2, 1, 3).reshape(nk, nb, 2 * M) @ Vi[0].T
                out.append(q.reshape(nk, nb, 2, M).permute(0, 2, 1, 3))
            else:
                out.append(torch.einsum("sxy,ksby->ksbx", Vi, pi))
        return out

    def scatter(self, into, cv):
        for k, c, x in self.rows(into):
            for I, idx in enumerate(self.idx):
                x.index_add_(1, idx, cv[I][k, c] @ self.G[k][I].conj().T)
        return into


def exact(case, seed):
    x = _inputs(case, seed)
    s, kind = x.system, case["kind"]
    if kind == "molecules":
        psi, EU = [], []
        for m, y, f in zip(s, x.psi, x.f):
            o = _Exact(m)
            p = o.project(y)
            r = o.potential(p, f)
            psi.append(o.scatter(y.to(torch.complex128), [-1j * DT * v for v in o.times(r.V, p)]))
            EU.append(np.float64(sum(r.E)))
        return dict(psi=psi, EU=EU)
    if kind == "setup":
        first = [next(i for i, a in enumerate(s.atoms) if a.species == sp) for sp in range(len(s.radials))]
        maps = [_sphere(s, s.atoms[i]) for i in first]
        return dict(npts=None, V=[_coulomb(s, s.atoms[i], m) for i, m in zip(first, maps)], idx=[None, None], image=[None, None],
                    phi=[m.phi for m in maps])
    if kind == "noalloc":
        return dict(p=s.grid.dV * ((x.rows.index_select(1, x.idx.long()).to(torch.complex128) * x.phase) @ x.phi.to(torch.complex128)))
    A = x.A if kind == "laser" else None
    o = _Exact(s, A)
    if kind == "rt":
        psi = x.psi.to(torch.complex128)
        x.psi = None
        for _ in range(case["steps"]):
            p = o.project(psi)
            r = o.potential(p, x.f)
            term, prev = None, p
            for j in range(1, 5):      # terms of the Taylor sum, each a vector on the grid
                cv = [(-1j * DT / j) * v for v in o.times(r.V, prev)]
                if term is None:
                    term = torch.zeros_like(psi)
                else:
                    term.zero_()
                o.scatter(term, cv)
                total = cv if j == 1 else [a + b for a, b in zip(total, cv)]
                if j < 4:
                    prev = o.project(term)
            del term
            o.scatter(psi, total)
        return dict(psi=psi, U=np.array(r.U), J=np.array(r.J), EU=np.float64(sum(r.E)))
    p = o.project(x.psi)
    r = o.potential(p, x.f)
    if kind == "scf":
        out = o.scatter(x.hpsi.to(torch.complex128), o.times(r.V, p))
        return dict(hpsi=out, n=r.n, U=np.array(r.U), J=np.array(r.J), EU_atom=np.array(r.E), EU=np.float64(sum(r.E)))
    wf = torch.from_numpy(s.wk).to(DEV)[:, None, None] * x.f
    Vp = o.times(r.V, p)
    if kind == "laser":
        cur = np.zeros(3)
        for a in range(3):
            q = o.project(x.psi, weight=lambda m: np.ascontiguousarray(m.d[:, a]))
            cur[a] = sum(float((2.0 * wf * (y.conj() * v).sum(-1).imag).sum()) for y, v in zip(q, Vp))
        return dict(hpsi=o.scatter(x.hpsi.to(torch.complex128), Vp), current=cur)
    F = np.zeros((len(s.atoms), 3))
    for a in range(3):
        g = o.project(x.dpsi[a])
        F[:, a] = [-float((2.0 * wf * (y.conj() * v).sum(-1).real).sum()) for y, v in zip(g, Vp)]
    return dict(forces=F)
