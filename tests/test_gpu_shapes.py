"""Edges of the kernels' splits against the oracle: band counts around a band group and its ragged tails, atoms
with a single tile and with many, transform lengths on both sides of the 16- and 8-line kernels, handle-free
projections of every orbital count, overlapping spheres in the set-up, and phase tables that do not hold a tile.
Where the states are noise, whose projections cancel, the bound is the arithmetic's own, relative to the terms that are
summed; elsewhere the tolerances are the parity tests'."""
import ctypes as C
import math

import numpy as np
import pytest
import torch

from oracle import dftu_oracle as O
from paper_1711_08935_gb300 import dftu, synth
from paper_1711_08935_gb300.synth import Atom, Grid, System
from tests import _cases
from tests._gpu import run_pass, split_p

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


def _random_states(s, nb, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((s.nk, s.nspin, nb, s.grid.npts, 2))
    return (x[..., 0] + 1j * x[..., 1]) / math.sqrt(s.grid.npts)


def _projection_bounds(s, st, psi, eps):
    """Per atom [M]: eps times dV N max|phi_m| max|psi| over the sphere's N points.  FP32 pairs: every split and every
    compensated product is good to 2^-46 of its chain's largest term, and 2^-44 covers their sum with the merges;
    complex64: at most 48 roundings of 2^-24 along the path of a term (32 points of a lane, five lane merges)."""
    out = []
    for sm in st:
        top = max(np.abs(psi[..., sm["idx"]]).max(), 1e-300)
        out.append(eps * s.grid.dV * len(sm["idx"]) * np.abs(sm["phi"]).max(axis=0) * top)
    return out


# ------------------------------------------------------------------- band groups, ragged tails, shell sizes
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("nb", [1, 8, 9, 16, 17, 31, 33, 41, 48, 65])
def test_noise_states_at_band_counts_around_a_group(dtype, nb):
    """Last groups of 1 to 8, 9 to 16 and more bands (32 and 16 lanes per band, and the full shape) beside full ones,
    and the smallest calls; a d and a p atom whose spheres cross the cell faces (tiles of very uneven size)."""
    s = _cases.periodic_two_atoms()
    st = O.setup_atoms(s)
    psi = _random_states(s, nb, seed=nb)
    seen = torch.from_numpy(psi).to(dtype).to(torch.complex128).numpy()
    f = np.random.default_rng(nb).uniform(0, 1, (s.nk, 2, nb))
    fixed = [(0.3, 0.02), (0.25, 0.01)]
    ref = O.hubbard_pass(s, st, seen, f, fixed_u=fixed)
    out = run_pass(s, psi, f, fixed_u=fixed, dtype=dtype)
    fp64 = dtype == torch.complex128
    bounds = _projection_bounds(s, st, seen, 2.0 ** -44 if fp64 else 48 * 2.0 ** -24)
    for I, p in enumerate(split_p(s, out["p"])):
        assert np.all(np.abs(p - ref["p"][I]) <= bounds[I]), I
    assert rel(out["psi_out"], ref["psi_out"]) < (1e-12 if fp64 else 1e-6)


@pytest.mark.parametrize("mode", [dftu.F64_PAIR, dftu.F64_NATIVE])
def test_every_shell_and_many_tiles(mode):
    """s, p, d and f shells in one isolated box (one to seven orbitals in the tile reduce, U and J kernels), with 1 to
    about 30 tiles per atom, 35 bands."""
    g = Grid((32, 36, 30), (0.3, 0.3, 0.3), periodic=False)
    at = [Atom((3.0, 3.2, 2.9), 0, 0, 0.8), Atom((4.5, 5.0, 4.4), 1, 1, 2.0), Atom((5.0, 5.5, 4.5), 2, 2, 4.4), Atom((4.8, 5.2, 4.6), 3, 3, 3.5)]
    rads = [synth.hydrogenic_radial(1, 0, 2.0), synth.hydrogenic_radial(2, 1, 3.0), synth.hydrogenic_radial(3, 2, 4.0), synth.hydrogenic_radial(4, 3, 5.0)]
    s = System(g, at, rads, np.zeros((1, 3)), np.ones(1), nspin=2)
    nb = 35
    psi = _cases.states_np(s, nb, seed=4)
    f = np.random.default_rng(4).uniform(0, 1, (1, 2, nb))
    rng = np.random.default_rng(5)
    coul = []
    for a in at:   # any integrals with the pair symmetry
        M = 2 * a.l + 1
        V = rng.uniform(0.1, 1.0, (M, M, M, M))
        coul.append(V + V.transpose(1, 0, 2, 3) + V.transpose(0, 1, 3, 2) + V.transpose(1, 0, 3, 2))
    st = O.setup_atoms(s)
    p = O.project(s, st, psi)
    occ = O.occupations(s, p, f)
    out = run_pass(s, psi, f, coulomb=coul, mode=mode)
    for I, q in enumerate(split_p(s, out["p"])):
        assert rel(q, p[I]) < 1e-12, I
    for I in range(1, 4):   # an s shell has no exchange pairs: J's denominator is zero there
        U, J, flag = O.acbn0_uj(occ[I][0], occ[I][1], coul[I], 2)
        assert not flag and abs(out["U"][I] - U) < 1e-11 * abs(U) and abs(out["J"][I] - J) < 1e-11 * abs(J)
    E = sum(O.hubbard_energy(occ[I][0], out["U"][I] - out["J"][I], 2) for I in range(4))
    assert abs(out["EU"] - E) < 1e-11 * abs(E)


# ------------------------------------------------------------------- Coulomb integrals: transform lengths
@pytest.mark.parametrize("l,h,R", [(0, (0.5, 0.4, 0.3), 1.6),       # one pair density: no partner for the imaginary part
                                   (1, (0.25, 0.5, 0.8), 2.0),      # six pairs, three lengths
                                   (2, (0.04, 0.5, 0.6), 1.9),      # 15 pairs (odd); a long axis (8 lines per CTA)
                                   (3, (0.6, 0.45, 0.55), 2.6)])
def test_coulomb_lengths_match_oracle(l, h, R):
    n = tuple(int(math.ceil(2 * (R + 0.6) / x)) + 1 for x in h)
    g = Grid(n, h, periodic=False)
    c = tuple(n[a] * h[a] / 2 + 0.03 for a in range(3))
    s = System(g, [Atom(c, 0, l, R)], [synth.hydrogenic_radial(l + 1, l, 3.0)], np.zeros((1, 3)), np.ones(1), nspin=1)
    st = O.setup_atoms(s)
    ref = O.coulomb_integrals(s.grid, s.atoms[0], st[0])
    nb, _ = O.poisson_box(s.grid, R)
    assert l != 2 or max(nb) >= 208
    hd = dftu.handle_for_system(s, 1)
    assert np.max(np.abs(hd.coulomb_integrals(0) - ref)) < 1e-10 * np.max(np.abs(ref))


# ------------------------------------------------------------------- handle-free projection
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 6, 7])
def test_noalloc_orbital_and_point_counts(dtype, M):
    """Every orbital count, with fewer points than lanes, one point past a tile, and several tiles; 1, 4 and 5 bands
    (a block takes four)."""
    lib = dftu.load()
    rng = np.random.default_rng(M)
    ld, dV = 5000, 0.027
    for npts, nb in ((1, 1), (31, 5), (513, 4), (1700, 5)):
        psi = torch.from_numpy(rng.standard_normal((nb, ld)) + 1j * rng.standard_normal((nb, ld))).cuda().to(dtype)
        idx = rng.integers(0, ld, npts).astype(np.int32)
        ph = np.exp(1j * rng.uniform(0, 6, npts))
        phi = rng.standard_normal((npts, M))
        out = torch.full((nb, M), float("nan"), dtype=torch.complex128, device="cuda")
        t = [torch.from_numpy(x).cuda() for x in (idx, ph, phi)]
        ptr = lambda x: C.c_void_p(x.data_ptr())  # noqa: E731
        assert lib.dftu_project_sphere_noalloc(ptr(psi), dftu.C128 if dtype == torch.complex128 else dftu.C64, nb, ld, ptr(t[0]), ptr(t[1]),
                                               ptr(t[2]), npts, M, dV, ptr(out), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        x = psi.to(torch.complex128).cpu().numpy()
        ref = dV * ((x[:, idx] * ph[None, :]) @ phi)
        assert np.max(np.abs(out.cpu().numpy() - ref)) < 1e-12 * dV * np.max(np.abs(x)) * np.sum(np.abs(phi), axis=0).max()


# ------------------------------------------------------------------- gauge phases and current
@pytest.mark.parametrize("ls", [(0,), (1, 2), (3, 0, 2)])
def test_current_of_every_shell(ls):
    """The current from the monomial tables: shells with one, two and three tables, alone and mixed, against the
    oracle's projections onto the displaced orbitals."""
    g = Grid((24, 22, 26), (0.4, 0.4, 0.4), periodic=True)
    pos = [(1.0, 1.2, 0.8), (5.5, 4.4, 5.0), (3.3, 6.1, 7.2)]
    at = [Atom(pos[i], i, l, 2.6) for i, l in enumerate(ls)]
    rads = [synth.hydrogenic_radial(l + 1, l, 2.5) for l in ls]
    s = System(g, at, rads, np.array([[0.11, -0.05, 0.2], [-0.2, 0.13, 0.04]]), np.array([0.5, 0.5]), nspin=2)
    nb = 11
    psi = _cases.states_np(s, nb, seed=8)
    f = np.random.default_rng(8).uniform(0, 1, (2, 2, nb))
    A = np.array([0.3, -0.2, 0.25])
    fixed = [(0.3, 0.02), (0.25, 0.01), (0.4, 0.05)][:len(ls)]
    st = O.setup_atoms(s)
    occ = O.occupations(s, O.project_gauge(s, st, psi, A), f)
    V = [np.stack([O.potential(occ[I][0][a], fixed[I][0] - fixed[I][1]) for a in range(2)]) for I in range(len(ls))]
    ref = O.hubbard_current(s, st, psi, f, V, A)
    # relative to the sum of the terms' moduli (the terms of a current cancel between states)
    p = O.project_gauge(s, st, psi, A)
    scale = 0.0
    for I, sm in enumerate(st):
        for a in range(3):
            q = O.project_gauge(s, [dict(sm, phi=sm["phi"] * sm["d"][:, a:a + 1])], psi, A)[0]
            scale = max(scale, 2 * np.einsum("ksn,ksnm,ksnq,smq->", s.wk[:, None, None] * f, np.abs(q), np.abs(p[I]), np.abs(V[I])))
    for dtype, tol in ((torch.complex128, 1e-12), (torch.complex64, 2e-6)):
        h = dftu.handle_for_system(s, nb)
        for I, (u, j) in enumerate(fixed):
            h.set_u(I, u, j)
        t, fd = torch.from_numpy(psi).cuda().to(dtype), torch.from_numpy(f).cuda()
        h.set_vector_potential(torch.from_numpy(A).cuda())
        h.project(t)
        h.occupations(fd)
        h.acbn0_uj()
        J, Jat = h.hubbard_current(t, fd, per_atom=True)
        assert np.max(np.abs(J - Jat.sum(axis=0))) <= 1e-15 * scale
        assert np.max(np.abs(J - ref)) < tol * scale


def test_gauge_phases_of_tiles_wider_than_the_tables():
    """A grid so fine along x that one tile spans more grid lines than the phase tables hold, beside one that fits."""
    for hx in (0.01, 0.2):
        nx = int(4.4 / hx)
        g = Grid((nx, 9, 9), (hx, 0.5, 0.5), periodic=False)
        s = System(g, [Atom((2.2, 2.1, 2.05), 0, 1, 2.0)], [synth.hydrogenic_radial(2, 1, 3.0)], np.zeros((1, 3)), np.ones(1), nspin=1)
        nb = 3
        psi = _random_states(s, nb, seed=6)
        A = np.array([0.7, -0.4, 0.9])
        st = O.setup_atoms(s)
        ref = O.project_gauge(s, st, psi, A)[0].reshape(1, nb, 3)
        bound = _projection_bounds(s, st, psi, 2.0 ** -43)[0]   # (one more bit: a rotated component grows by up to sqrt 2)
        h = dftu.handle_for_system(s, nb)
        h.set_vector_potential(torch.from_numpy(A).cuda())
        h.project(torch.from_numpy(psi).cuda())
        assert np.all(np.abs(h.projections(nb) - ref) <= bound)


# ------------------------------------------------------------------- set-up with shared grid points
@pytest.mark.parametrize("case", ["overlapping", "self"])
def test_real_time_overlaps_from_shared_points(case):
    """The overlap blocks of atom pairs and of an atom with its own images come from the grid points that several
    sphere points fall on: one large real-time step against the oracle's, term by term."""
    s = _cases.overlapping_three_atoms() if case == "overlapping" else _cases.periodic_tiny()
    nb = 4
    psi = _random_states(s, nb, seed=12)
    f = np.random.default_rng(12).uniform(0.2, 1.0, (s.nk, 1, nb))
    fixed = [(0.4, 0.05)] * len(s.atoms)
    ref, _ = O.taylor_step(s, O.setup_atoms(s), psi, f, 0.8, fixed_u=fixed)
    h = dftu.handle_for_system(s, nb)
    for I, (u, j) in enumerate(fixed):
        h.set_u(I, u, j)
    t = torch.from_numpy(psi).cuda()
    h.taylor_step(t, None, torch.from_numpy(f).cuda(), 0.8)
    assert rel(t.cpu().numpy(), ref) < 1e-12


@pytest.mark.parametrize("nb", [32, 33])
def test_wide_calls_are_their_narrow_parts(nb):
    """Calls wide enough for a reduce with a thread per state and orbital and for a recursion on 128 threads, with whole
    and with ragged groups of bands: copies of a narrow call's states, the copies empty, step as the narrow call does
    (which the oracle's step pins above)."""
    s = _cases.overlapping_three_atoms()
    copies = 3400 // nb
    psi = _random_states(s, nb, seed=nb)
    f = np.random.default_rng(nb).uniform(0.2, 1.0, (s.nk, 1, nb))
    narrow = torch.from_numpy(psi).cuda()
    wide = narrow.repeat(1, 1, copies, 1).contiguous()
    fw = torch.zeros((s.nk, 1, nb * copies), dtype=torch.float64, device="cuda")
    fw[:, :, :nb] = torch.from_numpy(f).cuda()
    for t, g in ((narrow, torch.from_numpy(f).cuda()), (wide, fw)):
        h = dftu.handle_for_system(s, t.shape[2])
        for I in range(len(s.atoms)):
            h.set_u(I, 0.4, 0.05)
        h.taylor_step(t, None, g, 0.8)
        h.close()
    for c in (0, copies // 2, copies - 1):
        part = wide[:, :, c * nb:(c + 1) * nb]
        assert float((part - narrow).abs().max()) <= 1e-12 * float(narrow.abs().max())
