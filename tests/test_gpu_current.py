"""The Hubbard current beyond the parity tests: occupation sums that are not Hermitian, and the error of its projections
against the arithmetic's on the displaced orbitals."""
import math

import numpy as np
import pytest
import torch

from oracle import dftu_oracle as O
from paper_1711_08935_gb300 import dftu, synth
from paper_1711_08935_gb300.synth import Atom, Grid, System
from tests import _cases

pytestmark = pytest.mark.gpu


def test_current_of_imported_sums_that_are_not_hermitian():
    """The current is Im sum V_mm' [conj(q_m) p_m' - conj(p_m) q_m'] of the potential as it stands: a caller may import
    any occupation sums, and V = U_eff (1/2 - n^T) has their anti-Hermitian part.  The bound is the parity tests',
    relative to the sum of the terms' moduli."""
    s = _cases.periodic_two_atoms()
    nb = 5
    psi = _cases.states_np(s, nb, seed=21)
    rng = np.random.default_rng(21)
    f = rng.uniform(0, 1, (s.nk, 2, nb))
    A = np.array([0.2, -0.3, 0.15])
    fixed = [(0.3, 0.02), (0.25, 0.01)]
    M = [2 * a.l + 1 for a in s.atoms]
    rho = [rng.uniform(-0.5, 0.5, (2, m, m)) + 1j * rng.uniform(-0.5, 0.5, (2, m, m)) for m in M]
    V = [(u - j) * (0.5 * np.eye(m) - r) for (u, j), r, m in zip(fixed, rho, M)]
    st = O.setup_atoms(s)
    ref = O.hubbard_current(s, st, psi, f, V, A)
    p = O.project_gauge(s, st, psi, A)
    scale = 0.0
    for I, sm in enumerate(st):
        for a in range(3):
            q = O.project_gauge(s, [dict(sm, phi=sm["phi"] * sm["d"][:, a:a + 1])], psi, A)[0]
            scale += np.einsum("ksn,ksnm,ksnq,smq->", s.wk[:, None, None] * f, np.abs(q), np.abs(p[I]), np.abs(V[I]))
    h = dftu.handle_for_system(s, nb)
    for I, (u, j) in enumerate(fixed):
        h.set_u(I, u, j)
    t, fd = torch.from_numpy(psi).cuda(), torch.from_numpy(f).cuda()
    h.set_vector_potential(torch.from_numpy(A).cuda())
    h.project(t)
    h.occupations(fd)
    flat = np.concatenate([r.reshape(-1) for r in rho] * 2)   # n^T, then Pbar (not read with fixed U)
    h.set_occupation_sums(torch.from_numpy(flat.view(np.float64)).cuda())
    h.acbn0_uj()
    assert np.max(np.abs(h.hubbard_current(t, fd) - ref)) < 1e-12 * scale


def _current_system(l):
    """One shell in an isolated box and 64 states of its size: random complex polynomials of degree two under a Gaussian,
    with 5 % noise (whole groups of bands, one image, no phases: every projection is the full shape's plain sum)."""
    h, n = 0.3, 32
    c = (4.83, 4.71, 4.94)
    s = System(Grid((n, n, n), (h, h, h), periodic=False), [Atom(c, 0, l, 4.2)], [synth.hydrogenic_radial(l + 1, l, 1.3 * (l + 1))],
               np.zeros((1, 3)), np.ones(1), nspin=1)
    rng = np.random.default_rng(100 + l)
    x = np.arange(n) * h
    d = np.stack([np.tile(x - c[0], n * n), np.tile(np.repeat(x - c[1], n), n), np.repeat(x - c[2], n * n)])
    poly = np.stack([np.ones(n ** 3), *d, d[0] * d[1], d[1] * d[2], d[2] * d[0], *(d * d)]) * np.exp(-0.6 * (d * d).sum(0))
    cf = rng.standard_normal((64, 10)) + 1j * rng.standard_normal((64, 10))
    psi = cf @ (poly / np.linalg.norm(poly, axis=1, keepdims=True))
    psi /= np.linalg.norm(psi, axis=1, keepdims=True)
    psi = psi + 0.05 / math.sqrt(2 * n ** 3) * (rng.standard_normal(psi.shape) + 1j * rng.standard_normal(psi.shape))
    return s, (psi / math.sqrt(s.grid.dV))[None, None], rng.uniform(0, 1, (1, 1, 64)) / 64, [(0.3, 0.02)]


# rms error over rms current of every state's current on _current_system(l), with the kernels' arithmetic (chains of eight
# points offset by a power of two, FP32 chunk sums; 512-point tiles) restated in NumPy on the displaced orbitals phi_m d_a
DISPLACED_ERROR = {0: (8.76e-14, 8.13e-9), 1: (1.085e-13, 6.46e-9), 2: (3.17e-13, 1.21e-8), 3: (3.14e-13, 8.03e-9)}


@pytest.mark.parametrize("l", [0, 1, 2, 3])
def test_current_is_as_accurate_as_on_the_displaced_orbitals(l):
    """The projections behind the current may be taken onto any functions that span phi_m d_a, at no loss: p and V are
    the native FP64 ones, and native FP64 is the reference.  192 numbers a side give the rms to 5 %, and 1.2 is three
    standard errors of the two sides' ratio."""
    s, psi, f, fixed = _current_system(l)
    nb = psi.shape[2]
    h = dftu.handle_for_system(s, nb)
    h.set_u(0, *fixed[0])
    t, fd = torch.from_numpy(psi).cuda(), torch.from_numpy(f).cuda()
    single = t.to(torch.complex64)

    def currents(x):
        return np.array([h.hubbard_current(x, torch.eye(nb, dtype=torch.float64, device="cuda")[b].reshape(1, 1, nb)) for b in range(nb)])

    def prepared(x):
        h.set_f64_mode(dftu.F64_NATIVE)
        h.project(x)
        h.occupations(fd)
        h.acbn0_uj()
        return currents(x)

    ref = prepared(t)
    h.set_f64_mode(dftu.F64_PAIR)
    pair = currents(t) - ref
    ref32 = prepared(single.to(torch.complex128))
    c64 = currents(single) - ref32
    for err, r, displaced in zip((pair, c64), (ref, ref32), DISPLACED_ERROR[l]):
        assert math.sqrt((err ** 2).mean() / (r ** 2).mean()) <= 1.2 * displaced
