"""The Hubbard current beyond the parity tests: occupation sums that are not Hermitian."""
import numpy as np
import pytest
import torch

from oracle import dftu_oracle as O
from paper_1711_08935_gb300 import dftu
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
