"""Calls large enough for the production shapes of the streaming kernels, which small systems never reach (they take the
small-call shapes): the FP32-pair and complex64 kernels against native FP64 on the same GPU, whose kernels have one shape
and are pinned to the oracle elsewhere, and native FP64 at these sizes against the oracle."""
import numpy as np
import pytest
import torch

from oracle import dftu_oracle as O
from paper_1711_08935_gb300 import dftu
from tests import _cases

pytestmark = pytest.mark.gpu

A = (0.3, -0.2, 0.25)


def _system(rows):
    """Three overlapping atoms (two d shells and a p shell; tiles of very uneven size) with `rows` k-points."""
    s = _cases.overlapping_three_atoms()
    rng = np.random.default_rng(4)
    s.kpts = rng.uniform(-0.3, 0.3, (rows, 3))
    s.wk = np.full(rows, 1.0 / rows)
    return s


def _random_states(s, nb, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(s.nk, 1, nb, s.grid.npts, 2, generator=gen, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(x) / s.grid.npts ** 0.5


def _bounds(s, st, psi, eps):
    """[sum M]: eps times dV N max|phi_m| max|psi| over the sphere's N points, the scale of the terms that are summed.
    FP32 pairs: 2^-44 (2^-43 with the rotation by a phase, whose component grows by up to sqrt 2)."""
    top = float(psi.abs().max())
    return np.concatenate([eps * s.grid.dV * len(sm["idx"]) * np.abs(sm["phi"]).max(axis=0) * top for sm in st])


# band counts: 8 groups of 32, whole and ragged; more than 8; fewer, with 1-8, 9-16 and more bands left over
@pytest.mark.parametrize("nb", [256, 250, 257, 264, 272, 232, 33, 40, 41, 48, 65, 76, 8, 12, 20])
def test_pair_projections_of_large_calls(nb):
    """At least two waves of 1024-point tiles with one group each (24 rows of at least 13 such tiles), so the balanced
    shape runs: eight groups fixed, fewer at run time, and the ragged last groups of 16 and 32 lanes per band; the same
    under a vector potential, and the current's tables."""
    s = _system(max(24, (2 * torch.cuda.get_device_properties(0).multi_processor_count + 12) // 13))
    st = O.setup_atoms(s)
    psi = _random_states(s, nb, seed=nb)
    f = torch.rand(s.nk, 1, nb, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda", dtype=torch.float64) / nb
    h = dftu.handle_for_system(s, nb)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    for vec, eps in ((None, 2.0 ** -44), (torch.tensor(A, dtype=torch.float64, device="cuda"), 2.0 ** -43)):
        h.set_vector_potential(vec)
        p, J = [], []
        for mode in (dftu.F64_NATIVE, dftu.F64_PAIR):
            h.set_f64_mode(mode)
            h.project(psi)
            p.append(h.projections(nb))
        assert np.all(np.abs(p[0] - p[1]) <= _bounds(s, st, psi, eps))
        h.set_f64_mode(dftu.F64_NATIVE)
        h.project(psi)
        h.occupations(f)
        h.acbn0_uj()
        for mode in (dftu.F64_NATIVE, dftu.F64_PAIR):
            h.set_f64_mode(mode)
            J.append(h.hubbard_current(psi, f, per_atom=True)[1])
        # relative to the sum of the terms' moduli, here its Cauchy-Schwarz bound over random signs
        assert np.max(np.abs(J[0] - J[1])) <= 1e-11 * np.max(np.abs(J[0]))
    assert h.sync_status() == dftu.DFTU_OK


@pytest.mark.parametrize("nb", [16, 17, 32, 33, 40, 41])
def test_gauge_apply_at_the_band_counts_where_its_shape_changes(nb):
    """Both lane counts of the FP32-pair gauge scatter against native FP64, with enough rows for the production shape."""
    s = _system(3 * torch.cuda.get_device_properties(0).multi_processor_count // 2)
    psi = _random_states(s, nb, seed=nb)
    f = torch.rand(s.nk, 1, nb, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda", dtype=torch.float64) / nb
    h = dftu.handle_for_system(s, nb)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    h.set_vector_potential(torch.tensor(A, dtype=torch.float64, device="cuda"))
    out = []
    h.set_f64_mode(dftu.F64_NATIVE)
    h.project(psi)
    h.occupations(f)
    h.acbn0_uj()
    for mode in (dftu.F64_NATIVE, dftu.F64_PAIR):
        h.set_f64_mode(mode)
        x = psi.clone()
        h.apply(x)
        out.append(x)
    assert float((out[0] - out[1]).abs().max()) < 1e-12 * float(out[0].abs().max())
