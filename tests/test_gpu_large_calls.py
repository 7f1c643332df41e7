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


def _apply_bands(s, extra):
    """Bands for which every colour of an apply, even one with a single tile, passes the small-call threshold (half of
    three blocks per SM, a block per tile, row and 64 bands), and `extra` more."""
    chunks = -(-3 * torch.cuda.get_device_properties(0).multi_processor_count // (2 * s.nk * s.nspin))
    return 64 * chunks + extra


def _subset(s, ks):
    sub = _cases.overlapping_three_atoms()
    sub.kpts, sub.wk = s.kpts[ks], s.wk[ks]
    return sub


# whole groups, and 5 or 13 bands more (ragged groups of 16 and 32 bands)
@pytest.mark.parametrize("extra", [0, 5, 13])
@pytest.mark.parametrize("kind", ["pair", "native", "complex64"])
@pytest.mark.parametrize("vector_potential", [None, A])
def test_apply_of_large_calls_matches_oracle(kind, extra, vector_potential):
    """The production shapes of the scatter, plain and with the gauge phases, in the three arithmetics: bands of the
    first, a middle and the last group at two k-points against the oracle's apply with the handle's own potential."""
    s = _system(48)
    nb = _apply_bands(s, extra)
    st = O.setup_atoms(s)
    dtype = torch.complex64 if kind == "complex64" else torch.complex128
    psi = _random_states(s, nb, seed=extra).to(dtype)
    f = torch.rand(s.nk, 1, nb, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda", dtype=torch.float64) / nb
    h = dftu.handle_for_system(s, nb)
    h.set_f64_mode(dftu.F64_NATIVE if kind == "native" else dftu.F64_PAIR)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    if vector_potential is not None:
        h.set_vector_potential(torch.tensor(vector_potential, dtype=torch.float64, device="cuda"))
    ks, bands = [0, 47], [0, 1, nb // 2, nb - 14, nb - 6, nb - 2, nb - 1]
    before = psi[ks][:, :, bands].to(torch.complex128).cpu().numpy()
    h.project(psi)
    h.occupations(f)
    h.acbn0_uj()
    h.apply(psi)
    got = psi[ks][:, :, bands].to(torch.complex128).cpu().numpy()
    V = [0.35 * (0.5 * np.eye(n.shape[-1]) - n.transpose(0, 2, 1)) for n in h.results()["n"]]
    sub, vec = _subset(s, ks), np.array(vector_potential or (0.0, 0.0, 0.0))
    ref = O.apply_gauge(sub, st, before, O.project_gauge(sub, st, before, vec), V, vec)
    assert np.max(np.abs(got - ref)) < (1e-6 if kind == "complex64" else 1e-12) * np.max(np.abs(ref))
    assert h.sync_status() == dftu.DFTU_OK


@pytest.mark.parametrize("extra", [0, 5])
def test_fused_real_time_steps_of_large_calls_match_oracle(extra):
    """Three fused complex64 steps whose scatters all take the production shape, on tiles of both kinds (spheres that
    overlap each other and their own images): states, projections and the handle's potential against the oracle's
    steps, on sampled bands with the potential of every step formed from all of them by single native FP64 steps."""
    s = _system(48)
    nb = _apply_bands(s, extra)
    st = O.setup_atoms(s)
    psi = _random_states(s, nb, seed=7 + extra).to(torch.complex64)
    f = torch.rand(s.nk, 1, nb, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda", dtype=torch.float64) / nb
    fused, native = dftu.handle_for_system(s, nb), dftu.handle_for_system(s, nb)
    native.set_f64_mode(dftu.F64_NATIVE)
    for h in (fused, native):
        for I in range(3):
            h.set_u(I, 0.4, 0.05)
    ks, bands, dt = [0, 47], [0, nb // 2, nb - 6, nb - 2, nb - 1], 0.5
    sub = _subset(s, ks)
    ref = psi[ks][:, :, bands].to(torch.complex128).cpu().numpy()
    t = psi.to(torch.complex128)
    fused.taylor_steps(psi, f, dt, 3)
    for _ in range(3):
        native.taylor_step(t, None, f, dt)
        V = [0.35 * (0.5 * np.eye(n.shape[-1]) - n.transpose(0, 2, 1)) for n in native.results()["n"]]
        term = out = ref
        for j in range(1, 5):
            term = O.apply(sub, st, np.zeros_like(term), O.project(sub, st, term), V, -1j * dt / j)
            out = out + term
        ref = out
    assert np.max(np.abs(t[ks][:, :, bands].cpu().numpy() - ref)) < 1e-11 * np.max(np.abs(ref))
    got = psi[ks][:, :, bands].to(torch.complex128).cpu().numpy()
    assert np.max(np.abs(got - ref)) < 2e-6 * np.max(np.abs(ref))
    assert float((psi.to(torch.complex128) - t).abs().max()) < 2e-6 * float(t.abs().max())
    p = fused.projections(nb)[ks][:, bands]
    p_ref = np.concatenate([x[:, 0] for x in O.project(sub, st, got)], axis=-1)
    assert np.max(np.abs(p - p_ref)) < 2e-6 * np.max(np.abs(p_ref))
    for a, b in zip(fused.results()["n"], native.results()["n"]):
        assert np.max(np.abs(a - b)) < 1e-6 * max(1.0, np.max(np.abs(b)))
    assert fused.sync_status() == dftu.DFTU_OK


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


@pytest.mark.parametrize("dtype,which,tol", [(torch.complex128, 2, 1e-12), (torch.complex64, 3, 1e-6)])
def test_every_apply_variant_on_a_large_call(dtype, which, tol):
    """Small calls run one shape whatever the variant; here every colour is large enough for the shape asked for, with
    a ragged last group, against native FP64 on the same states."""
    s = _system(48)
    nb = _apply_bands(s, 37)
    psi = _random_states(s, nb, seed=13).to(dtype)
    f = torch.rand(s.nk, 1, nb, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda", dtype=torch.float64) / nb
    h = dftu.handle_for_system(s, nb)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    h.set_f64_mode(dftu.F64_NATIVE)
    ref = psi.to(torch.complex128, copy=True)
    h.project(ref)
    h.occupations(f)
    h.acbn0_uj()
    h.apply(ref)
    h.set_f64_mode(dftu.F64_PAIR)
    top = float(ref.abs().max())
    for variant in range(h.lib.dftu_kernel_variants(which)):
        h.set_kernel_variant(which, variant)
        x = psi.clone()
        h.apply(x)
        assert float((x.to(torch.complex128) - ref).abs().max()) < tol * top, variant
