"""Members of a batch against the same calls made alone, bit for bit, at every size."""
import numpy as np
import pytest
import torch

from paper_1711_08935_gb300 import dftu
from tests import _cases

pytestmark = pytest.mark.gpu


def _wide_bands(s):
    """Enough bands that a tile reduce with a block per (k, spin, 32 bands, atom) takes more than four blocks per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 32 * (4 * sms // (s.nk * s.nspin * len(s.atoms)) + 1) + 5


@pytest.mark.parametrize("dtype,mode", [(torch.complex64, dftu.F64_PAIR), (torch.complex128, dftu.F64_PAIR), (torch.complex128, dftu.F64_NATIVE)])
def test_wide_members_of_a_batch_are_single_calls_bitwise(dtype, mode):
    """A member above and one below the size at which a single call reduces its tiles with a thread per state (three
    atoms with spheres of several images, two of them self-overlapping), bit for bit.  Complex128 pair projections take
    variant 1, the batch's shape, as single calls."""
    s = _cases.overlapping_three_atoms()
    gen = torch.Generator(device="cuda").manual_seed(3)
    single, member, psis, fs = [], [], [], []
    for nb in (_wide_bands(s), 7):
        x = torch.view_as_complex(torch.randn(s.nk, 1, nb, s.grid.npts, 2, generator=gen, device="cuda", dtype=torch.float64)).to(dtype)
        f = torch.rand(s.nk, 1, nb, generator=gen, device="cuda", dtype=torch.float64) / nb
        for hs in (single, member):
            h = dftu.handle_for_system(s, nb)
            h.set_f64_mode(mode)
            h.set_kernel_variant(0, 1)
            for I in range(3):
                h.set_u(I, 0.4, 0.05)
            hs.append(h)
        psis.append(x)
        fs.append(f)
    copies = [x.clone() for x in psis]
    for h, x, f in zip(single, psis, fs):
        h.project(x)
        h.occupations(f)
        h.acbn0_uj()
        h.apply(x)
    batch = dftu.Batch(member)
    batch.bind(copies, fs)
    batch.project()
    batch.occupations()
    batch.acbn0_uj()
    batch.apply()
    torch.cuda.synchronize()
    for a, b, x, y, f in zip(single, member, psis, copies, fs):
        assert np.array_equal(a.projections(f.shape[2]), b.projections(f.shape[2]))
        ra, rb = a.results(), b.results()
        assert all(np.array_equal(p, q) for p, q in zip(ra["n"], rb["n"])) and ra["EU"] == rb["EU"]
        assert torch.equal(x, y)
    batch.close()


def test_rebinding_with_other_band_counts():
    """Members of one capacity bound to ascending, then to descending band counts (the item lists follow the bound
    counts, longest first), complex64: every bind gives each member the bits of the same calls made alone."""
    s = _cases.overlapping_three_atoms()
    gen = torch.Generator(device="cuda").manual_seed(11)
    members = [dftu.handle_for_system(s, 90) for _ in range(3)]
    alone = dftu.handle_for_system(s, 90)
    for h in members + [alone]:
        for I in range(3):
            h.set_u(I, 0.4, 0.05)
    batch = dftu.Batch(members)
    for counts in ((3, 40, 90), (90, 40, 3), (40, 90, 3)):
        psis = [torch.view_as_complex(torch.randn(s.nk, 1, nb, s.grid.npts, 2, generator=gen, device="cuda")) for nb in counts]
        fs = [torch.rand(s.nk, 1, nb, generator=gen, device="cuda", dtype=torch.float64) / nb for nb in counts]
        refs = []
        for x, f in zip(psis, fs):
            y = x.clone()
            alone.project(y)
            alone.occupations(f)
            alone.acbn0_uj()
            alone.apply(y)
            refs.append((y, alone.results()["EU"]))
        batch.bind(psis, fs)
        batch.project()
        batch.occupations()
        batch.acbn0_uj()
        batch.apply()
        torch.cuda.synchronize()
        for h, x, (y, e) in zip(members, psis, refs):
            assert torch.equal(x, y) and h.results()["EU"] == e
    batch.close()
