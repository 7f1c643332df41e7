"""Kernel variants asked for by number run as they are, also in calls small enough for the default to switch shape."""
import re

import numpy as np
import pytest
import torch

from paper_1711_08935_gb300 import dftu
from tests import _cases

pytestmark = pytest.mark.gpu


def _scatter_lanes(run):
    """Lanes per band (the second template argument) of every scatter kernel that run() launches; the kernel records
    come from the driver's profiling interface, which one process at a time can use."""
    for _ in range(3):
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            run()
            torch.cuda.synchronize()
        names = [e.key for e in prof.key_averages()]
        if any("dftu::" in n for n in names):
            return {int(m.group(1)) for m in (re.search(r"k_apply<\(?[^,]*, (?:\(int\))?(\d+)", n) for n in names) if m}
    pytest.skip("no kernel records from the profiler")


@pytest.mark.parametrize("dtype,which,lanes", [(torch.complex128, 2, {1: 8, 2: 16, 3: 8}), (torch.complex64, 3, {1: 8, 2: 16, 3: 8})])
def test_apply_variants_launch_the_shape_asked_for(dtype, which, lanes):
    s = _cases.overlapping_three_atoms()
    nb = 6
    psi = torch.from_numpy(_cases.states_np(s, nb, seed=1)).cuda().to(dtype)
    f = torch.rand(s.nk, 1, nb, device="cuda", dtype=torch.float64)
    h = dftu.handle_for_system(s, nb)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    h.project(psi)
    h.occupations(f)
    h.acbn0_uj()
    out = []
    for variant, q in [(0, 32)] + list(lanes.items()):
        h.set_kernel_variant(which, variant)
        h.apply(psi.clone())   # first launch of the shape outside the profile
        assert _scatter_lanes(lambda: h.apply(psi.clone())) == {q}, variant
        x = psi.clone()
        h.apply(x)
        out.append(x.cpu().numpy())
    tol = 1e-12 if dtype == torch.complex128 else 1e-6
    assert all(np.max(np.abs(x - out[0])) < tol * np.max(np.abs(out[0])) for x in out)
