"""Kernels of a step start before the one before them has ended: a caller's own kernels between the calls, a second handle
on another stream, and a captured step whose capture forks and joins give the bits of the same calls made one at a time."""
import pytest
import torch

from paper_1711_08935_gb300 import dftu
from tests import _cases

pytestmark = pytest.mark.gpu


def _setup(dtype, nb, seed):
    s = _cases.overlapping_three_atoms()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.view_as_complex(torch.randn(s.nk, 1, nb, s.grid.npts, 2, generator=gen, device="cuda", dtype=torch.float64)).to(dtype)
    f = torch.rand(s.nk, 1, nb, generator=gen, device="cuda", dtype=torch.float64) / nb
    h = dftu.handle_for_system(s, nb)
    for I in range(3):
        h.set_u(I, 0.4, 0.05)
    return h, x / s.grid.npts ** 0.5, f


def _steps(h, psi, f, out, stream, wait, n):
    """n steps, the caller writing what the next call reads right before it and reading what it wrote right after it."""
    A = torch.zeros(3, dtype=torch.float64, device="cuda")
    for i in range(n):
        psi.mul_(0.98)
        h.project(psi, stream=stream)
        wait()
        f.mul_(0.97).add_(1e-3)
        h.occupations(f, stream=stream)
        wait()
        h.acbn0_uj(stream=stream)
        wait()
        out.copy_(psi)
        h.apply(out, stream=stream)
        wait()
        psi.add_(out, alpha=0.01)
        if psi.dtype == torch.complex128:
            A.fill_(0.1 * (i + 1))
            h.set_vector_potential(A, stream=stream)
            h.project(psi, stream=stream)
            wait()
            h.occupations(f, stream=stream)
            h.acbn0_uj(stream=stream)
            h.apply(psi, stream=stream)
            wait()
            h.set_vector_potential(None)
        h.taylor_steps(psi, f, 0.05, 2, stream=stream)
        wait()
    return psi, f, out


@pytest.mark.parametrize("nb", [7, 150])
def test_callers_kernels_between_the_calls_and_a_second_handle(nb):
    refs, runs = [], []
    for dtype, seed in ((torch.complex128, 1), (torch.complex64, 2)):
        h, x, f = _setup(dtype, nb, seed)
        refs.append(_steps(h, x, f, torch.empty_like(x), None, torch.cuda.synchronize, 6))
    for dtype, seed in ((torch.complex128, 1), (torch.complex64, 2)):
        h, x, f = _setup(dtype, nb, seed)
        runs.append((h, x, f, torch.empty_like(x), torch.cuda.Stream()))
    torch.cuda.synchronize()
    got = []
    for h, x, f, out, st in runs:   # both streams hold work at the same time
        with torch.cuda.stream(st):
            got.append(_steps(h, x, f, out, st, lambda: None, 6))
    torch.cuda.synchronize()
    for a, b in zip(refs, got):
        assert all(torch.equal(p, q) for p, q in zip(a, b))
    assert runs[0][0].sync_status() == dftu.DFTU_OK and runs[1][0].sync_status() == dftu.DFTU_OK


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_captured_step_with_a_fork_and_a_join(dtype):
    """A step on the capturing stream, a second handle's on a forked one, the caller's kernels between and a join."""
    pairs = []
    for _ in range(2):
        (ha, xa, fa), (hb, xb, fb) = _setup(dtype, 20, 3), _setup(dtype, 33, 4)
        pairs.append((ha, xa, fa, torch.empty_like(xa), hb, xb, fb))

    def step(ha, xa, fa, out, hb, xb, fb, main, side):
        xa.mul_(0.99)
        ha.project(xa, stream=main)
        side.wait_stream(main)
        with torch.cuda.stream(side):
            xb.mul_(0.99)
            hb.taylor_steps(xb, fb, 0.05, 2, stream=side)
        ha.occupations(fa, stream=main)
        ha.acbn0_uj(stream=main)
        out.copy_(xa)
        ha.apply(out, stream=main)
        main.wait_stream(side)
        hb.project(xb, stream=main)   # after the join: two predecessors
        xa.copy_(out)

    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(main):
        step(*pairs[0], main, side)   # first launches outside the capture, on both copies
        step(*pairs[1], main, side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        step(*pairs[1], main, side)
    torch.cuda.synchronize()
    for _ in range(4):
        with torch.cuda.stream(main):
            step(*pairs[0], main, side)
            graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(pairs[0], pairs[1]):
        if torch.is_tensor(a):
            assert torch.equal(a, b)
    assert (pairs[0][4].projections(33) == pairs[1][4].projections(33)).all()
