"""Poisson solves at the sizes where the solver's kernels change over (row lengths around the
direct sums, the fast transform and the tiled products; odd row counts; 1 to 5 right-hand sides),
and the launches that form their sources themselves against separate source kernels."""
import pytest
import torch

import oracle as O
from paper_2109_10277_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    from paper_2109_10277_gb300 import hq as _hq
    _hq.load()
    torch.cuda.set_device(0)
    return _hq


def rel(a, b):
    a, b = a.double().cpu(), b.double().cpu()
    return float(torch.linalg.norm(a - b) / (torch.linalg.norm(b) + 1e-300))


def solve_case(hq, nx, ny, nrhs, precision):
    g = dict(nx=nx, ny=ny, nzeta=2, xmin=-3.0, xmax=3.5, ymin=-2.0, ymax=2.0, zeta_min=0.0, zeta_max=1.0)
    grid = hq.Grid(g, precision=precision)
    gen = torch.Generator().manual_seed(nx * 7 + ny + nrhs)
    src = torch.randn(nrhs, ny, nx, generator=gen, dtype=torch.float64)
    if precision != "fp64":
        src = src.float()
    ref = [O.poisson_solve(O.GridSpec(**g), s.double()) for s in src]
    # the wall row and column of the sources are ignored, whatever they hold
    dirty = src.clone()
    dirty[:, 0, :] = float("nan")
    dirty[:, :, 0] = float("nan")
    dev = dirty.cuda()
    got = grid.poisson_solve(dev).cpu()
    assert bool((got[:, 0, :] == 0).all()) and bool((got[:, :, 0] == 0).all())
    hq._check(hq.load().hq_poisson_solve(grid.h, dev.data_ptr(), dev.data_ptr(), nrhs), grid.h)   # in place
    assert grid.sync() == 0
    again = dev.cpu()
    grid.close()
    return max(rel(a, b) for a, b in zip(got, ref)), bool((again == got).all())


@pytest.mark.parametrize("nx,ny,nrhs", [(8, 8, 1), (9, 64, 2), (63, 65, 5), (64, 66, 3), (128, 63, 2), (127, 128, 1),
                                        (256, 131, 3), (64, 1024, 2), (300, 200, 4), (2048, 16, 3)])
def test_poisson_fp64_sizes(hq, nx, ny, nrhs):
    """FP64 against the oracle's dense sine sums: 1e-12, the bar of a single linear operation."""
    err, same = solve_case(hq, nx, ny, nrhs, "fp64")
    print(f"fp64 {nx}x{ny} x {nrhs}: {err:.1e}")
    assert err <= 1e-12 and same


@pytest.mark.parametrize("nx,ny", [(48, 40), (128, 64), (64, 130)])
def test_fp64_sources_in_the_first_pass(hq, monkeypatch, nx, ny):
    """FP64 sweeps with the sources formed by the solve's first pass and the mixing done by its
    last, against separate kernels (HQ_SEPARATE_SRC=1): the same arithmetic apart from the
    unordered deposit sums, so within 1e-9 of each field's peak over these few slices."""
    g = I.scaled_grid(I.grid_params("linear64"), nx, ny, 12, zeta_min=-1.0, zeta_max=1.0)
    beam = I.random_beam(20_000, 0.4, 0.4, 0.4, 0.5)
    outs = []
    for mode in ("0", "1"):
        monkeypatch.setenv("HQ_SEPARATE_SRC", mode)
        grid = hq.Grid(dict(g, pc_residuals=1), precision="fp64")
        out = grid.alloc_out(("ez", "psi", "bx", "by", "bz"))
        grid.sweep([hq.Beam(beam)], out=out)
        assert grid.sync() == 0
        outs.append((out, grid.pc_residuals()))
        grid.close()
    for k in outs[0][0]:
        a, b = outs[0][0][k], outs[1][0][k]
        assert float((a - b).abs().max()) <= 1e-9 * float(b.abs().max()), k
    for a, b in zip(outs[0][1], outs[1][1]):
        assert abs(a - b) <= 1e-6 * b + 1e-12
