"""Explicit B_perp iterated as far as the entry point lets it (64 iterations), long past the rounding
floor of FP32, where the residual runs into the denormal numbers."""
import pytest
import torch

import oracle as O
from paper_2109_10277_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nx,ny,nz", [("fp32", 72, 40, 6), ("fp32", 256, 256, 3), ("tf32x3", 96, 130, 4)])
def test_explicit_at_the_iteration_limit(precision, nx, ny, nz):
    """Against the oracle: 1e-3, the bar of a recorded field of an FP32 sweep."""
    from paper_2109_10277_gb300 import hq
    g = dict(nx=nx, ny=ny, nzeta=nz, xmin=-4.0, xmax=4.0, ymin=-4.0, ymax=4.0, zeta_min=-0.6, zeta_max=0.6,
             n_pc_iter=64, bperp_solver="explicit")
    beam = I.random_beam(20_000, 0.4, 0.4, 0.3, 0.5)
    ref = O.sweep(O.GridSpec(**g), [O.as_beam(beam)], record=("bx", "by", "ez"))
    grid = hq.Grid(g, precision=precision)
    out = grid.alloc_out(("bx", "by", "ez"))
    grid.sweep([hq.Beam(beam)], out=out)
    assert grid.sync() == 0
    grid.close()
    for k in out:
        a, b = out[k].double().cpu(), ref.fields[k]
        dev = float(torch.linalg.norm(a - b) / torch.linalg.norm(b))
        print(f"{precision} {nx}x{ny} {k}: {dev:.1e}")
        assert dev <= 1e-3, k
