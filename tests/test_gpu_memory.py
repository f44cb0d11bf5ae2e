"""The trial cache (52 or 128 bytes per plasma particle) never makes a call fail that fits without it:
it is left out of a grid that does not fit with it, and given back for the reverse sweep's storage."""
import gc

import pytest
import torch

from paper_2109_10277_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    from paper_2109_10277_gb300 import hq as _hq
    _hq.load()
    torch.cuda.set_device(0)
    return _hq


def free_bytes():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def leave(nbytes):
    """A tensor that leaves about nbytes of device memory free."""
    return torch.empty(free_bytes() - nbytes, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("precision,cache", [("fp64", 128), ("fp32", 52)])
def test_grid_without_room_for_the_cache(hq, monkeypatch, precision, cache):
    """Free memory between what the grid needs without the cache and with it: it is created, and its
    sweep is that of HQ_NO_F4CACHE=1 (FP64 1e-9 of each field's peak, FP32 3e-5: unordered sums)."""
    g = I.scaled_grid(I.grid_params("linear64"), 1024, 1024, 3, ppc_x=2, ppc_y=2, zeta_min=-0.2, zeta_max=0.2)
    nbytes = cache * 4 * 1024 * 1024
    beam = I.random_beam(20_000, 0.4, 0.4, 0.1, 0.5)

    def sweep(grid):
        out = grid.alloc_out(("ez", "psi", "bx"))
        grid.sweep([hq.Beam(beam)], out=out)
        grid.sync()
        return {k: v.cpu() for k, v in out.items()}

    monkeypatch.setenv("HQ_NO_F4CACHE", "1")
    start = free_bytes()
    grid = hq.Grid(g, precision=precision)
    need = start - free_bytes()
    ref = sweep(grid)
    grid.close()
    monkeypatch.delenv("HQ_NO_F4CACHE")
    start = free_bytes()
    grid = hq.Grid(g, precision=precision)
    assert start - free_bytes() >= need + 0.9 * nbytes   # (it fits: the cache is there)
    grid.close()
    filler = leave(need + nbytes // 2)
    grid = hq.Grid(g, precision=precision)
    del filler
    torch.cuda.empty_cache()
    got = sweep(grid)
    grid.close()
    for k in ref:
        tol = 1e-9 if precision == "fp64" else 3e-5
        assert float((got[k] - ref[k]).abs().max()) <= tol * float(ref[k].abs().max()), k


def test_adjoint_takes_the_cache_back(hq):
    """Free memory for the reverse sweep's storage only without the cache: the gradients come, and are
    those of a grid with room (FP64, 1e-9: unordered sums), before and after a plain sweep."""
    g = I.scaled_grid(I.grid_params("linear64"), 512, 512, 4, ppc_x=2, ppc_y=2, zeta_min=-0.2, zeta_max=0.2)
    nbytes = 128 * 4 * 512 * 512
    d = hq.Beam(I.random_beam(20_000, 0.4, 0.4, 0.1, 0.5))
    w = hq.Beam(I.random_beam(5_000, 0.2, 0.2, 0.1, 0.5))

    def grads(grid):
        n0 = torch.ones((), dtype=torch.float64, device="cuda", requires_grad=True)
        ws = [b.t["w"].clone().requires_grad_() for b in (d, w)]
        loss = hq.SweepLoss.apply(grid, [d, w], 1, "mean", 2, n0, torch.zeros(0, dtype=torch.float64, device="cuda"), *ws)
        return [x.cpu() for x in torch.autograd.grad(loss, [n0, *ws])]

    for _ in range(2):   # (the first one also loads the kernels)
        grid = hq.Grid(g, precision="fp64")
        before = free_bytes()
        ref = grads(grid)
        need = before - free_bytes()
        grid.close()
    grid = hq.Grid(g, precision="fp64")
    grid.sweep([d, w])   # (a captured sweep that uses the cache)
    filler = leave(need - nbytes // 2)
    got = grads(grid)
    del filler
    torch.cuda.empty_cache()
    grid.sweep([d, w])
    again = grads(grid)
    assert grid.sync() == 0
    grid.close()
    for a, b, c in zip(got, again, ref):
        assert float((a - c).abs().max()) <= 1e-9 * float(c.abs().max())
        assert float((b - c).abs().max()) <= 1e-9 * float(c.abs().max())


def test_refused_allocation_is_reported_once(hq):
    """A grid, and a reverse sweep's storage, that do not fit are refused with HQ_ERR_OOM; the calls after
    that succeed once there is room."""
    g = I.scaled_grid(I.grid_params("linear64"), 256, 256, 4, ppc_x=4, ppc_y=4, zeta_min=-0.2, zeta_max=0.2)
    beam = hq.Beam(I.random_beam(2_000, 0.4, 0.4, 0.1, 0.5))
    start = free_bytes()
    grid = hq.Grid(g, precision="fp64")
    need = start - free_bytes()
    grid.close()
    filler = leave(need // 4)
    with pytest.raises(hq.HQError) as e:
        hq.Grid(g, precision="fp64")
    assert e.value.status == 3
    del filler
    torch.cuda.empty_cache()
    grid = hq.Grid(g, precision="fp64")
    sums = torch.zeros(3, dtype=torch.float64, device="cuda")
    filler = leave(need // 2)
    with pytest.raises(hq.HQError) as e:
        grid.forward_ckpt([beam], 0, sums, 1)
    assert e.value.status == 3
    del filler
    torch.cuda.empty_cache()
    grid.sweep([beam])
    grid.forward_ckpt([beam], 0, sums, 1)
    assert grid.sync() == 0
    grid.close()
