"""Paths taken beyond the sizes of the other solver tests: the FP64 solve whose first pass forms the
sources at long rows, beams pushed beside the final pass, beams binned into many slices, and the third
right-hand side of the clustered FP32 solve."""
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


def peak_dev(a, b):
    return float((a - b).abs().max()) / float(b.abs().max())


@pytest.mark.parametrize("nx,ny", [(1024, 40), (2048, 24), (4096, 16)])
def test_fp64_sources_at_long_rows(hq, monkeypatch, nx, ny):
    """FP64, three rows of 1024 and 2048 points per block (768 threads, 224 KB of shared memory) and rows
    too long for that: against separate source kernels (HQ_SEPARATE_SRC=1), the same arithmetic apart from
    the unordered deposit sums, so within 1e-9 of each field's peak over these few slices."""
    g = I.scaled_grid(I.grid_params("linear64"), nx, ny, 6, zeta_min=-0.5, zeta_max=0.5)
    beam = I.random_beam(20_000, 0.4, 0.4, 0.2, 0.05)
    outs = []
    for mode in ("0", "1"):
        monkeypatch.setenv("HQ_SEPARATE_SRC", mode)
        grid = hq.Grid(g, precision="fp64")
        out = grid.alloc_out(("ez", "psi", "bx", "by", "bz"))
        grid.sweep([hq.Beam(beam)], out=out)
        grid.sync()
        outs.append(out)
        grid.close()
    for k in outs[0]:
        assert peak_dev(outs[0][k], outs[1][k]) <= 1e-9, k


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-9), ("fp32", 3e-5)])
def test_pushed_beams_beside_the_final_pass(hq, monkeypatch, precision, bar, graph):
    """Two pushed beams and witness sums with the push and deposit on a second stream against one stream
    (HQ_NO_FORK=1): the same work in the same order per particle, so that only unordered sums differ
    (1e-9 of the peak in FP64, the bf16x3 error of a solve, 3e-5, in FP32; momenta and positions by their
    change in the step)."""
    g = I.scaled_grid(I.grid_params("linear64"), 64, 48, 24, zeta_min=-2.0, zeta_max=2.0)
    arrays = [I.random_beam(20_000, 0.4, 0.4, 0.6, 0.5, zeta0=0.4, energy_spread=1e-3),
              I.random_beam(5_000, 0.2, 0.2, 0.3, 0.5, zeta0=-1.2, gamma=200.0, seed=7)]
    monkeypatch.setenv("HQ_NO_GRAPH", "0" if graph else "1")
    runs = []
    for mode in ("0", "1"):
        monkeypatch.setenv("HQ_NO_FORK", mode)
        grid = hq.Grid(g, precision=precision)
        out = grid.alloc_out(("ez", "psi", "bx", "by"))
        sums = torch.zeros(3, dtype=torch.float64, device="cuda")
        beams = [hq.Beam(a) for a in arrays]
        start = [{k: v.clone() for k, v in b.t.items()} for b in beams]
        for _ in range(2):   # (the second step bins the pushed beams)
            grid.sweep(beams, dt=6.0, out=out, witness=1, witness_sums=sums)
        grid.sync()
        runs.append((out, sums, [{k: b.t[k] - s[k] for k in ("x", "y", "zeta", "ux", "uy", "uz")}
                                 for b, s in zip(beams, start)]))
        grid.close()
    (fa, sa, ba), (fb, sb, bb) = runs
    for k in fa:
        assert peak_dev(fa[k], fb[k]) <= bar, k
    assert float(((sa - sb) / sb).abs().max()) <= bar
    for x, y in zip(ba, bb):
        for k in x:
            assert peak_dev(x[k], y[k]) <= bar, k


def test_binning_into_more_slices_than_a_block_counts(hq):
    """8192 slices are counted per block in shared memory, 8200 one particle at a time: a box that is
    eight slices longer at its tail has the same slices before them, bit for bit in deterministic mode."""
    outs = []
    for nz in (8192, 8200):
        g = dict(nx=16, ny=16, nzeta=nz, xmin=-2.0, xmax=2.0, ymin=-2.0, ymax=2.0, zeta_min=-nz / 1024.0, zeta_max=0.0,
                 n_pc_iter=1, deterministic=1)
        beam = I.random_beam(50_000, 0.5, 0.5, 3.0, 0.01, zeta0=-4.0)
        grid = hq.Grid(g, precision="fp64")
        out = grid.alloc_out(("jz", "ez"))
        grid.sweep([hq.Beam(beam)], out=out)
        grid.sync()
        outs.append(out)
        grid.close()
    for k in outs[0]:
        assert float(outs[0][k].abs().max()) > 0.0
        assert torch.equal(outs[0][k], outs[1][k][:8192]), k


@pytest.mark.parametrize("nx,ny", [(72, 48), (128, 128), (256, 256)])
def test_clustered_solve_of_three_right_hand_sides(hq, monkeypatch, nx, ny):
    """psi, Ez and Bz of FP32 sweeps against HQ_NO_CLUSTER=1, with a driver that is off centre, elongated
    and drifts sideways, so that Bz is no small residual of two large terms: the bf16x3 error of a solve,
    3e-5 of each field."""
    g = I.scaled_grid(I.grid_params("linear64"), nx, ny, 16, zeta_min=-1.0, zeta_max=1.0)
    beam = I.random_beam(20_000, 0.3, 0.7, 0.4, 0.5)
    beam["x"] = torch.as_tensor(beam["x"]) + 0.8
    beam["ux"] = torch.as_tensor(beam["ux"]) + 0.2 * torch.as_tensor(beam["uz"])
    outs = []
    for mode in ("0", "1"):
        monkeypatch.setenv("HQ_NO_CLUSTER", mode)
        grid = hq.Grid(g, precision="fp32")
        out = grid.alloc_out(("ez", "psi", "bz"))
        grid.sweep([hq.Beam(beam)], out=out)
        assert grid.sync() == 0
        outs.append(out)
        grid.close()
    for k in outs[0]:
        a, b = outs[0][k].double(), outs[1][k].double()
        dev = float(torch.linalg.norm(a - b) / torch.linalg.norm(b))
        print(f"{nx}x{ny} {k}: {dev:.1e}")
        assert dev <= 3e-5, k


@pytest.mark.parametrize("precision,nx,ny,nrhs", [("fp32", 64, 48, 2), ("fp32", 128, 128, 5), ("fp32", 256, 256, 2),
                                                  ("fp32", 512, 512, 3), ("fp32", 328, 200, 2), ("tf32x3", 96, 72, 3)])
def test_poisson_into_an_unaligned_array(hq, precision, nx, ny, nrhs):
    """FP32 hq_poisson_solve into an array that is not 16-byte aligned (its sources are copied ahead of the
    solve) against the solve into an aligned one: the same operand splits and products, so the same values
    within the error of a solve (3e-5 bf16x3, 8e-6 TF32x3)."""
    g = dict(nx=nx, ny=ny, nzeta=2, xmin=-4.0, xmax=4.0, ymin=-4.0, ymax=4.0, zeta_min=0.0, zeta_max=1.0)
    src = torch.randn(nrhs, ny, nx, device="cuda", generator=torch.Generator(device="cuda").manual_seed(nx))
    grid = hq.Grid(g, precision=precision)
    ref = grid.poisson_solve(src)
    n = src.numel()
    buf = torch.zeros(n + 2, device="cuda")
    hq._check(hq.load().hq_poisson_solve(grid.h, src.data_ptr(), buf.data_ptr() + 4, nrhs), grid.h)
    assert grid.sync() == 0
    grid.close()
    assert float(buf[0]) == 0.0 and float(buf[n + 1]) == 0.0
    got = buf[1:n + 1].view_as(ref)
    dev = float(torch.linalg.norm((got - ref).double()) / torch.linalg.norm(ref.double()))
    print(f"{precision} {nx}x{ny} x {nrhs}: {dev:.1e}")
    assert dev <= (3e-5 if precision == "fp32" else 8e-6)


@pytest.mark.parametrize("nx,ny,nrhs", [(65, 65, 1), (67, 70, 4), (409, 37, 1), (37, 128, 5), (514, 66, 2), (516, 520, 1),
                                        (96, 1030, 3), (24, 100, 3)])
def test_fp64_sums_of_any_length(hq, nx, ny, nrhs):
    """FP64 rows of other lengths than powers of two, at the edges of the kernel's blocks (four rows, 32
    outputs of a parity, 256 folded terms) and behind direct sums, against the oracle's dense sine sums:
    1e-12, the bar of a single linear operation."""
    from test_gpu_solvers import solve_case
    err, same = solve_case(hq, nx, ny, nrhs, "fp64")
    print(f"fp64 {nx}x{ny} x {nrhs}: {err:.1e}")
    assert err <= 1e-12 and same


@pytest.mark.parametrize("n,ppc,order,trial,final", [(256, 2, 3, 2, 2), (256, 2, 2, 2, 1), (128, 2, 3, 1, 1), (256, 1, 3, 1, 1)])
def test_profiled_launches(hq, n, ppc, order, trial, final):
    """hq_profile_read counts every kernel launch: with four particles per cell in one thread a slice's first
    trial pass is two kernels, and so is the cubic final pass."""
    nz, iters = 4, 3
    g = I.scaled_grid(I.grid_params("linear64"), n, n, nz, ppc_x=ppc, ppc_y=ppc, shape_order=order, n_pc_iter=iters,
                      zeta_min=-0.2, zeta_max=0.2)
    grid = hq.Grid(g, precision="fp32")
    beams = [hq.Beam(I.random_beam(2_000, 0.4, 0.4, 0.1, 0.5))]
    grid.profile(True)
    grid.sweep(beams)
    prof = grid.profile_read()
    grid.profile(False)
    grid.sync()
    grid.close()
    assert prof["trial"][1] == nz * (iters - 1 + trial)
    assert prof["final"][1] == nz * final


@pytest.mark.parametrize("n,nrhs", [(512, 2), (512, 5), (256, 5), (256, 2)])
def test_solves_beside_other_work(hq, n, nrhs):
    """FP32 solves whose products wait for single tiles, on one stream, beside a sweep on another that takes
    some of the SMs, so that a product's tiles end far apart: every result is bit for bit that of the solve
    alone (the sums of a solve have a fixed order)."""
    g = dict(nx=n, ny=n, nzeta=2, xmin=-4.0, xmax=4.0, ymin=-4.0, ymax=4.0, zeta_min=0.0, zeta_max=1.0)
    src = [torch.randn(nrhs, n, n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k)) for k in range(4)]
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s1):
        grid = hq.Grid(g, precision="fp32")
        ref = [grid.poisson_solve(s) for s in src]
        grid.sync()
    with torch.cuda.stream(s2):
        other = hq.Grid(I.scaled_grid(I.grid_params("linear64"), 96, 96, 48), precision="fp32")
        beams = [hq.Beam(I.random_beam(20_000, 0.4, 0.4, 1.0, 0.5))]
        other.sweep(beams)
        other.sync()
    torch.cuda.synchronize()
    got = []
    for _ in range(6):
        with torch.cuda.stream(s2):
            other.sweep(beams)
        with torch.cuda.stream(s1):
            got += [grid.poisson_solve(s) for _ in range(10) for s in src]
    assert grid.sync() == 0
    other.sync()
    torch.cuda.synchronize()
    for k, x in enumerate(got):
        assert torch.equal(x, ref[k % len(src)]), k
    grid.close()
    other.close()
