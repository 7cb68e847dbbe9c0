"""The tile step kernel: tile edges of both precisions and every option against the FP64 oracle, and
the size rule that takes FP32 lattices to the strip kernels (the same bits on either side)."""
import numpy as np
import pytest

import oracle as O
from paper_2403_11167_gb300 import inputs
from helpers import gpu_context, oracle_params, pop_err

pytestmark = pytest.mark.gpu

PP, FE = 0, 1
F32, F64 = 0, 1
STEPS = 12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


# one cell, fewer columns than the halo, one column below / at / above a tile (FP32 60 and 56, FP64
# 30, 28 and 26 columns), two tiles, rows around the tile heights 1 .. 8
SHAPES = [(1, 1), (2, 5), (27, 1), (31, 9), (59, 4), (60, 8), (61, 7), (113, 17)]


@pytest.mark.parametrize("option", ["plain", "drive", "A", "walls", "onesided"])
@pytest.mark.parametrize("model", [PP, FE])
@pytest.mark.parametrize("precision", [F64, F32])
def test_tile_edges_against_oracle(model, precision, option):
    """Random densities: every population after 12 steps, FP64 within 1e-11 and FP32 within 5e-6 of
    its cell's density (12 steps of at most 3 roundings of 2^-24 on sums of up to a few densities)."""
    from paper_2403_11167_gb300 import lbm

    if model == PP and option in ("A", "onesided"):
        pytest.skip("free-energy terms")
    for nx, ny in SHAPES:
        walls = {"walls": 1, "onesided": 2}.get(option, 0)
        if walls and ny < 4:
            continue
        kw = dict(a=0.25, Tr=0.85, tau_nu=0.9, body_fx=1e-5, body_fy=0.0 if walls == 1 else -2e-5)
        if model == PP:
            kw.update(kappa_P=0.7, kappa_Li=-0.2)
        if option in ("A", "onesided"):
            kw["A"] = 0.1 if option == "A" or ny % 2 else 0.0
        ctx, rp, th = gpu_context(model, precision, nx, ny, walls=walls, **kw)
        rho0 = inputs.random_field(nx, ny, th.rho_v * 1.5, th.rho_l * 0.8, seed=nx + ny)
        p = oracle_params(rp, th, walls=walls)
        if option == "onesided":
            ctx.set_gravity(1e-5, 0.1, 0.5 * ny)
            p.g, p.rho_g, p.y_ref = 1e-5, 0.1, 0.5 * ny
        f0 = O.init_iwb(p, rho0) if option == "onesided" else O.init(model, rho0)
        ctx.set_density(rho0)
        if option == "drive":
            ctx.set_drive(5e-4, -3e-4, nx // 2, 2)
            p.drive_ax_lo, p.drive_ax_hi, p.drive_x_split = 5e-4, -3e-4, nx // 2
            f_ref = O.run_driven(model, p, f0, STEPS, t0=0, t_on=2)
        else:
            f_ref = O.run(model, p, f0, STEPS)
        ctx.step(STEPS)
        err = pop_err(ctx.populations(), f_ref)
        assert err < (1e-11 if precision == F64 else 5e-6), (nx, ny, err)
        assert ctx.observables(0)["status"] == lbm.LBM_OK
        ctx.close()


@pytest.mark.parametrize("model", [PP, FE])
@pytest.mark.parametrize("option", ["plain", "drive", "walls", "onesided"])
@pytest.mark.parametrize("nx,ny", [(31, 1), (29, 2), (50, 4), (101, 50), (28, 150), (200, 100), (256, 4), (57, 310)])
def test_shared_rows_match_unshared(model, option, nx, ny):
    """FP64 tiles with one or two rows left over by fours split them between two warps while there is one
    tile per SM; copies of the lattice side by side have more tiles and do not.  The same bits in every
    copy; with the drive the mean density is summed in another order, 1e-13 of the densities."""
    if option in ("walls", "onesided") and (ny < 4 or (option == "onesided" and model == PP)):
        pytest.skip("walls")
    walls = {"walls": 1, "onesided": 2}.get(option, 0)
    copies = -(-160 * 28 * 8 // (nx * ny)) + 1
    kw = dict(a=0.25, Tr=0.85, tau_nu=0.9, body_fx=1e-5, body_fy=-2e-5 if walls == 2 else 0.0)
    if model == PP:
        kw.update(kappa_P=0.7, kappa_Li=-0.2)
    got = []
    for k in (1, copies):
        ctx, rp, th = gpu_context(model, F64, nx * k, ny, walls=walls, **kw)
        rho0 = inputs.random_field(nx, ny, th.rho_v * 1.5, th.rho_l * 0.8, seed=nx + ny)
        ctx.set_density(np.tile(rho0, (1, k)))
        if option == "drive":
            ctx.set_drive(5e-4, 5e-4, nx * k, 2)
        ctx.step(STEPS)
        got.append(ctx.populations())
        ctx.close()
    small, big = got[0], got[1].reshape(9, ny, copies, nx)
    for c in range(copies):
        if option == "drive":
            assert np.max(np.abs(big[:, :, c] - small)) <= 1e-13 * np.max(small)
        else:
            assert np.array_equal(big[:, :, c], small), c


@pytest.mark.parametrize("Tr", [0.55, 0.7, 0.95])
def test_logarithm_over_the_phase_diagram(Tr):
    """FP64 free energy: ln rho from the vapour to the liquid density, every interval of the table and several
    exponents, against the oracle after two steps; 1e-12 of the cell's density (its exponents and the force
    stencil carry 1e-15)."""
    ctx, rp, th = gpu_context(FE, F64, 64, 40, a=0.25, Tr=Tr, tau_nu=0.9)
    x, y = np.meshgrid(np.arange(64), np.arange(40))
    t = 0.5 - 0.25 * (np.cos(2 * np.pi * x / 64) + np.cos(2 * np.pi * y / 40))
    rho0 = th.rho_v * (th.rho_l / th.rho_v) ** t
    f_ref = O.run(FE, oracle_params(rp, th), O.init(FE, rho0), 2)
    ctx.set_density(rho0)
    ctx.step(2)
    assert pop_err(ctx.populations(), f_ref) < 1e-12
    ctx.close()


@pytest.mark.parametrize("value", [-0.1, 0.0, np.nan, np.inf])
def test_no_logarithm_is_divergence(value):
    """A cell whose density has no logarithm ends in the divergence status, as with log()."""
    from paper_2403_11167_gb300 import lbm

    ctx, rp, th = gpu_context(FE, F64, 40, 20, a=0.25, Tr=0.85, tau_nu=0.9)
    ctx.set_density(np.full((20, 40), th.rho_l))
    f = ctx.populations()
    f[:, 7, 9] = value
    ctx.set_populations(f)
    ctx.step(3)
    assert ctx.observables(0)["status"] == lbm.LBM_ERR_DIVERGED
    ctx.close()


def _device_populations(ctx):
    import torch

    ctx.synchronize()
    ptr, pitch = ctx.device_populations()
    off = ptr - ctx.workspace.data_ptr()
    planes = ctx.workspace[off:off + 40 * pitch].view(torch.int32).view(10, pitch)
    n = ctx.nx * ctx.ny
    return planes[:9, :n].clone(), planes[9].view(torch.int16)[:n].clone()


@pytest.mark.parametrize("case", [
    (PP, 2196, 2192, {}), (PP, 8, 600400, {}), (PP, 600004, 8, {}), (PP, 4100, 1173, {}),
    (FE, 1684, 1680, {}), (FE, 8, 350400, {}), (FE, 300004, 10, {}), (FE, 484, 5801, {}),
    (FE, 1684, 1680, dict(A=0.15)), (FE, 300004, 10, dict(A=0.1)),
    (PP, 2284, 2280, dict(walls=1)), (FE, 1764, 1762, dict(walls=1)), (FE, 1764, 1762, dict(walls=2)),
    (PP, 1588, 1580, dict(drive=5e-4)), (FE, 1764, 1760, dict(drive=5e-4))])
def test_strips_match_tiles(case, monkeypatch):
    """Just above the size rule a lattice runs the strip kernels, with LBM_NO_TMA the tile kernel: the
    same bits, rest extensions included, after one graph of steps and some single ones (square, one
    narrow strip, few rows, uneven strips, walls, the drive).  The driven routes sum rho_ave in
    different units, which may change a force of 1e-4 by rounding: within 1e-6."""
    import torch

    model, nx, ny, opt = case
    walls = opt.get("walls", 0)
    kw = dict(a=0.25, Tr=0.85, tau_nu=0.8, body_fx=1e-6 if walls else 0.0, body_fy=-1e-6 if walls == 2 else 0.0)
    if "A" in opt:
        kw["A"] = opt["A"]
    rng = torch.Generator(device="cuda").manual_seed(nx)
    got = []
    for tiles in (False, True):
        if tiles:
            monkeypatch.setenv("LBM_NO_TMA", "1")
        ctx, rp, th = gpu_context(model, F32, nx, ny, walls=walls, **kw)
        if not tiles:
            rho = 0.5 * (th.rho_l + th.rho_v) * (0.98 + 0.04 * torch.rand((ny, nx), device="cuda", generator=rng))
            torch.cuda.synchronize()
        ctx.set_density_device(rho)
        if "drive" in opt:
            ctx.set_drive(opt["drive"], -opt["drive"], nx // 2, -1)
        ctx.step(67)
        got.append(_device_populations(ctx))
        ctx.close()
    (fa, qa), (fb, qb) = got
    if "drive" in opt:
        a, b = fa.view(torch.float32), fb.view(torch.float32)
        assert float((a - b).abs().max()) <= 1e-6 * float(b.abs().max())
    else:
        assert torch.equal(fa, fb) and torch.equal(qa, qb)


@pytest.mark.parametrize("model,A", [(PP, 0.0), (FE, 0.0), (FE, 0.1)])
def test_buffers_of_4_gb(model, A, monkeypatch):
    """From 4 GB a buffer's cells are not reached by 32-bit byte offsets: strips and tiles, the same bits
    after three steps (cells of a row above 2^31 bytes of a plane's offset included)."""
    import torch

    n = 10364
    assert n * n * 40 >= 2**32
    rng = torch.Generator(device="cuda").manual_seed(1)
    rho, want = None, None
    for tiles in (False, True):
        if tiles:
            monkeypatch.setenv("LBM_NO_TMA", "1")
        ctx, rp, th = gpu_context(model, F32, n, n, a=0.25, Tr=0.85, tau_nu=0.8, **(dict(A=A) if A else {}))
        if rho is None:
            rho = 0.5 * (th.rho_l + th.rho_v) * (0.98 + 0.04 * torch.rand((n, n), device="cuda", generator=rng))
            torch.cuda.synchronize()
        ctx.set_density_device(rho)
        ctx.step(3)
        got = _device_populations(ctx)
        ctx.close()
        if want is None:
            want = got
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_batch_lattice_of_4_gb():
    """A batch that holds a lattice of 4 GB takes the strip kernel with 64-bit addresses: the observables
    of single-lattice runs to FP64 rounding of their sums."""
    from paper_2403_11167_gb300 import lbm

    p = lbm.lbm_params_default(PP, precision=F32, a=0.25, Tr=0.85, tau_nu=0.8)
    _, th = lbm.lbm_resolve_params(p)
    specs, rhos = [], []
    for nx, ny in ((10364, 10364), (512, 64)):
        specs.append(dict(nx=nx, ny=ny, geometry=0, nsteps=3, params=p))
        rhos.append(inputs.random_field(nx, ny, 0.45 * (th.rho_l + th.rho_v), 0.55 * (th.rho_l + th.rho_v), seed=ny))
    b = lbm.Batch(specs, rhos)
    b.run()
    for got, s, r in zip(b.observables(), specs, rhos):
        ctx = lbm.Context(p, s["nx"], s["ny"])
        ctx.set_density(r)
        ctx.step(3)
        want = ctx.observables(0)
        ctx.close()
        for key in set(got) & set(want):
            assert got[key] == pytest.approx(want[key], rel=1e-9, abs=1e-12, nan_ok=True), key
    b.close()


def test_batch_strips_and_tiles_match_single_lattices():
    """A batch that starts above the batch's size rule (strips) and falls below it when the short lattices
    finish (tiles), some in the middle of a 64-step graph, with lattices narrower than a tile, of several
    tiles and of one: the same bits as single-lattice runs."""
    from paper_2403_11167_gb300 import lbm

    sizes = [(512, 512, 64), (512, 512, 70), (512, 512, 100), (512, 512, 130), (512, 512, 3), (512, 512, 64),
             (512, 512, 61), (512, 512, 129), (512, 512, 1), (512, 512, 0), (60, 76, 140), (64, 130, 131),
             (1200, 4, 66), (124, 37, 128), (8, 600, 65)]
    assert sum(nx * ny for nx, ny, _ in sizes) > 2500000
    specs, rhos = [], []
    for k, (nx, ny, steps) in enumerate(sizes):
        p = lbm.lbm_params_default(PP, precision=F32, a=0.25, Tr=0.8 + 0.005 * k, tau_nu=0.8, kappa_P=0.7, kappa_Li=-0.1)
        _, th = lbm.lbm_resolve_params(p)
        specs.append(dict(nx=nx, ny=ny, geometry=0, nsteps=steps, params=p))
        rhos.append(inputs.spinodal_noise(nx, ny, 0.5 * (th.rho_l + th.rho_v), 0.01, seed=k))
    b = lbm.Batch(specs, rhos)
    assert b.info()["n_resident"] == 0
    for _ in range(2):  # the second run starts again from the initial densities
        b.run()
        for i, (s, r) in enumerate(zip(specs, rhos)):
            ctx = lbm.Context(s["params"], s["nx"], s["ny"])
            ctx.set_density(r)
            ctx.step(s["nsteps"])
            assert np.array_equal(b.populations(i), ctx.populations()), (i, sizes[i])
            ctx.close()
    b.close()


@pytest.mark.parametrize("sizes", [
    [(1, 1), (1, 6), (5, 1), (3, 3), (31, 33), (101, 1)],                # odd widths, odd cell counts, one cell
    [(2, 1), (2, 3), (64, 4), (256, 4), (32, 32), (8, 141)],             # up to one pair per thread of 512
    [(43, 45), (1, 2047), (47, 49)], [(512, 4), (2, 1025), (40, 52)],    # the middle class, odd and even
    [(63, 65), (1, 4452), (61, 72)], [(64, 64), (4, 1113), (4452, 1)]])  # the largest, odd and even
def test_resident_lattices_match_single_lattices(sizes):
    """Resident lattices of every size class and parity of width, uneven step counts (0 and 1 among them):
    the same bits as single-lattice runs."""
    from paper_2403_11167_gb300 import lbm

    specs, rhos = [], []
    for k, (nx, ny) in enumerate(sizes):
        p = lbm.lbm_params_default(PP, precision=F32, a=0.25, Tr=0.8 + 0.01 * k, tau_nu=0.8, kappa_P=0.7, kappa_Li=-0.1,
                                   body_fx=1e-5)
        _, th = lbm.lbm_resolve_params(p)
        specs.append(dict(nx=nx, ny=ny, geometry=0, nsteps=(40, 0, 1, 33)[k % 4], params=p))
        rhos.append(inputs.spinodal_noise(nx, ny, 0.5 * (th.rho_l + th.rho_v), 0.01, seed=k))
    b = lbm.Batch(specs, rhos)
    assert b.info()["n_resident"] == len(sizes)
    b.run()
    for i, (s, r) in enumerate(zip(specs, rhos)):
        ctx = lbm.Context(s["params"], s["nx"], s["ny"])
        ctx.set_density(r)
        ctx.step(s["nsteps"])
        assert np.array_equal(b.populations(i), ctx.populations()), sizes[i]
        ctx.close()
    b.close()
