"""The strip kernels on lattices below the size rule, which the library gives to the tile kernel: with
LBM_STRIPS set a context runs them wherever their row copies can be made (nx % 4 == 0).  Single,
ragged, uneven and thin strips against the tile kernel, bit for bit, and against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2403_11167_gb300 import inputs
from helpers import gpu_context, oracle_params, pop_err, rho_err
from test_gpu_tile import _device_populations

pytestmark = pytest.mark.gpu

PP, FE = 0, 1
F32 = 0


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


def _both(monkeypatch, model, nx, ny, rho0, steps, setup=lambda ctx, th: None, walls=0, **kw):
    """(populations and device bits) with strips and with tiles, and the resolved parameters."""
    out = []
    for strips in (True, False):
        if strips:
            monkeypatch.setenv("LBM_STRIPS", "1")
        else:
            monkeypatch.delenv("LBM_STRIPS")
        ctx, rp, th = gpu_context(model, F32, nx, ny, walls=walls, **kw)
        r = rho0(th) if callable(rho0) else rho0
        ctx.set_density(r)
        setup(ctx, th)
        ctx.step(steps)
        out.append((ctx.populations(), [a.cpu().numpy() for a in _device_populations(ctx)]))
        assert ctx.observables(0)["status"] == 0
        ctx.close()
    return out, rp, th, r


def _same_bits(out):
    (_, (fa, qa)), (_, (fb, qb)) = out
    assert np.array_equal(fa, fb) and np.array_equal(qa, qb)


# one tile and one strip, several strips, few rows, uneven strips, a last strip of 4 columns
@pytest.mark.parametrize("model", [PP, FE])
@pytest.mark.parametrize("shape", [(8, 4), (300, 200), (132, 7), (1024, 70), (244, 9), (484, 33), (4100, 6)])
def test_plain(model, shape, monkeypatch):
    """70 steps (a graph and single steps): the tile kernel's bits, and densities within 1e-5 of the oracle."""
    nx, ny = shape
    out, rp, th, rho0 = _both(monkeypatch, model, nx, ny,
                              lambda th: inputs.spinodal_noise(nx, ny, 0.5 * (th.rho_l + th.rho_v), 0.01, seed=7), 70,
                              Tr=0.85, tau_nu=0.8)
    _same_bits(out)
    f_ref = O.run(model, oracle_params(rp, th), O.init(model, rho0), 70)
    assert rho_err(out[0][0].sum(0), f_ref.sum(0)) < 1e-5


@pytest.mark.parametrize("model,walls", [(PP, 1), (FE, 1), (FE, 2)])
@pytest.mark.parametrize("shape", [(8, 6), (204, 61), (484, 33), (1024, 77)])
def test_walls(model, walls, shape, monkeypatch):
    """Strips over the whole lattice and tiles next to the walls, after 70 steps of a sine-perturbed channel
    with a body force: the bits of tiles alone, and densities within 1e-5 of the oracle."""
    nx, ny = shape
    out, rp, th, rho0 = _both(monkeypatch, model, nx, ny,
                              lambda th: inputs.plate_channel(nx, ny, th.rho_v, th.rho_l, amp=min(3.0, ny / 8)), 70,
                              walls=walls, a=0.25, Tr=0.8, tau_nu=0.9, body_fx=1e-5, body_fy=-2e-6)
    # the wall rows' slots that no step reads hold whatever the last kernel stored there
    assert np.array_equal(out[0][0], out[1][0])
    p = oracle_params(rp, th, walls=walls)
    rho_ref = O.macro(model, p, O.run(model, p, O.init(model, rho0), 70))[0]
    assert rho_err(out[0][0].sum(0), rho_ref) < 1e-5


@pytest.mark.parametrize("shape,A,g", [((8, 64), 0.2, 0.0), ((128, 96), 0.15, 0.0), ((456, 120), 0.15, 0.0),
                                       ((300, 64), 0.15, 2e-6), ((300, 64), 0.0, 2e-6), ((132, 7), 0.1, 1e-5)])
def test_full_free_energy(shape, A, g, monkeypatch):
    """Viscosity tuning and buoyancy (gravity with reference density 0) on a droplet, 100 steps: the tile
    kernel's bits, and populations within 1e-5 of the oracle."""
    nx, ny = shape
    out, rp, th, rho0 = _both(monkeypatch, FE, nx, ny, lambda th: inputs.droplet(nx, ny, ny / 4, th.rho_v, th.rho_l), 100,
                              setup=lambda ctx, th: ctx.set_gravity(g, 0.0) if g else None,
                              a=0.25, Tr=0.8, tau_nu=1.0, tau_e=0.9, A=A)
    _same_bits(out)
    p = oracle_params(rp, th)
    p.g = g
    f_ref = O.run(FE, p, O.init_iwb(p, rho0), 100)
    assert rho_err(out[0][0].sum(0), f_ref.sum(0)) < 1e-5
    assert pop_err(out[0][0], f_ref) < 1e-5


@pytest.mark.parametrize("model", [PP, FE])
@pytest.mark.parametrize("shape", [(256, 128), (484, 33), (132, 28)])
def test_drive(model, shape, monkeypatch):
    """A droplet pair driven from t = 0 for 200 steps: rho_ave from the masses that strips and tiles store in
    their own units, so within 1e-6 of the tile kernel, and densities within 1e-5 of the oracle."""
    nx, ny = shape
    out, rp, th, rho0 = _both(monkeypatch, model, nx, ny,
                              lambda th: inputs.two_droplets(nx, ny, [(nx / 4, ny / 2), (3 * nx / 4, ny / 2)], 0.23 * ny,
                                                             th.rho_v, th.rho_l), 200,
                              setup=lambda ctx, th: ctx.set_drive(5e-5, -5e-5, nx // 2, 0),
                              a=0.25, Tr=0.8, tau_nu=1.0, **({"match_kappa": 0.5} if model == PP else {}))
    assert pop_err(out[0][0], out[1][0]) < 1e-6
    p = oracle_params(rp, th)
    p.drive_ax_lo, p.drive_ax_hi, p.drive_x_split = 5e-5, -5e-5, nx // 2
    f_ref = O.run_driven(model, p, O.init(model, rho0), 200, t0=0, t_on=0)
    assert rho_err(out[0][0].sum(0), f_ref.sum(0)) < 1e-5


@pytest.mark.parametrize("model", [PP, FE])
def test_strips_after_a_timed_out_wait(model, monkeypatch):
    """After a bounded wait that ran out, the TMA-fed step still runs and reproduces a run made before."""
    from paper_2403_11167_gb300 import lbm

    monkeypatch.setenv("LBM_STRIPS", "1")
    nx, ny = 244, 33
    ctx, rp, th = gpu_context(model, F32, nx, ny, Tr=0.85, tau_nu=0.8)
    rho0 = inputs.spinodal_noise(nx, ny, 0.5 * (th.rho_l + th.rho_v), 0.01, seed=3)
    ctx.set_density(rho0)
    ctx.step(20)
    before = ctx.populations()
    assert lbm.lbm_selftest_bounded_wait(False, 500) == lbm.LBM_ERR_TIMEOUT
    ctx.set_density(rho0)
    ctx.step(20)
    assert np.array_equal(ctx.populations(), before)
    assert ctx.observables(0)["status"] == lbm.LBM_OK
    ctx.close()


def _kernels(fn):
    """Names of the kernels that fn launches (the first sessions of a process may record nothing)."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    for _ in range(4):
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            fn()
            torch.cuda.synchronize()
        names = " ".join(e.name for e in prof.events())
        if names:
            return names
    pytest.skip("no kernel records on this machine")


@pytest.mark.parametrize("model,kw,name", [(PP, {}, "pp_step_pair"), (FE, {}, "fe_step_pair"), (FE, {"A": 0.1}, "fe_iwb_pair")])
def test_which_kernels_run(model, kw, name, monkeypatch):
    """The variable changes the route (by the names of the kernels that a step launches)."""
    for strips in (True, False):
        if strips:
            monkeypatch.setenv("LBM_STRIPS", "1")
        else:
            monkeypatch.delenv("LBM_STRIPS")
        ctx, rp, th = gpu_context(model, F32, 64, 32, a=0.25, Tr=0.85, tau_nu=0.8, **kw)
        ctx.set_density(np.full((32, 64), th.rho_l))
        ran = _kernels(lambda: ctx.step(2))
        assert (name in ran) == strips and ("tile_step" in ran) != strips, ran
        ctx.close()
