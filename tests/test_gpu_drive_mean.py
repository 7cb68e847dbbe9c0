"""The mean density that driven tile steps take from the masses the step before stored (steps 2 .. 64 of
a captured graph; the first step and single steps reduce the populations)."""
import math

import numpy as np
import pytest

import oracle as O
from paper_2403_11167_gb300 import inputs
from helpers import gpu_context, oracle_params, pop_err
from test_gpu_tile import SHAPES

pytestmark = pytest.mark.gpu

PP, FE = 0, 1
F32, F64 = 0, 1
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("nx,ny", [(61, 7), (200, 100), (400, 300), (1022, 511)])
@pytest.mark.parametrize("model", [PP, FE])
def test_uniform_fp64_lattice_is_at_its_mean(model, nx, ny):
    """A uniform lattice: |rho - rho_ave| is rho_ave's rounding, and with a_x = 1 everywhere the momentum after
    one graph is its sum over the steps.  Per step at most half a unit, 2^(e - 56) with 2^e >= 4 / b, and three
    roundings of the scaling; in the first step the reduction's, 16 roundings of rho."""
    for frac in (0.0103, 0.0377, 0.31, 0.4321):
        ctx, rp, th = gpu_context(model, F64, nx, ny, a=0.25, Tr=0.85, tau_nu=0.9)
        rho = frac * 4.0 / rp.b
        ctx.set_density(np.full((ny, nx), rho))
        ctx.set_drive(1.0, 1.0, nx, -1)
        ctx.step(64)
        j = np.tensordot(CX, ctx.populations(), 1)
        e = math.frexp(4.0 / rp.b)[1]
        bound = 63 * (2.0 ** (e - 56) + 3 * 2.0**-53 * rho) + 16 * 2.0**-53 * rho
        assert np.max(np.abs(j)) <= bound, (frac, np.max(np.abs(j)) / bound)
        ctx.close()


@pytest.mark.parametrize("nx,ny", [(61, 7), (200, 100), (403, 301)])
@pytest.mark.parametrize("model", [PP, FE])
def test_uniform_fp32_lattice_is_at_its_mean(model, nx, ny):
    """The same in FP32, whose unit is below the rounding of every density that it meets: rho_ave rounds to
    rho, so only the first step's reduction (two roundings of rho) and the rounding of the populations (one
    of rho per step, against a_x = 100) leave momentum."""
    for frac in (0.00373, 0.0103, 0.31):
        ctx, rp, th = gpu_context(model, F32, nx, ny, a=0.25, Tr=0.85, tau_nu=0.9)
        rho = frac * 4.0 / rp.b
        ctx.set_density(np.full((ny, nx), rho))
        ctx.set_drive(100.0, 100.0, nx, -1)
        ctx.step(64)
        j = np.tensordot(CX, ctx.populations(), 1)
        bound = (2 * 100.0 + 64) * 2.0**-24 * rho
        assert np.max(np.abs(j)) <= bound, (frac, np.max(np.abs(j)) / bound)
        ctx.close()


@pytest.mark.parametrize("model,A", [(PP, 0.0), (FE, 0.0), (FE, 0.1)])
@pytest.mark.parametrize("precision", [F64, F32])
def test_graph_of_driven_steps(model, precision, A):
    """Switch-on after three steps, one graph of 64 and five single steps, over the tile edges, odd widths, shared
    rows and one-cell lattices.  FP64: the oracle, 1e-11 of a cell's density.  FP32: single steps, which reduce
    the populations every time; a rounding of 2^-24 per driven step, 5e-6.  (A cell left out of the mean of
    the largest lattice shifts a force of 5e-4 |rho - rho_ave| by more than either in 64 steps.)"""
    for nx, ny in SHAPES + [(29, 2), (50, 4), (101, 50), (256, 4), (30, 33)]:
        kw = dict(a=0.25, Tr=0.85, tau_nu=0.9, **({"A": A} if A else {}))
        ctx, rp, th = gpu_context(model, precision, nx, ny, **kw)
        rho0 = inputs.random_field(nx, ny, th.rho_v * 1.5, th.rho_l * 0.8, seed=nx + ny)
        ctx.set_density(rho0)
        ctx.set_drive(5e-4, -3e-4, nx // 2, 2)
        ctx.step(72)
        f = ctx.populations()
        ctx.close()
        if precision == F64:
            p = oracle_params(rp, th)
            p.drive_ax_lo, p.drive_ax_hi, p.drive_x_split = 5e-4, -3e-4, nx // 2
            err = pop_err(f, O.run_driven(model, p, O.init(model, rho0), 72, t0=0, t_on=2))
            assert err < 1e-11, (nx, ny, err)
        else:
            ctx, _, _ = gpu_context(model, precision, nx, ny, **kw)
            ctx.set_density(rho0)
            ctx.set_drive(5e-4, -3e-4, nx // 2, 2)
            for _ in range(72):
                ctx.step(1)
            err = pop_err(f, ctx.populations())
            ctx.close()
            assert err < 5e-6, (nx, ny, err)


@pytest.mark.parametrize("precision", [F64, F32])
@pytest.mark.parametrize("model,A", [(PP, 0.0), (FE, 0.0), (FE, 0.1)])
def test_divergence_reaches_the_mean(model, A, precision):
    """One cell of negative density (neither psi nor the logarithm exists) turns into NaN at the first step
    of a graph, two or three columns a step wider at each further one.  Its mean is NaN from the second step
    on and every force with it, in a graph as in single steps: no cell stays finite."""
    from paper_2403_11167_gb300 import lbm

    nx, ny = 500, 20
    for steps in ([64], [1] * 64):
        ctx, rp, th = gpu_context(model, precision, nx, ny, a=0.25, Tr=0.85, tau_nu=0.9, **({"A": A} if A else {}))
        ctx.set_density(inputs.random_field(nx, ny, th.rho_v * 1.5, th.rho_l * 0.8, seed=5))
        f = ctx.populations()
        f[:, 7, 9] *= -0.5
        ctx.set_populations(f)
        ctx.set_drive(5e-4, -3e-4, nx // 2, -1)
        for n in steps:
            ctx.step(n)
        assert np.all(np.isnan(ctx.populations().sum(0)))
        assert ctx.observables(0)["status"] == lbm.LBM_ERR_DIVERGED
        ctx.close()
