"""Options of one free-energy lattice taken together (viscosity tuning A, gravity, the droplet-collision
drive) against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2403_11167_gb300 import inputs
from helpers import gpu_context, oracle_params, pop_err
from test_gpu_tile import SHAPES

pytestmark = pytest.mark.gpu

FE = 1
F32, F64 = 0, 1
STEPS = 12


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("A,g", [(0.15, 0.0), (0.1, 1e-5), (0.0, 1e-5)])
@pytest.mark.parametrize("precision", [F64, F32])
def test_full_model_with_drive(precision, A, g):
    """Drive with another acceleration on either side of the split, so that the columns on the two sides of
    the periodic x edge are driven apart: the full model takes the velocity, and so the force, of a column's
    neighbours.  Every population after 12 steps at the bars of test_tile_edges_against_oracle (FP64 1e-11,
    FP32 5e-6 of its cell's density)."""
    for nx, ny in SHAPES:
        ctx, rp, th = gpu_context(FE, precision, nx, ny, a=0.25, Tr=0.85, tau_nu=0.9, body_fx=1e-5, body_fy=-2e-5, A=A)
        rho0 = inputs.random_field(nx, ny, th.rho_v * 1.5, th.rho_l * 0.8, seed=nx + ny)
        p = oracle_params(rp, th)
        if g:
            ctx.set_gravity(g, 0.0)
            p.g = g
        ctx.set_density(rho0)
        ctx.set_drive(5e-4, -3e-4, nx // 2, 2)
        p.drive_ax_lo, p.drive_ax_hi, p.drive_x_split = 5e-4, -3e-4, nx // 2
        f_ref = O.run_driven(FE, p, O.init_iwb(p, rho0), STEPS, t0=0, t_on=2)
        ctx.step(STEPS)
        err = pop_err(ctx.populations(), f_ref)
        assert err < (1e-11 if precision == F64 else 5e-6), (nx, ny, err)
        ctx.close()
