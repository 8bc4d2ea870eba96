"""The two kernels of the 2D FP64 upwind step (tiles of cells with all velocities in shared memory, a
thread per cell), chosen by the grid: every N_v on grids of either side of the choice, ragged widths
and odd sizes, against the oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import lattice as O
from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi

# few cells and many, N_x on and off the tiles' and the blocks' widths (8, 16, 32 and 128 cells)
CASES = [(1, 40, 7), (1, 1030, 300), (3, 33, 20), (3, 384, 152), (5, 45, 31), (5, 256, 152),
         (9, 41, 17), (13, 39, 18), (13, 128, 300), (17, 35, 12), (17, 127, 152), (19, 37, 11),
         (19, 128, 152), (21, 43, 9), (21, 256, 60), (33, 21, 5), (33, 128, 60), (33, 128, 152)]


@pytest.mark.parametrize("nv, nx, ny", CASES)
def test_fp64_step_against_the_oracle(lat, nv, nx, ny):
    tau_p, kappa, steps = L, 1e-3, 2
    dx = L / nx
    dt = I.choose_dt(2, nx, L, max(nv, 3), tau_p, kappa)
    dv = dx / dt
    f0 = I.random_initial((nv, nv, ny, nx), nv + nx)
    fl = I.flow2d_inputs(9, steps, nx, ny, dx)
    lt = lat.Lattice(torch.tensor(f0, device="cuda"), d=2, nx=nx, ny=ny, nv=nv, L=L, tau_p=tau_p,
                     kappa=kappa, dt=dt)
    lt.set_flow_modes_2d(fl.kvec, fl.a, fl.phi0, fl.tau_f)
    lt.set_noise(fl.noise)
    lt.step(steps)
    got = lt.state.cpu().numpy()
    lt.close()
    want = O.run_2d(f0, steps, tau_p=tau_p, kappa=kappa, dt=dt, dv=dv, dx=dx, kvec=fl.kvec, a=fl.a,
                    phi0=fl.phi0, tau_f=fl.tau_f, noise=fl.noise)[0]
    assert np.abs(got - want).sum() <= 1e-13 * np.abs(want).sum()
