"""Flow velocities that are not numbers: every step kernel takes the drag of such a column as zero (the
maximum and minimum of a NaN and zero are zero), so the state stays finite, a column's neighbours in
a warp or tile do not matter, and the launch variants agree."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def field(n, seed, frac=0.2):
    u = 0.3 * np.random.default_rng(seed).standard_normal(n)
    u[np.random.default_rng(seed + 1).random(n) < frac] = np.nan
    return u


def lattice_1d(lat, dtype, scheme, nx, nv, kernel):
    mu = 2.0 / 3.0
    dt = I.choose_dt(1, nx, L, nv, L, 1e-3, cfl_factor=1.0 + mu)
    t = torch.tensor(I.random_initial((nv, nx), 3), dtype=dtype, device="cuda")
    lt = lat.Lattice(t, d=1, nx=nx, nv=nv, L=L, tau_p=L, kappa=1e-3, dt=dt)
    lt.set_scheme(scheme, mu)
    lt._u = torch.tensor(field(nx, 5), dtype=dtype, device="cuda")
    lt.set_flow_field(lt._u)
    if kernel:
        lt.set_launch(kernel=kernel)
    lt.step(12)
    out = lt.state.clone()
    assert lt.status() == lat.LAT_OK
    lt.close()
    return out


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("nx, nv", [(6000, 9), (1001, 33), (2048, 33), (2048, 65), (300, 17)])
def test_fp32_1d_batches_equal_single_steps(lat, scheme, nx, nv):
    a = lattice_1d(lat, torch.float32, scheme, nx, nv, 0)
    b = lattice_1d(lat, torch.float32, scheme, nx, nv, 1)
    assert torch.isfinite(b).all()
    assert torch.equal(a, b)


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("kernel", [0, 1])
def test_fp64_1d_takes_no_drag_from_it(lat, scheme, kernel):
    a = lattice_1d(lat, torch.float64, scheme, 300, 17, kernel)
    b = lattice_1d(lat, torch.float32, scheme, 300, 17, 1).double()
    assert torch.isfinite(a).all()
    assert (a - b).abs().sum() < 1e-5 * a.abs().sum()


def lattice_2d(lat, dtype, nv, kernel):
    nx, ny = 140, 12
    dt = I.choose_dt(2, nx, L, nv, L, 1e-3)
    t = torch.tensor(I.random_initial((nv, nv, ny, nx), 2), dtype=dtype, device="cuda")
    lt = lat.Lattice(t, d=2, nx=nx, ny=ny, nv=nv, L=L, tau_p=L, kappa=1e-3, dt=dt)
    lt._u = torch.tensor(field(2 * nx * ny, 7), dtype=dtype, device="cuda")
    lt.set_flow_field(lt._u)
    if kernel:
        lt.set_launch(kernel=kernel)
    lt.step(4)
    out = lt.state.clone()
    assert lt.status() == lat.LAT_OK
    lt.close()
    return out


@pytest.mark.parametrize("nv", [9, 17])
def test_fp64_2d_takes_no_drag_from_it(lat, nv):
    a = lattice_2d(lat, torch.float64, nv, 0)
    b = lattice_2d(lat, torch.float32, nv, 1).double()
    assert torch.isfinite(a).all()
    assert (a - b).abs().sum() < 1e-5 * a.abs().sum()
