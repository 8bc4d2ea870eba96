"""Small 1D lattices advanced in one launch (csrc/line1d.cu) against one step per launch: the same
bits, in FP32 and FP64, from one column to more cells than threads, with columns left over for the
last blocks and with N_x below the cluster's block count; moments of a batch; the flow formed ahead
for the plain-load kernels (multi1d.cu, k_flow_steps) in FP64 and for any N_v."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def lattice(lat, dtype, nx, nv, flow, rows, one_by_one, seed=1):
    dt = I.choose_dt(1, nx, L, nv, L, 1e-3)
    f0 = torch.tensor(I.random_initial((nv, nx), seed), dtype=dtype, device="cuda")
    lt = lat.Lattice(f0, d=1, nx=nx, nv=nv, L=L, tau_p=L, kappa=1e-3, dt=dt)
    if one_by_one:
        lt.set_launch(kernel=1)
    fl = I.flow1d_inputs(seed + 1, rows)
    if flow == "modes":
        lt.set_flow_modes_1d(fl.k, fl.amp0[0], fl.tau_f, fl.sigma)
        lt.set_noise(fl.noise[:, 0, :])
    elif flow == "field":
        lt._u = torch.tensor(np.random.default_rng(3).standard_normal(nx), dtype=dtype,
                             device="cuda")
        lt.set_flow_field(lt._u)
    return lt


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("flow", ["modes", "field", "none"])
@pytest.mark.parametrize("nx,nv", [(1, 3), (5, 9), (17, 1), (64, 33), (256, 33), (333, 65),
                                   (450, 21), (130, 129), (1021, 17)])
def test_same_bits_as_one_step_per_launch(lat, dtype, flow, nx, nv):
    a = lattice(lat, dtype, nx, nv, flow, 30, False)
    b = lattice(lat, dtype, nx, nv, flow, 30, True)
    for n in (2, 7, 1, 10):
        a.step(n)
        b.step(n)
        assert torch.equal(a.state, b.state), n
    ca, *ma = a.step_moments(4)
    cb, *mb = b.step_moments(4)
    assert ca == cb == 0
    assert torch.equal(a.state, b.state) and a.steps_done == b.steps_done == 24
    for x, y in zip(ma[:3], mb[:3]):
        assert torch.equal(x, y)
    assert np.allclose(ma[3], mb[3], rtol=1e-12, atol=1e-12 * abs(mb[3][2]) + 1e-15)
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


def test_several_lattices_and_exhausted_noise(lat):
    sizes, nv = (64, 100, 37), 17
    out = []
    for one_by_one in (False, True):
        dt = np.array([I.choose_dt(1, s, L, nv, L, 1e-3) for s in sizes])
        f0 = np.concatenate([I.random_initial((nv, s), s).ravel() for s in sizes])
        e = lat.Ensemble(torch.tensor(f0, dtype=torch.float64, device="cuda"), nv=nv, nx=sizes,
                         L=np.full(3, L), tau_p=np.full(3, L), kappa=np.full(3, 1e-3), dt=dt)
        if one_by_one:
            e.set_launch(kernel=1)
        fl = I.flow1d_inputs(9, 8, n_inst=3)
        e.set_flow_modes(fl.k, fl.amp0, fl.tau_f, fl.sigma)
        e.set_noise(fl.noise)
        e.step(6)
        assert e.status() == lat.LAT_OK
        e.step(5)
        assert e.status() == lat.LAT_ENOISE
        out.append((e.state.clone(), e.get_state()))
        e.close()
    assert torch.equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("dtype,nx,nv", [(torch.float64, 5000, 33), (torch.float32, 6001, 21),
                                         (torch.float64, 3000, 49)])
def test_flow_formed_ahead_of_plain_steps(lat, dtype, nx, nv):
    a = lattice(lat, dtype, nx, nv, "modes", 20, False)
    b = lattice(lat, dtype, nx, nv, "modes", 20, True)
    for n in (1, 5, 7):
        a.step(n)
        b.step(n)
        assert torch.equal(a.state, b.state), n
    assert a.status() == b.status() == lat.LAT_OK
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()
