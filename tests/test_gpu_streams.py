"""Contexts on a non-blocking stream: the tables that set-up calls fill from host memory are there when
the kernels of that stream read them, also with earlier work still running on it.  The states equal
those of contexts on the default stream bit for bit."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def run_1d(lat, stream):
    sizes = [int(s) for s in np.random.default_rng(1).integers(40, 700, 2000)]
    n, nv = len(sizes), 9
    tau = np.full(n, L)
    dt = np.array([I.choose_dt(1, s, L, nv, L, 1e-3) for s in sizes])
    f0 = I.random_initial((nv * sum(sizes),), 3)
    with torch.cuda.stream(stream):
        t = torch.tensor(f0, dtype=torch.float32, device="cuda")
        torch.cuda._sleep(20_000_000)  # work ahead of the set-up calls
        ens = lat.Ensemble(t, nv=nv, nx=sizes, L=np.full(n, L), tau_p=tau,
                           kappa=np.full(n, 1e-3), dt=dt)
        fl = I.flow1d_inputs(5, 22, n_inst=n)
        for _ in range(3):
            ens.set_flow_modes(fl.k, fl.amp0, fl.tau_f, fl.sigma)
            ens.set_noise(fl.noise)
            ens.step(7)
        assert ens.status() == lat.LAT_OK
        out = ens.state.clone()
    stream.synchronize()
    ens.close()
    return out


def run_2d(lat, stream):
    nx, ny, nv = 136, 24, 9
    dt = I.choose_dt(2, nx, L, nv, L, 1e-3)
    with torch.cuda.stream(stream):
        t = torch.tensor(I.random_initial((nv, nv, ny, nx), 2), dtype=torch.float32, device="cuda")
        torch.cuda._sleep(20_000_000)
        lt = lat.Lattice(t, d=2, nx=nx, ny=ny, nv=nv, L=L, tau_p=L, kappa=1e-3, dt=dt)
        fl = I.flow2d_inputs(5, 9, nx, ny, L / nx)
        for _ in range(3):
            lt.set_flow_modes_2d(fl.kvec, fl.a, fl.phi0, fl.tau_f)
            lt.set_noise(fl.noise)
            lt.step(3)
        assert lt.status() == lat.LAT_OK
        out = lt.state.clone()
    stream.synchronize()
    lt.close()
    return out


@pytest.mark.parametrize("run", [run_1d, run_2d])
def test_non_blocking_stream_gives_the_default_streams_bits(lat, run):
    want = run(lat, torch.cuda.default_stream())
    for _ in range(3):
        assert torch.equal(run(lat, torch.cuda.Stream()), want)
