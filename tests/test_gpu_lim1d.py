"""The flux-limited 1D step in two lanes per thread (csrc/lim1d.cu) against the kernels that take one
column per thread (a pinned launch kernel): the same values (a zero may have the other sign).

The shapes cover instances narrower than a tile and than the velocity lattice's reach, ragged sizes
(element copies) and multiples of four (bulk copies, wrapping windows), several tiles per instance,
the shortest and the longest column, every flow kind, flows that keep c a of one sign over the whole
column and that change it within it, and the noise table running out."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def ensemble(lat, sizes, nv, flow, rows, pinned, mu=2.0 / 3.0):
    n = len(sizes)
    tau = np.array([(0.1, 1.0, 10.0)[i % 3] * L for i in range(n)])
    J = (nv - 1) // 2
    dt = np.array([I.choose_dt(1, int(s), L, nv, t, 1e-4, cfl_factor=1.0 + mu)
                   for s, t in zip(sizes, tau)])
    f0 = np.concatenate([I.random_initial((nv, s), i).ravel() for i, s in enumerate(sizes)])
    ens = lat.Ensemble(torch.tensor(f0, dtype=torch.float32, device="cuda"), nv=nv, nx=sizes,
                       L=np.full(n, L), tau_p=tau, kappa=np.full(n, 1e-4), dt=dt)
    ens.set_scheme(lat.SCHEME_KOREN, mu)
    if pinned:
        ens.set_launch(kernel=1)
    fl = I.flow1d_inputs(5, rows, n_inst=n)
    if flow == "modes":
        ens.set_flow_modes(fl.k, fl.amp0, fl.tau_f, fl.sigma)
        ens.set_noise(fl.noise)
    elif flow == "frozen":
        ens.set_flow_modes(fl.k, fl.amp0, math.inf, 0.0)
    elif flow in ("field", "fast"):
        u = np.random.default_rng(3).standard_normal(int(np.sum(sizes)))
        if flow == "fast":  # |u| beyond the velocity lattice in half of the columns, both signs
            dv = np.concatenate([np.full(s, L / s / d) for s, d in zip(sizes, dt)])
            u = np.sign(np.roll(u, 1)) * np.where(np.arange(u.size) // 150 % 2, 1.2 * J, 0.4 * J) * dv
        ens._u = torch.tensor(u, dtype=torch.float32, device="cuda")
        ens.set_flow_field(ens._u)
    return ens


@pytest.mark.parametrize("nv", [9, 17, 33, 65])
@pytest.mark.parametrize("sizes", [(3, 40, 333, 1001), (132, 256, 1024, 2048)])
@pytest.mark.parametrize("flow", ["modes", "frozen", "field", "fast", "none"])
def test_same_values_as_one_column_per_thread(lat, nv, sizes, flow):
    a = ensemble(lat, sizes, nv, flow, 40, False)
    b = ensemble(lat, sizes, nv, flow, 40, True)
    for n in (1, 5, 6, 20):
        a.step(n)
        b.step(n)
        assert torch.equal(a.state, b.state), (n, nv)
    assert a.status() == b.status()
    assert a.steps_done == b.steps_done == 32
    a.close()
    b.close()


def test_noise_running_out(lat):
    a = ensemble(lat, (256, 300), 17, "modes", 7, False)
    b = ensemble(lat, (256, 300), 17, "modes", 7, True)
    a.step(10)
    b.step(10)
    assert torch.equal(a.state, b.state)
    assert a.status() == b.status() == lat.LAT_ENOISE
    a.close()
    b.close()
