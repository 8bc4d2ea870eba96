"""Several steps per launch on chip (csrc/multi1d.cu) against one step per launch: the same bits.

A pinned launch kernel (lat_set_launch) takes one step per launch; the default takes five while as
many remain.  The shapes cover instances narrower than a tile and than the velocity lattice's reach,
ragged sizes (element copies) and multiples of four (bulk copies, wrapping windows), several tiles
per instance, step counts with and without single steps left over, every flow kind, and the noise
table running out within a launch."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def ensemble(lat, sizes, nv, flow, rows, one_by_one):
    n = len(sizes)
    tau = np.array([(0.1, 1.0, 10.0)[i % 3] * L for i in range(n)])
    dt = np.array([I.choose_dt(1, int(s), L, nv, t, 1e-3) for s, t in zip(sizes, tau)])
    f0 = np.concatenate([I.random_initial((nv, s), i).ravel() for i, s in enumerate(sizes)])
    ens = lat.Ensemble(torch.tensor(f0, dtype=torch.float32, device="cuda"), nv=nv, nx=sizes,
                       L=np.full(n, L), tau_p=tau, kappa=np.full(n, 1e-3), dt=dt)
    if one_by_one:
        ens.set_launch(kernel=1)
    fl = I.flow1d_inputs(5, rows, n_inst=n)
    if flow == "modes":
        ens.set_flow_modes(fl.k, fl.amp0, fl.tau_f, fl.sigma)
        ens.set_noise(fl.noise)
    elif flow == "frozen":
        ens.set_flow_modes(fl.k, fl.amp0, math.inf, 0.0)
    elif flow == "field":
        u = np.random.default_rng(3).standard_normal(int(np.sum(sizes)))
        ens._u = torch.tensor(u, dtype=torch.float32, device="cuda")
        ens.set_flow_field(ens._u)
    return ens


@pytest.mark.parametrize("nv", [9, 17, 33, 65])
@pytest.mark.parametrize("sizes", [(3, 40, 333, 1001), (132, 256, 1024, 2048)])
@pytest.mark.parametrize("flow", ["modes", "frozen", "field", "none"])
def test_same_bits_as_one_step_per_launch(lat, nv, sizes, flow):
    a = ensemble(lat, sizes, nv, flow, 40, False)
    b = ensemble(lat, sizes, nv, flow, 40, True)
    for n in (5, 12, 1, 20):
        a.step(n)
        b.step(n)
        assert torch.equal(a.state, b.state), (n, nv)
    sa, sb = a.status(), b.status()
    assert sa == sb
    assert a.steps_done == b.steps_done == 38
    ia, ib = a.get_state(), b.get_state()  # the amplitudes and the unused noise rows too
    assert np.array_equal(ia, ib)
    a.close()
    b.close()


def test_noise_running_out_within_a_launch(lat):
    a = ensemble(lat, (256, 300), 17, "modes", 7, False)
    b = ensemble(lat, (256, 300), 17, "modes", 7, True)
    a.step(10)
    b.step(10)
    assert torch.equal(a.state, b.state)
    assert a.status() == b.status() == lat.LAT_ENOISE
    a.close()
    b.close()


def test_autotuned_context_keeps_several_steps_and_bits(lat):
    a = ensemble(lat, (1024, 2048), 33, "modes", 20, False)
    b = ensemble(lat, (1024, 2048), 33, "modes", 20, True)
    a.autotune(reps=1)
    a.step(15)
    b.step(15)
    assert torch.equal(a.state, b.state)
    a.close()
    b.close()


def test_stalled_copies_time_out(lat):
    a = ensemble(lat, (256, 512), 33, "modes", 20, False)
    a.debug_stall(True)
    a.step(5)
    code = a.status()
    a.debug_stall(False)
    assert code == lat.LAT_ETIMEOUT
    a.step(1)
    assert a.status() == lat.LAT_OK
    a.close()
