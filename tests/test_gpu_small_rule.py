"""Which 1D lattices take a batch of steps in one cluster launch: only those for which that is faster
than a launch per step (or per five steps).  The sizes are some where the cluster's blocks have many
columns for each velocity, and where more clusters are asked for than run at a time; the bits are
the same either way."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


def ensemble(lat, dtype, nx, n, nv, flow, kernel):
    dt = I.choose_dt(1, nx, L, nv, L, 1e-4)
    f0 = torch.tensor(I.random_initial((nv * nx * n,), 3), dtype=dtype, device="cuda")
    ens = lat.Ensemble(f0, nv=nv, nx=[nx] * n, L=np.full(n, L), tau_p=np.full(n, L),
                       kappa=np.full(n, 1e-4), dt=np.full(n, dt))
    if flow == "modes":
        fl = I.flow1d_inputs(5, 1, n_inst=n)
        ens.set_flow_modes(fl.k, fl.amp0, math.inf, 0.0)
    if kernel:
        ens.set_launch(kernel=kernel)
    return ens


def best_us(ens, n):
    out = math.inf
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(20):
        a.record()
        ens.step(n)
        b.record()
        b.synchronize()
        out = min(out, 1e3 * a.elapsed_time(b))
    return out


@pytest.mark.parametrize("dtype, nx, n, nv, flow", [
    (torch.float32, 8888, 1, 3, "modes"),
    (torch.float32, 3000, 8, 9, "modes"),
    (torch.float64, 8888, 1, 5, "modes"),
    (torch.float64, 8888, 8, 5, "modes"),
    (torch.float64, 4096, 4, 9, "none"),
])
def test_batches_are_not_slower_than_single_steps(lat, dtype, nx, n, nv, flow):
    a = ensemble(lat, dtype, nx, n, nv, flow, 0)
    b = ensemble(lat, dtype, nx, n, nv, flow, 1)
    a.step(10)
    b.step(10)
    assert torch.equal(a.state, b.state)
    ta, tb = best_us(a, 10), best_us(b, 10)
    assert ta < 1.25 * tb, (ta, tb)
    a.close()
    b.close()
