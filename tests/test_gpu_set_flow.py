"""lat_set_flow between steps.  A field or no flow is set without waiting for the work in flight and
without memory changing hands (a program may hand over a new field before every step); tables that
depend on the wavenumbers follow every change of them."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi
SIZES = (300, 1024, 517, 40)


def ensemble(lat, dtype=torch.float32, nv=17, n=4, f0=None):
    sizes = [SIZES[i % 4] for i in range(n)]
    dt = np.array([I.choose_dt(1, s, L, nv, L, 1e-3) for s in sizes])
    if f0 is None:
        f0 = torch.tensor(I.random_initial((nv * sum(sizes),), 4), dtype=dtype, device="cuda")
    return lat.Ensemble(f0.clone(), nv=nv, nx=sizes, L=np.full(n, L), tau_p=np.full(n, L),
                        kappa=np.full(n, 1e-3), dt=dt)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_field_and_no_flow_are_set_without_waiting(lat, dtype):
    ens = ensemble(lat, dtype, n=40)
    u = [torch.full((int(ens.xoff[-1]),), 0.1 * q, dtype=dtype, device="cuda") for q in (1, 2)]
    for _ in range(2):  # first calls load kernels
        ens.set_flow_field(u[0])
        ens.set_flow_none()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    done = torch.cuda.Event()
    torch.cuda._sleep(2_000_000_000)  # about a second
    done.record()
    for q in range(6):
        ens.set_flow_field(u[q % 2])
        ens.set_flow_none()
    assert not done.query()
    assert torch.cuda.mem_get_info()[0] == free
    torch.cuda.synchronize()
    ens.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("scheme", [0, 1])
def test_tables_follow_the_wavenumbers(lat, dtype, scheme):
    ens = ensemble(lat, dtype)
    ens.set_scheme(scheme, 0.5)
    u = torch.tensor(0.3 * np.random.default_rng(2).standard_normal(int(ens.xoff[-1])), dtype=dtype,
                     device="cuda")
    rng = np.random.default_rng(3)
    for k in ((1, 2, 3), (4, 1), None, (4, 1), (4, 2), (9, 8, 7, 6, 5, 4), (1, 2, 3), (1, 2, 3)):
        before = ens.state.clone()
        amp = 0.2 * rng.standard_normal((4, 2 * len(k or (1,))))
        fresh = ensemble(lat, dtype, f0=before)
        fresh.set_scheme(scheme, 0.5)
        for e in (ens, fresh):
            if k is None:
                e.set_flow_field(u)
            else:
                e.set_flow_modes(np.array(k), amp, math.inf, 0.0)
            e.step(6)
        assert torch.equal(ens.state, fresh.state), k
        fresh.close()
    assert ens.status() == lat.LAT_OK
    ens.close()
