"""lat_decode of 16-bit states in its vector and element forms (N_x a multiple of 8 or not, lines shorter
than a warp, one value more than a warp's pass): stored values times their line's scale, exactly."""
import math

import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("nv, nx, ny", [(1, 7, 3), (3, 13, 5), (5, 100, 9), (5, 129, 4), (9, 257, 3),
                                        (9, 264, 3), (3, 1028, 2), (3, 2056, 2)])
def test_decode_is_code_times_line_scale(lat, dtype, nv, nx, ny):
    dt = I.choose_dt(2, nx, L, max(nv, 3), L, 1e-3)
    src = torch.tensor(I.random_initial((nv, nv, ny, nx), nx), dtype=torch.float32, device="cuda")
    src *= 2.0 ** torch.arange(ny, device="cuda")[:, None]  # lines of different scales
    lt = lat.Lattice(torch.zeros(src.shape, dtype=dtype, device="cuda"), d=2, nx=nx, ny=ny, nv=nv, L=L,
                     tau_p=math.inf, kappa=0.0, dt=dt)
    lt.encode(src)
    got, scales = lt.decode()
    want = lt.state.float() * scales.view(nv, nv, ny, 1)
    assert torch.equal(got, want)
    assert ((got - src).abs() <= src.abs().amax() * 2.0**-7).all()
    lt.close()
