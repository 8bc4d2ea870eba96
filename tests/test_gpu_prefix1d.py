"""<rho_r^2> of 1D instances against exactly summed windows, at the edges of the prefix kernel's threads
(8 cells) and chunks (1024 cells).

Tolerance: rho >= 0, so a window sum is right to 3 u (u = 2^-53: the difference of two sums, of their
low parts, and their addition), r = m dx to 4 u, r^2 to 9 u, the mean to 11 u; 16 u allowed."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

L = 2 * math.pi


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("sizes", [(3, 7, 8, 9), (255, 256, 257, 264), (1023, 1024, 1025, 1032),
                                   (2047, 2049, 4097)])
def test_windows_of_edge_sizes(lat, sizes, dtype):
    nv, n = 5, len(sizes)
    rng = np.random.default_rng(7)
    f0 = rng.random(nv * sum(sizes)) * np.exp(6 * rng.random(nv * sum(sizes)))
    ens = lat.Ensemble(torch.tensor(f0, dtype=dtype, device="cuda"), nv=nv, nx=sizes,
                       L=np.full(n, L), tau_p=np.full(n, 1.0), kappa=np.zeros(n),
                       dt=np.full(n, 1e-3))
    widths = [1, 2, min(sizes)]
    got = ens.coarse_moment(widths)
    rho = ens.moments(per_cell=True)[1].cpu().numpy()
    at = 0
    for i, nx in enumerate(sizes):
        r, dx = rho[at:at + nx], L / nx
        at += nx
        for q, w in enumerate(widths):
            m = [math.fsum(r[(x + np.arange(w)) % nx]) * dx for x in range(nx)]
            want = math.fsum(v * v for v in m) / nx
            assert abs(got[i, q] - want) <= 16 * 2.0 ** -53 * want, (nx, w)
    ens.close()
