"""Per-cell moments and globals of 2D lattices in every form of the moment kernel (a thread per cell, a
block per 32 cells, two cells per thread) and every storage type: sizes on either side of the
choices, odd widths, last blocks with few cells, against FP64 sums of the stored state."""
import math

import numpy as np
import pytest
import torch

from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi
U32 = 2.0**-24

GRIDS = [(1, 50, 31), (3, 40, 29), (3, 512, 512), (5, 256, 130), (5, 600, 442), (9, 180, 180),
         (9, 512, 306), (9, 513, 307), (13, 184, 181), (13, 458, 341), (17, 186, 180), (17, 400, 392),
         (19, 202, 166), (19, 400, 392), (21, 150, 41), (21, 390, 402), (33, 64, 33), (33, 159, 80)]
CASES = [(d, *g) for g in GRIDS for d in ("f64", "f32", "f16", "bf16")
         if not (g[0] == 19 and d in ("f16", "bf16"))]
TYPES = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


@pytest.mark.parametrize("dtype, nv, nx, ny", CASES)
def test_per_cell_moments_and_globals(lat, dtype, nv, nx, ny):
    dt = I.choose_dt(2, nx, L, max(nv, 3), L, 1e-3)
    dx = L / nx
    dv = dx / dt
    gen = torch.Generator(device="cuda").manual_seed(nv * nx)
    src = torch.rand((nv, nv, ny, nx), generator=gen, device="cuda", dtype=torch.float64) + 0.1
    src *= 1.0 + torch.arange(nx, device="cuda") / nx  # neighbours, rows and velocities differ
    half = dtype in ("f16", "bf16")
    buf = torch.zeros(src.shape, dtype=TYPES[dtype], device="cuda") if half else src.to(TYPES[dtype])
    lt = lat.Lattice(buf, d=2, nx=nx, ny=ny, nv=nv, L=L, tau_p=math.inf, kappa=0.0, dt=dt)
    if half:
        lt.encode(src.float())
    f = (lt.decode()[0] if half else lt.state).double()
    code, rho, mv, mv2, glob = lt.moments()
    code2, *_, glob2 = lt.moments(per_cell=False)
    assert code == code2 == lat.LAT_OK
    v = (torch.arange(nv, device="cuda", dtype=torch.float64) - (nv - 1) // 2) * dv
    m0 = f.sum((0, 1))
    m1 = torch.einsum("jkyx,k->yx", f, v), torch.einsum("jkyx,j->yx", f, v)
    m2 = torch.einsum("jkyx,jk->yx", f, v[None, :] ** 2 + v[:, None] ** 2)
    a1 = torch.einsum("jkyx,k->yx", f, v.abs()), torch.einsum("jkyx,j->yx", f, v.abs())
    # FP64 sums of N_v^2 positive or signed terms; FP32 weighted sums: one rounding per value
    tol = 1e-13 if dtype == "f64" else nv * nv * U32
    assert ((rho.view(ny, nx) - m0 * dv**2).abs() <= 1e-13 * m0 * dv**2).all()
    for c in range(2):
        got = mv.view(2, ny, nx)[c]
        assert ((got - m1[c] / m0).abs() <= tol * a1[c] / m0 + 1e-300).all(), c
    assert ((mv2.view(ny, nx) - m2 / m0).abs() <= tol * m2 / m0 + 1e-300).all()
    w = (dx * dv) ** 2
    want = np.array([m0.sum().item(), m1[0].sum().item(), m1[1].sum().item(), m2.sum().item()]) * w
    scale = np.array([m0.sum().item(), a1[0].sum().item(), a1[1].sum().item(), m2.sum().item()]) * w
    for g in (glob, glob2):
        err = np.abs(g - want)
        assert err[0] <= 1e-12 * scale[0]
        assert (err[1:] <= 2 * tol * scale[1:] + 1e-300).all(), (err, scale)
    lt.close()
