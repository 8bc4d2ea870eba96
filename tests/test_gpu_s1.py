"""S1 over groups of separations: any number of them (groups of eight, four, two and one), instances
of one and of many runs of columns, several cells per thread, against the oracle; scratch that grows
with the columns, not with instances times the longest one; and a single separation that does not
pay for eight."""
import math

import numpy as np
import pytest
import torch

from oracle import observables as B
from paper_1508_02899_gb300 import inputs as I

pytestmark = pytest.mark.gpu

L = 2 * math.pi
U32 = 2.0**-24


def ensemble(lat, sizes, nv, dtype, seed=4):
    n = len(sizes)
    dts = {s: I.choose_dt(1, int(s), L, nv, L, 1e-4) for s in set(sizes)}
    dt = np.array([dts[s] for s in sizes])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f0 = torch.rand(nv * int(sum(sizes)), generator=gen, dtype=torch.float64, device="cuda")
    ens = lat.Ensemble(f0.to(dtype), nv=nv, nx=sizes, L=np.full(n, L), tau_p=np.full(n, L),
                       kappa=np.full(n, 1e-4), dt=dt)
    return ens, np.array([L / s / d for s, d in zip(sizes, dt)])


def check(ens, dv, nv, dtype, seps, instances):
    num, den = ens.s1(seps)
    for k in instances:
        f = ens.instance_view(k).double().cpu().numpy()
        want_n, want_d = B.s1_terms(f, dv[k], seps)
        np.testing.assert_allclose(den[k], want_d, rtol=1e-12)
        # FP32: four running sums of positive terms, each off by about N_v u
        np.testing.assert_allclose(num[k], want_n, rtol=1e-12 if dtype == torch.float64
                                   else 4 * nv * U32)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("ns", [1, 2, 3, 7, 8, 9, 17])
def test_any_number_of_separations(lat, dtype, ns):
    nv, sizes = 9, (127, 129, 20, 500, 128, 19)
    ens, dv = ensemble(lat, sizes, nv, dtype)
    check(ens, dv, nv, dtype, [(5 * q) % 19 for q in range(ns)], range(len(sizes)))
    ens.close()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("columns", [700_000, 2_600_000])
def test_several_cells_per_thread(lat, dtype, columns):
    nv = 3
    rng = np.random.default_rng(columns)
    sizes = [200, 1000, 260_000, 2049, 1023]
    while sum(sizes) < columns:
        sizes.append(int(rng.integers(200, 6000)))
    ens, dv = ensemble(lat, sizes, nv, dtype)
    check(ens, dv, nv, dtype, [0, 1, 7, 64, 150, 199, 3, 2, 100],
          [0, 1, 2, 3, 4, len(sizes) // 2, len(sizes) - 1])
    ens.close()


def test_scratch_follows_the_columns(lat):
    ens, dv = ensemble(lat, [1_000_000] + [40] * 10000, 3, torch.float32)
    ens.moments()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    check(ens, dv, 3, torch.float32, [1, 2, 3, 4, 5, 6, 7, 8], [0, 1, 5000, 10000])
    assert free - torch.cuda.mem_get_info()[0] < 256 << 20  # 11 MB of densities, the blocks' sums
    ens.close()


def test_one_separation_does_not_pay_for_eight(lat):
    rng = np.random.default_rng(4)
    ens, _ = ensemble(lat, list(map(int, rng.choice([1024, 2048, 4096], 512))), 9, torch.float32)

    def best(seps):
        out = math.inf
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for _ in range(12):
            a.record()
            ens.s1(seps)
            b.record()
            b.synchronize()
            out = min(out, a.elapsed_time(b))
        return out

    one, eight = best([1]), best(list(range(1, 9)))
    assert one < 0.75 * eight, (one, eight)
    ens.close()
