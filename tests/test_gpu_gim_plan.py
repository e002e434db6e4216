"""Gimenez plans: what creating one costs, and the tables of plans at the
ends of the accepted orders and depths.

A plan is one allocation, one upload and one kernel.  What the driver takes
for a block of the plan's size differs by several times between machines, so
a table of the Mandel-Agol terms (MATable) of as many bytes, one allocation and one kernel, is
timed beside it.  To that come the host's tables, the upload and the longer
kernel (75 us at N = 8, n_j = 192, 250 at N = 16, n_j = 512), allowed about twice.
Creation with nine allocations, seven uploads and two FP64 passes took 330 and
660 us more than the table.

The light curves' bounds are those of the series' depth test: at k <= 0.7 1e-6,
up to 1.5 2.5e-6 (rows 9e-8 and 6e-7 in 64 bits, FP32 roundings, sum |C_n| <= 2).
"""
import time

import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit

pytestmark = pytest.mark.gpu


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("N,n_j,n_k,n_z,allowed_us", [(8, 192, 128, 2976, 150.0), (16, 512, 2048, 2408, 500.0)])
def test_creation_time(N, n_j, n_k, n_z, allowed_us):
    torch = _torch()
    import paper_1504_07433_gb300 as pt
    torch.zeros(1, device="cuda")

    def median(make):
        out = []
        for _ in range(25):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            x = make()
            torch.cuda.synchronize()
            x.close()
            out.append(time.perf_counter() - t0)
        return sorted(out)[12]

    table, plan = median(lambda: pt.MATable(0.05, 0.2, n_k, n_z)), median(lambda: pt.GimenezPlan(N, n_j))
    print("table %.0f us, plan %.0f us" % (table * 1e6, plan * 1e6))
    assert plan <= table + 1e-6 * allowed_us, (plan, table)


@pytest.mark.parametrize("N,n_j", [(1, 2), (16, 2), (1, 33), (16, 32), (3, 65), (1, 512)])
def test_tables_at_the_ends_of_the_range(N, n_j):
    torch = _torch()
    import paper_1504_07433_gb300 as pt
    ks = np.array([0.05, 0.3, 0.7, 1.0, 1.5])
    n_v, n_t = ks.size, 700
    rng = np.random.default_rng(N * 1000 + n_j)
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, n_gim=max(2, N))
    o = wl["orbit"]
    o["t0"], o["P"], o["a"], o["b"] = np.full(n_v, 0.1), np.full(n_v, 3.0), np.full(n_v, 8.0), rng.uniform(0.0, 0.4, n_v)
    o["e"] = o["w"] = None
    o["inc"] = W.inc_from_b(o["b"], o["a"])
    wl["t"] = 0.1 + np.linspace(-0.18, 0.18, n_t)
    wl["k"] = ks
    u = W.quad_to_general(*W.q_to_u(rng.uniform(0, 1, (n_v, 1)), rng.uniform(0, 1, (n_v, 1))), max(2, N))[..., :N]
    if N > 2:
        u[..., 2:] = rng.uniform(-0.005, 0.005, (n_v, 1, N - 2))
    wl["ld"] = u
    t, orb, k, ld = gpu_inputs(wl)
    plan = pt.GimenezPlan(N, n_j)
    f, _ = pt.gimenez(plan, t, orb, k, ld)
    torch.cuda.synchronize()
    ref, _ = oracle.lc_gimenez(wl["t"], oracle_orbit(o), f32(ks), f32(u), n_j)
    err = np.abs(f.cpu().numpy() - ref).max(axis=(1, 2))
    assert (err <= np.where(ks <= 0.7, 1e-6, 2.5e-6)).all(), (ks, err)
    plan.close()
