"""Gimenez light curves against the FP64 oracle's series of the same depth, at
depths on both sides of where the rows' interval width stops growing and at
radius ratios up to above 1.

Bounds, from the rows' error in 64 bits (pt_gim.cuh) and FP32 roundings: a
coefficient of a row is rounded to 2^-24 of sums of magnitudes up to 1.5 (5e-8 at
k = 0.5, 9e-8 at 1.5), the separation to 1e-7 with |df/dz| <= 2, the flux to 6e-8;
sum |C_n| <= 2.  k <= 0.7: 2 (9e-8 + 5e-8) + 2e-7 + 6e-8 < 1e-6 (the light curves'
bound elsewhere); k = 1 .. 1.5: 2 (6e-7 + 9e-8) + 4e-7 + 6e-8 < 2.5e-6."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit


@pytest.mark.gpu
@pytest.mark.parametrize("N,n_j", [(2, 2), (8, 24), (4, 64), (8, 95), (8, 96), (2, 97), (8, 190), (8, 193), (4, 512)])
def test_series_depths_and_radius_ratios(N, n_j):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    ks = np.array([0.05, 0.3, 0.5, 0.7, 0.97, 1.0, 1.05, 1.5])
    n_v, n_t = ks.size, 900
    rng = np.random.default_rng(n_j)
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, n_gim=max(2, N))
    o = wl["orbit"]
    o["t0"], o["P"], o["a"], o["b"] = np.full(n_v, 0.1), np.full(n_v, 3.0), np.full(n_v, 8.0), rng.uniform(0.0, 0.4, n_v)
    o["e"] = o["w"] = None
    o["inc"] = W.inc_from_b(o["b"], o["a"])
    wl["t"] = 0.1 + np.linspace(-0.18, 0.18, n_t)
    wl["k"] = ks
    u = W.quad_to_general(*W.q_to_u(rng.uniform(0, 1, (n_v, 1)), rng.uniform(0, 1, (n_v, 1))), N)
    if N > 2:
        u[..., 2:] = rng.uniform(-0.02, 0.02, (n_v, 1, N - 2))
    wl["ld"] = u
    t, orb, k, ld = gpu_inputs(wl)
    plan = pt.GimenezPlan(N, n_j)
    f, _ = pt.gimenez(plan, t, orb, k, ld)
    torch.cuda.synchronize()
    ref, _ = oracle.lc_gimenez(wl["t"], oracle_orbit(o), f32(ks), f32(u), n_j)
    err = np.abs(f.cpu().numpy() - ref).max(axis=(1, 2))
    tol = np.where(ks <= 0.7, 1e-6, 2.5e-6)
    assert (ref[:, 0] < 1).sum(axis=1).min() > 200
    assert (err <= tol).all(), (ks, err)
    plan.close()
