"""Batched evaluation at the edges of the row tables' rule and layout: radius
ratios outside the tables' range (exact terms per point) beside ones inside
it, passband counts that leave a group or a chunk of four partly filled,
light curves around a tile's length, too few points for tables, weights,
supersamples, and times in any order; against the FP64 oracle at the exact
path's 1e-6 (k <= 1), residual sums to FP32 summation of the same residuals
(2e-5, as for the other residual sums)."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit

pytestmark = pytest.mark.gpu

TOL = 1e-6


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library()
    return torch


CASES = [
    # n_v, n_b, lengths, n_ss, ecc, odd radius ratios, shuffled, weights
    (3, 1, (700,), 1, False, False, False, False),
    (4, 17, (63, 64, 65, 129, 400), 1, False, True, False, True),
    (3, 5, (300, 301, 302), 3, True, True, True, False),
    (5, 20, (1, 200, 640), 1, True, False, True, True),
    (2, 3, (90, 100), 2, False, True, False, False),
]


@pytest.mark.parametrize("n_v,n_b,lengths,n_ss,ecc,odd_k,shuffled,weights", CASES)
def test_batch_rows_vs_oracle(torch_cuda, n_v, n_b, lengths, n_ss, ecc, odd_k, shuffled, weights):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    wl = W.batched(n_walkers=n_v, n_pb=n_b, n_lc=len(lengths), len_lo=100, len_hi=100)
    rng = np.random.default_rng(17 * n_b + n_ss)
    width = 0.36
    t = [3.0 * j + np.linspace(-0.5 * width, 0.5 * width, n) for j, n in enumerate(lengths)]
    if shuffled:
        t = [rng.permutation(x) for x in t]
    wl["lc_offsets"] = np.concatenate([[0], np.cumsum(lengths)])
    wl["t"] = np.concatenate(t)
    n_t = wl["t"].size
    wl["y"] = 1.0 + rng.normal(0.0, 1e-3, (n_b, n_t))
    if odd_k:   # the ends of the tables' range and values outside it
        wl["k"].flat[::2] = rng.choice([0.5, 0.5000001, 0.62, 0.97, 1e-6, 5e-7, 0.02, 0.3], wl["k"].flat[::2].size)
    if ecc:
        wl["orbit"]["e"], wl["orbit"]["w"] = rng.uniform(0.0, 0.2, n_v), rng.uniform(0.0, 2 * np.pi, n_v)
        wl["orbit"]["inc"] = W.inc_from_b(wl["orbit"]["b"], wl["orbit"]["a"], wl["orbit"]["e"], wl["orbit"]["w"])
    wl["n_ss"], wl["t_exp"] = n_ss, 0.004 if n_ss > 1 else 0.0
    tt, orb, k, ld = gpu_inputs(wl)
    y = torch.as_tensor(wl["y"], dtype=torch.float32, device="cuda")
    wt_np = rng.uniform(0.5, 2.0, wl["y"].shape).astype(np.float32) if weights else np.ones(wl["y"].shape, np.float32)
    wt = torch.as_tensor(wt_np, device="cuda") if weights else None
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    kw = dict(n_ss=n_ss, t_exp=wl["t_exp"], n_bad=bad)
    both = pt.BatchPlan(tt, wl["lc_offsets"], orb, k, ld, y=y, wt=wt, want_flux=True, want_ssr=True, **kw)
    only_ssr = pt.BatchPlan(tt, wl["lc_offsets"], orb, k, ld, y=y, wt=wt, want_flux=False, want_ssr=True, **kw)
    only_flux = pt.BatchPlan(tt, wl["lc_offsets"], orb, k, ld, want_flux=True, autotune=False, **kw)
    flux, ssr = both.run()
    ssr2 = only_ssr.run()[1]
    flux2 = only_flux.run()[0]
    torch.cuda.synchronize()
    assert int(bad.item()) == 0
    ref = oracle.lc_ma(wl["t"], oracle_orbit(wl["orbit"]), f32(wl["k"]), f32(wl["ld"]), n_ss=n_ss,
                       t_exp=wl["t_exp"])[0]
    assert (ref < 1).mean() > 0.1
    f = flux.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(f - ref)) <= TOL
    assert torch.equal(flux, flux2)
    yy = np.asarray(wl["y"], np.float32).astype(np.float64)
    own = np.sum(wt_np.astype(np.float64)[None] * (yy[None] - f) ** 2, axis=2)
    assert np.allclose(ssr.cpu().numpy(), own, rtol=2e-5)
    assert np.allclose(ssr2.cpu().numpy(), own, rtol=2e-5)
