"""More geometries than one launch's grid takes along y (65,535 blocks of 8),
with few times each: every vector's fluxes and residual sums are, bit for bit,
those of a small call with that vector, and within 1e-6 of the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit


@pytest.mark.gpu
@pytest.mark.parametrize("n_v,n_t", [(524281, 7), (600000, 20)])
def test_short_series_of_many_vectors(n_v, n_t):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, cadence=0.01)
    wl["orbit"]["t0"] = np.random.default_rng(n_t).uniform(0.0, 0.01 * n_t, n_v)   # transits within the few times
    t, orb, k, ld = gpu_inputs(wl)
    y = torch.full((1, n_t), 0.999, dtype=torch.float32, device="cuda")
    kw = dict(y=y, want_ssr=True)
    flux, ssr = pt.ma_quad(t, orb, k, ld, **kw)
    torch.cuda.synchronize()
    pick = np.r_[0:50, 524200:524281, n_v - 1]   # on both sides of the first launch's end
    idx = torch.as_tensor(pick, device="cuda")
    part = {key: (None if v is None else v[idx].contiguous()) for key, v in orb.items()}
    f1, s1 = pt.ma_quad(t, part, k[idx].contiguous(), ld[idx].contiguous(), **kw)
    torch.cuda.synchronize()
    assert torch.equal(flux[idx], f1) and torch.equal(ssr[idx], s1)
    o = {key: (None if v is None else np.asarray(v)[pick]) for key, v in oracle_orbit(wl["orbit"]).items()}
    ref, _ = oracle.lc_ma(wl["t"], o, f32(wl["k"])[pick], f32(wl["ld"])[pick])
    assert (ref < 1).sum() > 50
    assert np.abs(f1.cpu().numpy() - ref).max() <= 1e-6


@pytest.mark.gpu
def test_passbands_with_their_own_radius_ratios():
    """The second launch starts inside a vector's passbands (524,280 is no
    multiple of 7): its passbands keep their own data."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    n_v, n_b, n_t = 75000, 7, 20
    rng = np.random.default_rng(7)
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, cadence=0.01)
    wl["orbit"]["t0"] = rng.uniform(0.0, 0.01 * n_t, n_v)
    wl["k"] = wl["k"][:, None] * rng.uniform(0.9, 1.1, (n_v, n_b))
    wl["ld"] = np.repeat(wl["ld"][:, :1], n_b, axis=1)
    t, orb, k, ld = gpu_inputs(wl)
    y = torch.as_tensor(rng.normal(1.0, 1e-3, (n_b, n_t)).astype(np.float32), device="cuda")
    flux, ssr = pt.ma_quad(t, orb, k, ld, y=y, want_ssr=True)
    lo = 524280 // n_b - 10
    part = {x: None if v is None else v[lo:lo + 40].contiguous() for x, v in orb.items()}
    f1, s1 = pt.ma_quad(t, part, k[lo:lo + 40].contiguous(), ld[lo:lo + 40].contiguous(), y=y, want_ssr=True)
    assert torch.equal(flux[lo:lo + 40], f1) and torch.equal(ssr[lo:lo + 40], s1)
