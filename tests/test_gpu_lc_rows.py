"""Light curves from row tables at the edges of their rules and layout, against
the FP64 oracle at the exact path's 1e-6 flux (k <= 1): radius ratios outside
the tables' range beside ones inside it, one row per passband (up to 8) and the
rows of the terms (more), light curves that end inside a tile or on it, times
in any order, exposures too long for the f and g series, residual sums (2e-5 of
the FP64 sums of the same residuals) with and without weights, and a call in
which every time is in transit."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit



TOL = 1e-6

# n_t, n_v, n_b, own radius ratios, n_ss, exposure (days; None: the long cadence's), cadence, shuffled, odd k, weights
CASES = [
    (512, 5, 1, False, 1, 0.0, 0.013, False, True, False),
    (513, 6, 8, False, 3, None, 0.013, False, False, True),
    (770, 5, 9, False, 2, None, 0.011, True, True, False),
    (1025, 7, 3, True, 5, 0.3, 0.007, False, False, True),
    (300, 33, 1, False, 10, None, 0.02, True, False, False),
    (4096, 40, 2, True, 2, 0.01, 0.0005, False, True, True),
    (700, 64, 1, False, 1, 0.0, 0.00005, False, False, True),
]


@pytest.mark.gpu
@pytest.mark.parametrize("n_t,n_v,n_b,own_k,n_ss,t_exp,cadence,shuffled,odd_k,weights", CASES)
def test_ma_rows_vs_oracle(n_t, n_v, n_b, own_k, n_ss, t_exp, cadence, shuffled, odd_k, weights):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=n_ss, cadence=cadence)
    rng = np.random.default_rng(n_t + n_b)
    if cadence < 1e-3:   # around one transit
        wl["orbit"]["t0"] = 0.5 * n_t * cadence + rng.normal(0.0, 0.002, n_v)
    if t_exp is not None:
        wl["t_exp"] = t_exp
    wl["ld"] = np.stack(W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), axis=-1)
    if odd_k:
        wl["k"][::2] = rng.choice([0.5, 0.5000001, 0.7, 1e-6, 5e-7, 0.02], wl["k"][::2].size)
    if own_k:
        wl["k"] = wl["k"][:, None] * rng.uniform(0.95, 1.05, (n_v, n_b))
    if shuffled:
        wl["t"] = rng.permutation(wl["t"])
    t, orb, k, ld = gpu_inputs(wl)
    y_np = rng.normal(1.0, 1e-3, (n_b, n_t)).astype(np.float32)
    w_np = rng.uniform(0.5, 2.0, (n_b, n_t)).astype(np.float32) if weights else np.ones((n_b, n_t), np.float32)
    y = torch.as_tensor(y_np, device="cuda")
    wt = torch.as_tensor(w_np, device="cuda") if weights else None
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    kw = dict(n_ss=n_ss, t_exp=wl["t_exp"], n_bad=bad)
    flux, _ = pt.ma_quad(t, orb, k, ld, **kw)
    flux2, ssr = pt.ma_quad(t, orb, k, ld, y=y, wt=wt, want_ssr=True, **kw)
    _, ssr2 = pt.ma_quad(t, orb, k, ld, y=y, wt=wt, want_flux=False, want_ssr=True, **kw)
    # an output that does not start on 16 bytes
    raw = torch.empty(n_v * n_b * n_t + 1, device="cuda")
    flux3, _ = pt.ma_quad(t, orb, k, ld, flux=raw[1:].view(n_v, n_b, n_t), **kw)
    f = flux.cpu().numpy().astype(np.float64)
    ref = oracle.lc_ma(wl["t"], oracle_orbit(wl["orbit"]), f32(wl["k"]), f32(wl["ld"]), n_ss=n_ss,
                       t_exp=wl["t_exp"])[0]
    assert int(bad.item()) == 0 and (ref < 1).sum() > 0
    assert np.max(np.abs(f - ref)) <= TOL
    assert torch.equal(flux, flux2) and torch.equal(flux, flux3) and torch.equal(ssr, ssr2)
    own = np.sum(w_np.astype(np.float64) * (y_np.astype(np.float64) - f) ** 2, axis=2)
    assert np.allclose(ssr.cpu().numpy(), own, rtol=2e-5)


def test_f_and_g_series_remainder():
    """The bound that fg_valid uses, in 64 bits over eccentricities and phases."""
    rng = np.random.default_rng(0)
    for e_lo, e_hi in ((0.0, 0.3), (0.3, 0.6), (0.6, 0.95)):
        e, M = rng.uniform(e_lo, e_hi, 50000), rng.uniform(0, 2 * np.pi, 50000)

        def state(m):
            E = m + e * np.sin(m)
            for _ in range(60):
                E = E - (E - e * np.sin(E) - m) / (1 - e * np.cos(E))
            e1 = 1 / (1 - e * np.cos(E))
            b = np.sqrt(1 - e * e)
            return np.array([np.cos(E) - e, b * np.sin(E)]), np.array([-np.sin(E) * e1, b * np.cos(E) * e1]), e1, e * np.sin(E)
        r, v, e1, es = state(M)
        for s in (5e-4, 2e-3):
            u, p, q = e1 ** 3, es * e1 ** 2, e1 * e1 * (e1 - 1)
            x = np.sqrt(s / u)
            f = (1 - u * x ** 2 / 2 + u * p * x ** 3 / 2 + u * (3 * q - 15 * p * p + u) / 24 * x ** 4
                 + u * p * (7 * p * p - 3 * q - u) / 8 * x ** 5)
            g = x - u * x ** 3 / 6 + u * p * x ** 4 / 4 + u * (9 * q - 45 * p * p + u) / 120 * x ** 5
            assert np.all(np.abs(f * r + g * v - state(M + x)[0]) <= (0.02 + 0.4 * e * e) * s ** 3 + 1e-14)
