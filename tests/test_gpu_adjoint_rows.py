"""The adjoint's two ways to the limb terms (per-vector rows of polynomials;
exact elliptic integrals) and its two block sizes, against the FP64 oracle.

The cases stand at the edges of the rule: radius ratios at, just outside and
well outside [0.02, 0.5]; just under and over 1,280 points a vector; one
vector, and more than the wide blocks take; circular orbits; one and several
supersamples; times packed around the inner contact, where the derivatives'
w^2 log w term sits.  The tolerance is test_gpu_adjoint's error model (flux
1e-6, derivatives 1e-5, the rows' interpolation error of 3.4e-6 included).
"""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from test_gpu_adjoint import _bound, _theta_rows, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_v,n_t,n_ss,k,b,ecc,check", [
    (7, 1279, 1, 0.1, 0.3, True, 7),            # exact terms: too few points
    (7, 1281, 1, 0.1, 0.3, True, 7),            # rows, last tile of one time
    (1, 430, 3, 0.1, 0.3, True, 1),             # rows by the supersamples
    (8, 1300, 1, 0.02, 0.3, True, 8),           # k below, at and above the lower edge
    (8, 1300, 1, 0.5, 0.5, True, 8),            # the upper edge
    (3, 1300, 2, 0.3, 0.75, False, 3),          # grazing, circular
    (3, 1300, 1, 1.2, 0.1, True, 3),            # the planet larger than the star
    (640, 1300, 1, 0.1, 0.3, True, 4),          # narrow blocks
])
def test_adjoint_rows_and_exact_terms(torch_cuda, n_v, n_t, n_ss, k, b, ecc, check):  # noqa: F811
    torch = torch_cuda
    import paper_1504_07433_gb300 as pt
    wl = W.adjoint(n_v=n_v, n_t=n_t, spread=0.5)
    th = wl["theta"]
    rng = np.random.default_rng(n_t + n_v)
    th["k"] = k * (1.0 + 2e-3 * rng.normal(size=n_v))
    th["b"] = b * (1.0 + 1e-2 * rng.normal(size=n_v))
    if not ecc:
        th["e"] = np.zeros(n_v)
        th["w"] = np.full(n_v, 0.5 * np.pi)
    # half of the times over the transit, half within 1% of its length around the inner contact
    half = 0.5 * np.sqrt(max((1.0 - k) ** 2 - b * b, 0.01)) * 3.0 / (np.pi * 12.0)
    t = np.concatenate([0.25 * wl["t"][::2], half + 5e-4 * np.linspace(-1.0, 1.0, n_t - (n_t + 1) // 2)])
    t_exp = 0.004 if n_ss > 1 else 0.0
    rows = _theta_rows(th, slice(0, check))
    # data near, not at, the first vector's light curve
    y = np.array([oracle.flux_theta(tj, rows[0], n_ss, t_exp) for tj in t])
    y = (1.0 + 0.98 * (y - 1.0) + rng.normal(0, 1e-4, n_t)).astype(np.float32)
    ssr, grad, flux = pt.ma_quad_bwd(torch.as_tensor(t, dtype=torch.float64, device="cuda"), pt.theta_to_device(th),
                                     torch.as_tensor(y, device="cuda"), n_ss=n_ss, t_exp=t_exp, want_flux=True)
    f_ref = np.array([[oracle.flux_theta(tj, rows[v], n_ss, t_exp) for tj in t] for v in range(check)])
    assert np.max(np.abs(flux.cpu().numpy()[:check].astype(np.float64) - f_ref)) <= 1e-6
    ssr_r, grad_r = oracle.ssr_grad(t, rows, y.astype(np.float64), n_ss=n_ss, t_exp=t_exp)
    assert np.allclose(ssr.cpu().numpy()[:check], ssr_r, rtol=2e-4, atol=1e-9)
    err = np.abs(grad.cpu().numpy()[:check].astype(np.float64) - grad_r)
    tol = _bound(t, rows, y.astype(np.float64), None, n_ss, t_exp)
    with np.errstate(invalid="ignore"):   # dw of a circular orbit: zero by zero
        ratio = err / tol
    worst = np.unravel_index(np.nanargmax(ratio), err.shape)
    print("largest error / bound %.3f at %s" % (ratio[worst], worst))
    assert np.all(err <= tol), (worst, err[worst], tol[worst])
