"""Batch plans whose passbands have no row table (radius ratios outside the
tables' range, plans with few points): one orbit solution for a group's
passbands, beside passbands with tables in the same group of sixteen, against the
FP64 oracle (1e-6 in flux, 3e-6 above k = 1 as in test_gpu_ma.py, where FP32 resolves
lambda_d to about 1e-6; residual sums to 2e-5 of the FP64 sums of the returned
fluxes).
A plan of short light curves takes less time than the same curves by pt_ma_quad
(a passband at a time it took more than twice as long)."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, oracle_orbit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    return torch


def _inputs(torch, n_v, n_b, lens, k):
    import paper_1504_07433_gb300 as pt
    rng = np.random.default_rng(n_b)
    o = dict(t0=rng.normal(0.0, 1e-3, n_v), P=np.full(n_v, 3.0), a=rng.uniform(8.0, 10.0, n_v), e=None, w=None)
    o["inc"] = W.inc_from_b(rng.uniform(0.0, 0.4, n_v), o["a"])
    t = np.concatenate([3.0 * j + np.linspace(-0.2, 0.2, n) for j, n in enumerate(lens)])
    offs = np.concatenate([[0], np.cumsum(lens)])
    ld = np.stack(W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), -1)
    f = lambda x: torch.as_tensor(np.asarray(x, np.float32), device="cuda").contiguous()   # noqa: E731
    y, wt = rng.normal(1.0, 1e-3, (n_b, t.size)).astype(np.float32), rng.uniform(0.5, 2.0, (n_b, t.size)).astype(np.float32)
    dev = (torch.as_tensor(t, dtype=torch.float64, device="cuda"), offs, pt.orbit_to_device(o), f(k), f(ld))
    return o, t, ld, y, wt, dev, f


# passbands, light curves, radius ratios (cycled over the passbands), supersamples
CASES = [
    (1, [40], [0.1], 1), (5, [100, 64], [0.1, 0.6], 1), (17, [30, 65, 1], [0.1], 2), (4, [300, 1, 210], [0.7, 1.1], 1),
    (18, [400, 370], [0.1, 0.7, 0.1, 0.1, 0.5000001, 5e-7], 1), (16, [700], [0.8], 3), (37, [767], [0.1] * 20 + [0.9], 1),
    (37, [769], [0.1] * 20 + [0.9], 1),
]


@pytest.mark.parametrize("n_b,lens,ks,n_ss", CASES)
@pytest.mark.parametrize("weights", [False, True])
def test_plans_without_tables(torch_cuda, n_b, lens, ks, n_ss, weights):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    n_v = 6
    k = np.resize(ks, n_b)[None] * np.linspace(1.0, 1.02, n_v)[:, None]
    k = np.where(np.isin(np.resize(ks, n_b)[None], [5e-7, 0.5000001]), np.resize(ks, n_b)[None], k)
    o, t, ld, y, wt, dev, f = _inputs(torch, n_v, n_b, lens, k)
    t_exp = 0.003 if n_ss > 1 else 0.0
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    kw = dict(n_ss=n_ss, t_exp=t_exp, y=f(y), wt=f(wt) if weights else None, n_bad=bad)
    p = pt.BatchPlan(*dev, want_flux=True, want_ssr=True, **kw)
    q = pt.BatchPlan(*dev, want_flux=False, want_ssr=True, autotune=False, **kw)
    flux, ssr = p.run()
    _, ssr2 = q.run()
    torch.cuda.synchronize()
    fl = flux.cpu().numpy().astype(np.float64)
    ref, _ = oracle.lc_ma(t, oracle_orbit(o), f32(k), f32(ld), n_ss=n_ss, t_exp=t_exp)
    err = np.abs(fl - ref).max(axis=2)
    assert (ref < 1).any() and (err <= np.where(k <= 1.0, 1e-6, 3e-6)).all() and bad.item() == 0
    s = ((wt if weights else 1.0) * (y.astype(np.float64)[None] - fl) ** 2).sum(axis=2)
    assert np.abs(ssr.cpu().numpy() / s - 1).max() <= 2e-5 and np.abs(ssr2.cpu().numpy() / s - 1).max() <= 2e-5
    p.close()
    q.close()


def test_short_plans_are_no_slower_than_single_calls(torch_cuda):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    n_v, n_b, n_t = 1000, 16, 300
    k = np.full((n_v, n_b), 0.1)
    _, _, _, y, _, dev, f = _inputs(torch, n_v, n_b, [100, 100, 100], k)
    t, _, orb, kk, ld = dev
    plan = pt.BatchPlan(*dev, y=f(y), want_flux=False, want_ssr=True)
    work = torch.empty(int(pt.load_library().pt_ma_quad_work_bytes(n_t, n_v, n_b, 1)), dtype=torch.uint8, device="cuda")
    ssr = torch.empty((n_v, n_b), dtype=torch.float32, device="cuda")
    yy = f(y)
    us = {}
    for name, call in (("plan", plan.run), ("ma_quad", lambda: pt.ma_quad(t, orb, kk, ld, y=yy, want_flux=False, want_ssr=True,
                                                                        work=work, ssr=ssr))):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(6):
            a.record()
            for _ in range(10):
                call()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 100.0)
        us[name] = best
    plan.close()
    assert us["plan"] < us["ma_quad"], us
