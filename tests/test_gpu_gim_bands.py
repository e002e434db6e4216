"""Gimenez light curves of passbands that share a radius ratio.  Their rows are
formed from the terms' products: a passband has, bit for bit, the fluxes of a
call with that passband alone, and a vector those of its own call, at every
tile form of the product (2 to 5,003 vectors; orders of one, several and partly
filled chains).
More than eight passbands read the terms' rows (N + 1 of them, in groups, the
depth carried through the flux); above 96 KB a geometry's rows stay in global
memory.  All against the FP64 oracle: 1e-6 in flux, the z-interpolated model
against the oracle's own z tables, residual sums to 2e-5 of the FP64 sums of the
returned fluxes.  And passbands are cheap: eight of them cost less than 2.5 times
one (an evaluation per passband is a quarter of a shared product's time; as
products of their own they took 6.2 times)."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32, gpu_inputs, oracle_orbit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    return torch


def _workload(n_v, n_t, n_b, N, n_ss=1, cadence=0.01):
    rng = np.random.default_rng(n_v + n_b)
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=n_ss, cadence=cadence, n_gim=max(2, N))
    u = W.quad_to_general(*W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), max(2, N))[..., :N]
    if N > 2:
        u[..., 2:] = rng.uniform(-0.02, 0.02, (n_v, n_b, N - 2))
    wl["ld"] = u
    return wl


@pytest.mark.parametrize("N,n_j,n_v,n_b", [(1, 20, 40, 4), (3, 33, 2, 4), (8, 64, 9, 4), (8, 64, 100, 4), (8, 192, 256, 4),
                                           (2, 64, 1000, 2), (16, 24, 33, 4), (2, 64, 4600, 3), (8, 50, 5003, 2),
                                           (2, 64, 4600, 9), (16, 40, 100, 9), (10, 140, 3001, 1), (10, 140, 3001, 9)])
def test_passbands_have_the_bits_of_their_own_call(torch_cuda, N, n_j, n_v, n_b):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    wl = _workload(n_v, 150, n_b, N)
    t, orb, k, ld = gpu_inputs(wl)
    plan = pt.GimenezPlan(N, n_j)
    f, _ = pt.gimenez(plan, t, orb, k, ld)
    for b in range(n_b if n_b <= 8 else 0):   # (more read the terms' rows, rounded once more)
        f1, _ = pt.gimenez(plan, t, orb, k, ld[:, b:b + 1].contiguous())
        assert torch.equal(f[:, b:b + 1], f1), b
    one = {x: None if orb[x] is None else orb[x][n_v - 1:].contiguous() for x in orb}
    f2, _ = pt.gimenez(plan, t, one, k[n_v - 1:].contiguous(), ld[n_v - 1:].contiguous())
    assert torch.equal(f2[0], f[n_v - 1])
    pick = slice(max(0, n_v - 3), n_v)
    o = {x: (None if v is None else np.asarray(v)[pick]) for x, v in oracle_orbit(wl["orbit"]).items()}
    ref = oracle.lc_gimenez(wl["t"], o, f32(wl["k"])[pick], f32(wl["ld"])[pick], n_j)[0]
    assert (ref < 1).any() and np.max(np.abs(f[pick].cpu().numpy() - ref)) <= 1e-6
    plan.close()


@pytest.mark.parametrize("model,N,n_j,n_b,n_ss", [("gim", 2, 40, 9, 3), ("gim", 8, 64, 12, 2), ("gim", 16, 33, 9, 1),
                                                   ("gim", 16, 512, 9, 1), ("gim", 8, 64, 8, 2), ("gim", 8, 64, 5, 2),
                                                   ("zi", 8, 64, 12, 2), ("zi", 16, 33, 10, 1), ("zi", 4, 48, 5, 3),
                                                   ("interp", 2, 0, 9, 2), ("interp", 2, 0, 6, 3)])
def test_many_passbands_on_one_radius_ratio(torch_cuda, model, N, n_j, n_b, n_ss):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    n_v, n_t = 7, 700
    wl = _workload(n_v, n_t, n_b, N, n_ss)
    rng = np.random.default_rng(n_b)
    if model == "interp":
        wl["ld"] = np.stack(W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), -1)
    t, orb, k, ld = gpu_inputs(wl)
    y_np = rng.normal(1.0, 1e-3, (n_b, n_t)).astype(np.float32)
    y = torch.as_tensor(y_np, device="cuda")
    kw = dict(n_ss=n_ss, t_exp=wl["t_exp"] if n_ss > 1 else 0.0)
    oo, kk, uu = oracle_orbit(wl["orbit"]), f32(wl["k"]), f32(wl["ld"])
    plan = pt.GimenezPlan(N, n_j) if model != "interp" else None
    if model == "gim":
        call = lambda **x: pt.gimenez(plan, t, orb, k, ld, **kw, **x)   # noqa: E731
        ref = oracle.lc_gimenez(wl["t"], oo, kk, uu, n_j, **kw)[0]
    elif model == "zi":
        call = lambda **x: pt.gimenez_zi(plan, t, orb, k, ld, n_in=32, n_edge=24, **kw, **x)   # noqa: E731
        ref = oracle.lc_gimenez_zi(wl["t"], oo, kk, uu, n_j, n_in=32, n_edge=24, **kw)[0]
    else:
        table = pt.MATable(0.03125, 0.25, 32, 64)
        call = lambda **x: pt.ma_quad_interp(table, t, orb, k, ld, **kw, **x)   # noqa: E731
        ref = oracle.lc_ma_interp(oracle.MATable(0.03125, 0.25, 32, 64), wl["t"], oo, kk, uu, **kw)[0]
    flux, _ = call()
    flux2, ssr = call(y=y, want_ssr=True)
    _, ssr2 = call(y=y, want_ssr=True, want_flux=False)
    torch.cuda.synchronize()
    assert torch.equal(flux, flux2) and torch.equal(ssr, ssr2)
    f = flux.cpu().numpy().astype(np.float64)
    assert (ref < 1).any() and np.max(np.abs(f - ref)) <= 1e-6
    s = ((y_np.astype(np.float64)[None] - f) ** 2).sum(axis=2)
    assert np.max(np.abs(ssr.cpu().numpy() / s - 1)) <= 2e-5
    if plan is not None:
        plan.close()


def test_passbands_share_the_product(torch_cuda):
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    plan = pt.GimenezPlan(8, 192)
    us = {}
    for n_b in (1, 8):
        t, orb, k, ld = gpu_inputs(_workload(1000, 100, n_b, 8))
        work = torch.empty(plan.work_bytes(100, 1000, n_b, 0), dtype=torch.uint8, device="cuda")
        flux = torch.empty((1000, n_b, 100), dtype=torch.float32, device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(6):
            a.record()
            for _ in range(10):
                pt.gimenez(plan, t, orb, k, ld, work=work, flux=flux)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 100.0)
        us[n_b] = best
    plan.close()
    assert us[8] < 2.5 * us[1], us
