"""Calls of different sizes from several host threads: what one call sets on a
kernel (its shared-memory limit) does not refuse or change another's launch."""
import threading

import numpy as np
import pytest

from paper_1504_07433_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    return torch


def _f32(torch, x):
    return torch.as_tensor(np.asarray(x, np.float32), device="cuda").contiguous()


def _call(torch, n_v, n_t, n_b, plan=None):
    """A call with residual sums of n_b passbands that share k; its work buffer is kept."""
    import paper_1504_07433_gb300 as pt
    rng = np.random.default_rng(n_b)
    N = plan.N if plan is not None else 2
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, n_gim=max(2, N))
    t = torch.as_tensor(wl["t"], dtype=torch.float64, device="cuda")
    orb = pt.orbit_to_device(wl["orbit"])
    ld = np.stack(W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), -1)
    if plan is not None:
        ld = W.quad_to_general(ld[..., 0], ld[..., 1], N)
    y = 1.0 + 1e-3 * rng.standard_normal((n_b, n_t))
    args = (t, orb, _f32(torch, wl["k"]), _f32(torch, ld))
    kw = dict(n_ss=1, t_exp=0.0, y=_f32(torch, y), want_flux=False, want_ssr=True)
    if plan is None:
        work = torch.empty(int(pt.load_library().pt_ma_quad_work_bytes(n_t, n_v, n_b, 0)), dtype=torch.uint8, device="cuda")
        return lambda: pt.ma_quad(*args, work=work, **kw)[1]
    work = torch.empty(plan.work_bytes(n_t, n_v, n_b, 0), dtype=torch.uint8, device="cuda")
    return lambda: pt.gimenez(plan, *args, work=work, **kw)[1]


def _run_threads(torch, jobs, n):
    errors, outs = [], [None] * len(jobs)
    start = threading.Barrier(len(jobs))

    def worker(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                start.wait()
                for _ in range(n):
                    outs[i] = jobs[i]()
            s.synchronize()
        except Exception as e:   # reported below: a thread's failure must fail the test
            errors.append(e)

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(len(jobs))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors, errors
    return outs


@pytest.mark.parametrize("model", ["ma", "gimenez"])
def test_light_curve_calls_of_two_sizes(torch_cuda, model):
    """Two and three passbands (Mandel-Agol: 64 and 52 KB of shared memory in
    the row kernel), plans of two depths (Gimenez: 134 and 52 KB in the
    preparation), on two threads each: every call runs and gives bitwise the
    residual sums of a call made alone."""
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    if model == "ma":
        jobs = [_call(torch, 160, 16000, nb) for nb in (2, 3, 2, 3)]
        n = 400
    else:
        plans = [pt.GimenezPlan(4, 512), pt.GimenezPlan(4, 192)]
        jobs = [_call(torch, 6, 1000, 1 + i // 2, plans[i % 2]) for i in range(4)]
        n = 300
    refs = [job().clone() for job in jobs]
    torch.cuda.synchronize()
    for out, ref in zip(_run_threads(torch, jobs, n), refs):
        assert torch.equal(out, ref)


def test_batch_plans_of_two_sizes(torch_cuda):
    """Batch plans on tables of two lengths (64 and 51 KB of staged rows),
    created on two threads."""
    import paper_1504_07433_gb300 as pt
    torch = torch_cuda
    rng = np.random.default_rng(3)
    n_v, n_b, n_t = 6, 16, 300
    o = dict(t0=rng.normal(0, 1e-4, n_v), P=np.full(n_v, 3.0), a=np.full(n_v, 10.0), e=None, w=None)
    o["inc"] = W.inc_from_b(np.full(n_v, 0.2), o["a"])
    orb = pt.orbit_to_device(o)
    t = torch.linspace(-0.15, 0.15, n_t, dtype=torch.float64, device="cuda")
    k = _f32(torch, rng.uniform(0.09, 0.11, (n_v, n_b)))
    ld = _f32(torch, np.full((n_v, n_b, 2), 0.3))
    y = torch.ones((n_b, n_t), dtype=torch.float32, device="cuda")
    tables = [pt.MATable(0.08, 0.12, 16, n_z) for n_z in (1024, 800)]

    plans = []   # kept until the threads have ended

    def job(table):
        def run():
            p = pt.BatchPlan(t, [0, n_t], orb, k, ld, y=y, want_flux=False, want_ssr=True, autotune=False, k_mode=2,
                             table=table)
            plans.append(p)
            return p.run()[1]
        return run

    jobs = [job(tb) for tb in tables]
    refs = [j() for j in jobs]
    torch.cuda.synchronize()
    for out, ref in zip(_run_threads(torch, jobs, 60), refs):
        assert torch.equal(out, ref)
    for p in plans:
        p.close()
