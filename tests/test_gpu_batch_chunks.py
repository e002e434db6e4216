"""A batch plan whose row tables pass 2 GB (60,000 walkers x 48 passbands x 768
bytes) makes them for half of the walkers at a time: it allocates less than 2 GB,
and walkers on both sides of the cut have the residual sums of a plan of their own
(to 1e-6: its slices of the times, and so the sums' order, may differ) and follow
new contents of the bound buffers."""
import numpy as np
import pytest

from paper_1504_07433_gb300 import workloads as W


@pytest.mark.gpu
def test_walkers_beyond_two_gigabytes_of_tables():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    n_v, n_b, n_t = 60000, 48, 800
    rng = np.random.default_rng(48)
    o = dict(t0=rng.normal(0.0, 1e-3, n_v), P=np.full(n_v, 3.0), a=rng.uniform(9.0, 11.0, n_v), e=None, w=None)
    o["inc"] = W.inc_from_b(rng.uniform(0.0, 0.4, n_v), o["a"])
    orb = pt.orbit_to_device(o)
    t = torch.linspace(-0.15, 0.15, n_t, dtype=torch.float64, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    k = 0.09 + 0.02 * torch.rand((n_v, n_b), generator=g, device="cuda")
    ld = torch.rand((n_v, n_b, 2), generator=g, device="cuda") * 0.5
    y = 1.0 + 1e-3 * torch.randn((n_b, n_t), generator=g, device="cuda")
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    plan = pt.BatchPlan(t, [0, n_t], orb, k, ld, y=y, want_flux=False, want_ssr=True, autotune=False)
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] < 2e9
    for _ in range(2):
        _, ssr = plan.run()
        for lo in (0, 29950, n_v - 100):
            part = {x: None if v is None else v[lo:lo + 100].contiguous() for x, v in orb.items()}
            small = pt.BatchPlan(t, [0, n_t], part, k[lo:lo + 100].contiguous(), ld[lo:lo + 100].contiguous(), y=y,
                                 want_flux=False, want_ssr=True, autotune=False)
            _, s = small.run()
            torch.cuda.synchronize()
            assert ((ssr[lo:lo + 100] / s - 1).abs() <= 1e-6).all()
            small.close()
        k.mul_(1.02)
        y.sub_(1e-4)
    plan.close()
