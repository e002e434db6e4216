"""Residual sums of a batch plan over a million times in one slice.  The planet
stays behind the star and its window covers the period, so that every time is
evaluated with depth 0 and the sum is n (y - 1)^2 exactly, for the FP32 y.  Equal
terms make every thread round alike.  Bound: the longest chain of roundings, 64
terms of a chunk, five levels of the warp's tree, 61 chunks and eight warps, 138 x
2^-24 = 8.2e-6.  (One chain per thread over the whole slice was off by 4e-5.)"""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("n_b", [1, 3])
def test_long_residual_sums(n_b):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    n_v, n_t = 600, 1000000
    o = dict(t0=np.zeros(n_v), P=np.full(n_v, 1.0), a=np.full(n_v, 1.05), inc=np.full(n_v, 1.5), e=None, w=None)
    t = 0.5 + 0.1 * (np.arange(n_t) / n_t - 0.5)
    val = np.array([1.0137, 1.01, 0.9871], np.float32)[:n_b]
    y = torch.as_tensor(np.repeat(val[:, None], n_t, axis=1), device="cuda")
    k = torch.full((n_v, n_b), 0.1, dtype=torch.float32, device="cuda")
    ld = torch.full((n_v, n_b, 2), 0.2, dtype=torch.float32, device="cuda")
    plan = pt.BatchPlan(torch.as_tensor(t, dtype=torch.float64, device="cuda"), [0, n_t], pt.orbit_to_device(o), k, ld,
                        y=y, want_flux=False, want_ssr=True, autotune=False)
    assert plan.info()["items"] == n_v   # one slice
    _, ssr = plan.run()
    torch.cuda.synchronize()
    ref = n_t * (val.astype(np.float64) - 1.0) ** 2
    err = np.abs(ssr.cpu().numpy() / ref[None] - 1.0).max()
    assert err <= 8.2e-6, err
    plan.close()
