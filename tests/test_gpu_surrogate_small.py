"""Serving calls on both sides of the classification's block size (2^21 points) give
bitwise the same points, and few tiles spread over the SMs: 40 tiles of the network
take no longer than 1.3 times one (four to an SM, as before, they took 1.6
times)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    return torch


def test_block_sizes_bitwise(torch_cuda):
    torch = torch_cuda
    import paper_1504_07433_gb300.surrogate as S
    table = (np.random.default_rng(2).uniform(size=(64, 64)) < 0.5).astype(np.uint8)
    model = S.SurrogateModel(S.init_params(1), table)
    many = 1 << 21
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    k = 0.005 + 0.3 * torch.rand(many + 300, generator=g, device="cuda")
    z = 1.0 - k + (2.1 * torch.rand(many + 300, generator=g, device="cuda") - 0.05) * k
    fb = torch.zeros(4, dtype=torch.int32, device="cuda")
    outs = [model.terms(k[:n].contiguous(), z[:n].contiguous(), n_fallback=fb[i:i + 1])
            for i, n in enumerate((many + 300, many, many - 1, many - 255))]
    torch.cuda.synchronize()
    for out in outs[1:]:
        assert all(torch.equal(a, b[:a.numel()]) for a, b in zip(out, outs[0]))
    exact = S.exact_terms(k, z)
    served = torch.stack([a != b for a, b in zip(outs[0], exact)]).any(dim=0)   # (differs: certainly the network's)
    for i, n in enumerate((many + 300, many, many - 1, many - 255)):
        assert 0.2 * n < fb[i].item() <= n - int(served[:n].sum())
    assert not model.timed_out()


def test_few_tiles_run_beside_each_other(torch_cuda):
    torch = torch_cuda
    import paper_1504_07433_gb300.surrogate as S
    model = S.SurrogateModel(S.init_params(1), np.zeros((64, 64), np.uint8))
    us = {}
    for n in (128, 40 * 128):
        X = torch.rand((n, 2), device="cuda") * 2 - 1
        model.network(X)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()   # (the launches' host time left out)
        with torch.cuda.graph(g):
            for _ in range(20):
                model.network(X)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(6):
            a.record()
            g.replay()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 50.0)
        us[n] = best
    assert us[40 * 128] < 1.3 * us[128], us
