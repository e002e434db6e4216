"""Serving kernels at the edges of the network's tiles (128 points, several
groups of a CTA in flight) and of the classification's blocks (2,048 points):
every point is independent of the others, so a call on a prefix of the points
gives bitwise the prefix of the whole call's results, and the count of points
the exact terms served is that of the same classification on the host."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = (1, 127, 128, 129, 511, 513, 2047, 2049, 4 * 128 * 152 + 1)


def test_prefixes_bitwise():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300.surrogate as S
    rng = np.random.default_rng(2)
    table = (rng.uniform(size=(64, 64)) < 0.5).astype(np.uint8)
    model = S.SurrogateModel(S.init_params(1), table)
    N = 2 * 4 * 128 * 152 + 77
    X = torch.rand((N, 2), device="cuda") * 2 - 1
    Y = model.network(X)
    k = 0.005 + 0.3 * torch.rand(N, device="cuda")          # a few below the band's range
    z = 1.0 - k + (2.1 * torch.rand(N, device="cuda") - 0.05) * k   # a few on either side of the band
    ref = model.terms(k, z)
    s = (z - (1.0 - k).abs()) / (2.0 * k)
    lo, hi = torch.tensor(S.K_LO, device="cuda"), torch.tensor(S.K_HI, device="cuda")
    ck = ((k - lo) / (hi - lo) * 64).int().clamp(0, 63).long()
    cs = (s * 64).int().clamp(0, 63).long()
    net = (k >= lo) & (k <= hi) & (s >= 0) & (s < 1) & (torch.as_tensor(table, device="cuda")[ck, cs] == 0)
    assert 0.2 < net.float().mean().item() < 0.8
    for n in SIZES:
        assert torch.equal(model.network(X[:n].contiguous()), Y[:n]), n
        fb = torch.zeros(1, dtype=torch.int32, device="cuda")
        out = model.terms(k[:n].contiguous(), z[:n].contiguous(), n_fallback=fb)
        assert all(torch.equal(a, b[:n]) for a, b in zip(out, ref)), n
        assert int(fb.item()) == int((~net[:n]).sum()), n
    assert not model.timed_out()
