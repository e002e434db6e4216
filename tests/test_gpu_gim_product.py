"""The Gimenez rows' product at each of its tile widths (1, 2, 3 columns per
thread in tiles of 8 rows, 6 and 8 in tiles of 32; 856 columns at N = 8,
n_j = 192, so every last tile is cut off): a vector's light curve does not
depend on the other vectors of its call (the sums run in the same order at
every width), so it has the bits of the vector's own call, and that one is
compared with the FP64 oracle at 1e-6 flux."""
import numpy as np
import pytest

import oracle
from paper_1504_07433_gb300 import workloads as W
from tests.helpers import f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_v", [5, 64, 100, 256, 1000])
def test_product_widths(n_v):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library()
    wl = W.long_cadence(n_v=n_v, n_t=600, n_ss=2, cadence=0.01)
    plan = pt.GimenezPlan(8, 192)
    t = torch.as_tensor(wl["t"], dtype=torch.float64, device="cuda")
    orb = pt.orbit_to_device(wl["orbit"], "cuda")
    k = torch.as_tensor(wl["k"], dtype=torch.float32, device="cuda")
    ld = torch.as_tensor(wl["ld_gim"], dtype=torch.float32, device="cuda")
    f, _ = pt.gimenez(plan, t, orb, k, ld, n_ss=2, t_exp=wl["t_exp"])
    f = f.cpu().numpy()
    for v in sorted({0, 7 % n_v, n_v // 2, n_v - 1}):
        one = {x: None if orb[x] is None else orb[x][v:v + 1].contiguous() for x in orb}
        g, _ = pt.gimenez(plan, t, one, k[v:v + 1].contiguous(), ld[v:v + 1].contiguous(), n_ss=2, t_exp=wl["t_exp"])
        assert np.array_equal(g.cpu().numpy()[0], f[v]), v
    v = n_v - 1
    o = wl["orbit"]
    ov = dict(t0=o["t0"][v:v + 1], P=o["P"][v:v + 1], **{x: f32(np.asarray(o[x])[v:v + 1]) for x in ("a", "inc", "e", "w")})
    ref = oracle.lc_gimenez(wl["t"], ov, f32(wl["k"][v:v + 1]), f32(wl["ld_gim"][v:v + 1]), 192, n_ss=2, t_exp=wl["t_exp"])
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.max(np.abs(f[v].astype(np.float64) - np.asarray(ref).reshape(f[v].shape))) <= 1e-6
