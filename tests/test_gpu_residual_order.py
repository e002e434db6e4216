"""Residual sums are formed in an order that the number of times alone fixes: a
vector has, bit for bit, the sums of a small call with it, whatever shape the
large call's tiles have (rows of 3.4 and 4 KB: tiles of several blocks of
times).  Infinite sums stay infinite and NaN observations give NaN."""
import numpy as np
import pytest

from paper_1504_07433_gb300 import workloads as W
from tests.helpers import gpu_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,n_b", [("ma", 1), ("ma", 3), ("gim", 1), ("gim", 2), ("interp", 1), ("zi", 1)])
def test_sum_of_a_vector_does_not_depend_on_the_call(model, n_b):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300 as pt
    pt.load_library(build_if_missing=True)
    n_v, n_t = 1000, 3000
    rng = np.random.default_rng(n_b)
    wl = W.long_cadence(n_v=n_v, n_t=n_t, n_ss=1, cadence=0.01)
    u = np.stack(W.q_to_u(rng.uniform(0, 1, (n_v, n_b)), rng.uniform(0, 1, (n_v, n_b))), -1)
    plan = pt.GimenezPlan(8, 192) if model in ("gim", "zi") else None
    table = pt.MATable(0.03125, 0.25, 32, 1024) if model == "interp" else None
    wl["ld"] = u if plan is None else W.quad_to_general(u[..., 0], u[..., 1], 8)
    t, orb, k, ld = gpu_inputs(wl)
    y_np = rng.normal(1.0, 1e-3, (n_b, n_t)).astype(np.float32)

    def call(orb, k, ld, y, **kw):
        args = (t, orb, k, ld)
        fn = {"ma": pt.ma_quad, "gim": lambda *a, **q: pt.gimenez(plan, *a, **q),
              "zi": lambda *a, **q: pt.gimenez_zi(plan, *a, **q),
              "interp": lambda *a, **q: pt.ma_quad_interp(table, *a, **q)}[model]
        return fn(*args, y=torch.as_tensor(y, device="cuda"), want_ssr=True, **kw)

    flux, ssr = call(orb, k, ld, y_np)
    for lo in (0, 500, n_v - 6):
        part = {x: None if v is None else v[lo:lo + 6].contiguous() for x, v in orb.items()}
        f1, s1 = call(part, k[lo:lo + 6].contiguous(), ld[lo:lo + 6].contiguous(), y_np)
        assert torch.equal(f1, flux[lo:lo + 6]) and torch.equal(s1, ssr[lo:lo + 6])
    y_inf, y_nan = y_np.copy(), y_np.copy()
    y_inf[0, 100], y_nan[0, 2000] = 1e25, np.nan
    assert torch.isinf(call(orb, k, ld, y_inf, want_flux=False)[1][:, 0]).all()
    assert torch.isnan(call(orb, k, ld, y_nan, want_flux=False)[1][:, 0]).all()
