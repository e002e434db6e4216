"""Training kernels at the edges of the sample tiles (16, 32, 64 and 112 rows,
several tiles per SM) and of the weight gradients' chunks, with parameters and
work buffer that start at any float: outputs, loss and gradient against the
FP64 oracle network, with the tolerances of the other training test (FP32
sums: 1e-5 of the largest output, 1e-4 of the largest gradient)."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (15, 1), (16, 0), (17, 3), (2433, 0), (4865, 1), (9729, 2), (17025, 0)])
def test_tiles_vs_oracle(n, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300.surrogate as S
    from paper_1504_07433_gb300 import _ptr, _stream
    L = S.lib()
    rng = np.random.default_rng(n)
    p = S.init_params(n, device="cpu").numpy().copy()
    p[S._OFF["b1"]:S._OFF["W2"]] = rng.normal(0, 0.1, 128)
    p[S._OFF["b4"]:] = rng.normal(0, 0.1, 2)
    X = rng.uniform(-1, 1, (n, 2)).astype(np.float32)
    T = rng.normal(0, 1, (n, 2)).astype(np.float32)
    buf = torch.zeros(S.N_PARAMS + 8, device="cuda")
    pt_ = buf[shift:shift + S.N_PARAMS]
    pt_.copy_(torch.as_tensor(p))
    Xt, Tt = torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda")
    need = int(L.pt_mlp_work_bytes(n))
    raw = torch.full((need + 64,), 255, dtype=torch.uint8, device="cuda")
    work = raw[4 * shift:4 * shift + need]
    g = torch.empty(S.N_PARAMS + 8, device="cuda")[shift:shift + S.N_PARAMS]
    loss = torch.empty(1, device="cuda")
    Y = torch.empty((n, 2), device="cuda")
    ptr = lambda x: ctypes.c_void_p(x.data_ptr())  # noqa: E731
    assert L.pt_mlp_forward(ptr(pt_), _ptr(Xt), n, 0, _ptr(Y), ptr(work), need, _stream()) == 0
    assert L.pt_mlp_loss_grad(ptr(pt_), _ptr(Xt), _ptr(Tt), n, 0, ptr(g), _ptr(loss), ptr(work), need, _stream()) == 0
    pd = p.astype(np.float64)
    Yr = oracle.mlp_forward(pd, X.astype(np.float64))
    assert np.max(np.abs(Y.cpu().numpy() - Yr)) <= 1e-5 * max(1.0, np.max(np.abs(Yr)))
    loss_r, g_r = oracle.mlp_loss_grad(pd, X.astype(np.float64), T.astype(np.float64))
    assert float(loss.item()) == pytest.approx(loss_r, rel=1e-5)
    err = np.abs(g.cpu().numpy().astype(np.float64) - g_r)
    assert np.all(err <= 1e-4 * np.max(np.abs(g_r)) + 1e-3 * np.abs(g_r)), np.argmax(err)
