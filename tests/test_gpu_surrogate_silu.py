"""The last hidden layer's SiLU is FP32.  With W3 = 0 its inputs are exactly the
biases b3, and one-hot W4 rows give two of its units per model, each unchanged: the
128 values over [-20, 8] against 64 bits.  Bound, relative: e/(1 + e) <= 1 times expf's
2^-23, the sum's 2^-24, the quotient's 2^-24 (1.1 with its correction), 2.5e-7 (the
exponential by ex2.approx of a rounded product was off by up to 1e-6)."""
import numpy as np
import pytest


@pytest.mark.gpu
def test_last_layer_silu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300.surrogate as S
    x = np.linspace(-20.0, 8.0, 128).astype(np.float32)
    p = S.init_params(1, device="cpu").numpy().copy()
    p[S._OFF["W3"]:S._OFF["b3"]] = 0.0
    p[S._OFF["b3"]:S._OFF["b3"] + 128] = x
    p[S._OFF["b4"]:S._OFF["b4"] + 2] = 0.0
    X = torch.rand((300, 2), device="cuda") * 2 - 1
    got = np.empty(128)
    for j in range(64):
        w4 = np.zeros((2, 128), np.float32)
        w4[0, j], w4[1, 127 - j] = 1.0, 1.0
        p[S._OFF["W4"]:S._OFF["b4"]] = w4.ravel()
        model = S.SurrogateModel(torch.as_tensor(p, device="cuda"))
        Y = model.network(X).cpu().numpy().astype(np.float64)
        assert (Y == Y[0]).all()
        got[j], got[127 - j] = Y[0]
        model.close()
    x64 = x.astype(np.float64)
    ref = x64 / (1.0 + np.exp(-x64))
    err = np.abs(got / ref - 1.0).max()
    assert err <= 2.5e-7, err
