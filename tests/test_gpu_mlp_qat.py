"""Quantisation-aware training's loss and gradient at the tiles' edges, against
a 64-bit restatement that rounds the same operands to BF16 (W2 and W3, and
the activations after layers 1 and 2) and passes gradients straight through
the rounding.

Tolerances, per parameter block: FP32 sums give 1e-4 of the block's largest
entry and 1e-3 of an entry, as without rounding.  An activation that FP32
places on the other side of a BF16 boundary moves by 2^-8 of itself; about one in
20,000 does (an error of 2e-7 over a spacing of 2^-8), so a tile of 16
samples holds at most one as a rule: 2^-8 / 16 = 2.5e-4 of one gradient entry, and
1e-4 / 16 of an output's weight in the loss, which is held to 1e-4.  The reference
without rounding misses the same bounds, so rounding left out would be seen.
"""
import ctypes

import numpy as np
import pytest

N_IN, N_H = 2, 128


def _bf16(x):
    """Round to nearest even at 8 significand bits."""
    m, e = np.frexp(x)
    return np.ldexp(np.rint(m * 256.0), e - 8)


def _silu(z):
    s = 1.0 / (1.0 + np.exp(-z))
    return z * s, s * (1.0 + z * (1.0 - s))


def loss_grad(p, X, T, rnd):
    """Loss, and the gradient's blocks by name, of L = mean_i sum_o (y_io - t_io)^2 (64 bits)."""
    q = _bf16 if rnd else (lambda x: x)
    shapes = (("W1", (N_H, N_IN)), ("b1", (N_H,)), ("W2", (N_H, N_H)), ("b2", (N_H,)), ("W3", (N_H, N_H)), ("b3", (N_H,)),
              ("W4", (2, N_H)), ("b4", (2,)))
    w, at = {}, 0
    for name, sh in shapes:
        w[name] = p[at:at + int(np.prod(sh))].reshape(sh)
        at += int(np.prod(sh))
    assert at == p.size
    W2, W3 = q(w["W2"]), q(w["W3"])
    h1, d1 = _silu(X @ w["W1"].T + w["b1"])
    h1 = q(h1)
    h2, d2 = _silu(h1 @ W2.T + w["b2"])
    h2 = q(h2)
    h3, d3 = _silu(h2 @ W3.T + w["b3"])
    e = h3 @ w["W4"].T + w["b4"] - T
    dy = 2.0 * e / X.shape[0]
    z3 = (dy @ w["W4"]) * d3
    z2 = (z3 @ W3) * d2
    z1 = (z2 @ W2) * d1
    g = dict(W1=z1.T @ X, b1=z1.sum(0), W2=z2.T @ h1, b2=z2.sum(0), W3=z3.T @ h2, b3=z3.sum(0), W4=dy.T @ h3, b4=dy.sum(0))
    return float((e * e).sum() / X.shape[0]), {name: g[name].reshape(-1) for name, _ in shapes}


def _case(n):
    import paper_1504_07433_gb300.surrogate as S
    rng = np.random.default_rng(n + 7)
    p = S.init_params(n, device="cpu").numpy().copy()
    p[S._OFF["b1"]:S._OFF["W2"]] = rng.normal(0, 0.1, 128)
    p[S._OFF["b4"]:] = rng.normal(0, 0.1, 2)
    return p, rng.uniform(-1, 1, (n, 2)).astype(np.float32), rng.normal(0, 1, (n, 2)).astype(np.float32)


def _misses(g, ref):
    out = []
    for name, r in ref.items():
        if np.any(np.abs(g[name] - r) > 1e-4 * np.max(np.abs(r)) + 1e-3 * np.abs(r)):
            out.append(name)
    return out


def test_reference_is_the_oracle_without_rounding_and_differs_with_it():
    import oracle
    p, X, T = (a.astype(np.float64) for a in _case(33))
    loss, g = loss_grad(p, X, T, False)
    loss_o, g_o = oracle.mlp_loss_grad(p, X, T)
    assert loss == pytest.approx(loss_o, rel=1e-12)
    assert np.allclose(np.concatenate(list(g.values())), g_o, rtol=1e-9, atol=1e-12 * np.max(np.abs(g_o)))
    _, gq = loss_grad(p, X, T, True)
    assert set(_misses(g, gq)) >= {"W1", "b1", "W2", "b2", "W3", "b3"}
    assert _bf16(np.array([1.0 + 2.0 ** -8, 1.0 + 3 * 2.0 ** -8, -0.3])).tolist() == [1.0, 1.0 + 2.0 ** -6, -0.30078125]


@pytest.mark.gpu
@pytest.mark.parametrize("n,shift", [(1, 0), (16, 3), (17, 1), (2433, 0), (4865, 2), (9729, 0), (17025, 1)])
def test_qat_loss_and_gradient(n, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1504_07433_gb300.surrogate as S
    from paper_1504_07433_gb300 import _ptr, _stream
    L = S.lib()
    p, X, T = _case(n)
    par = torch.zeros(S.N_PARAMS + 8, device="cuda")[shift:shift + S.N_PARAMS]
    par.copy_(torch.as_tensor(p))
    Xt, Tt = torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda")
    need = int(L.pt_mlp_work_bytes(n))
    work = torch.full((need,), 255, dtype=torch.uint8, device="cuda")
    grad, loss = torch.empty(S.N_PARAMS, device="cuda"), torch.empty(1, device="cuda")
    assert L.pt_mlp_loss_grad(ctypes.c_void_p(par.data_ptr()), _ptr(Xt), _ptr(Tt), n, 1, _ptr(grad), _ptr(loss), _ptr(work), need,
                              _stream()) == 0
    loss_r, ref = loss_grad(p.astype(np.float64), X.astype(np.float64), T.astype(np.float64), True)
    assert float(loss.item()) == pytest.approx(loss_r, rel=1e-4)
    g, at = {}, 0
    for name, r in ref.items():
        g[name] = grad.cpu().numpy()[at:at + r.size].astype(np.float64)
        at += r.size
    assert not _misses(g, ref)
