"""The cost model's forward and backward kernels at the edges of their blocks
(16 samples, 64 outputs, gradient tiles of 8 rows, the batch shared by eight
blocks), against the float64 oracle with the tolerances of test_mlp_gpu."""
import numpy as np
import pytest

from oracle import mlp

from .test_mlp_gpu import setup, to_list

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B", [(1, 1), (1, 17), (8, 16), (78, 7), (64, 33), (65, 513), (130, 100)])
def test_forward_and_backward_edges(alp, C, B):
    import torch
    flat, X, T, Mk, d = setup(C, B, seed=50 + C + B)
    Mk[0, 0] = 1.0   # at least one element counts
    dP = d(flat)
    new = lambda *s: torch.full(s, float("nan"), dtype=torch.float32, device="cuda")
    Y, cache, grads = new(B, C), new(B, 128), new(len(flat))
    work, loss = new(B * (C + 128)), new(2)
    alp.alp_mlp_forward(dP, C, d(X), B, Y, cache)
    alp.alp_mlp_backward(dP, C, d(X), B, cache, Y, d(T), d(Mk), grads, work, loss)
    P = to_list(flat, C)
    y, cch = mlp.forward(P, X.astype(np.float64))
    assert np.allclose(Y.cpu().numpy(), y, rtol=1e-5, atol=1e-5)
    c = cache.cpu().numpy()
    assert np.allclose(c[:, :64], cch[1], rtol=1e-5, atol=1e-5)
    assert np.allclose(c[:, 64:], cch[3], rtol=1e-5, atol=1e-5)
    g_ref = mlp.backward(P, cch, y, T.astype(np.float64), Mk.astype(np.float64))
    for a, b in zip(to_list(grads.cpu().numpy(), C), g_ref):
        tol = 1e-4 * np.abs(b) + 1e-5 * np.abs(b).max() + 1e-12
        assert np.all(np.abs(a - b) <= tol)
    assert abs(loss[0].item() - mlp.loss(y, T, Mk)) <= 1e-5 * mlp.loss(y, T, Mk)
    assert loss[1].item() == Mk.sum()
