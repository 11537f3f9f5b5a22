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


@pytest.mark.parametrize("case", ["zeros and ones", "fractions", "subnormals", "infinity", "masked nan"])
def test_loss_of_masks_and_values(alp, case):
    """The loss's two summations: masks of zeros and ones over zero or normal
    values, and everything else.  Y and T are given, so the loss is one sum of
    130 * 70 terms m (y - t)^2 in double, rounded to float once: 2^-24 of it,
    and the terms' and additions' own 2^-53 errors are far below."""
    import torch
    C, B = 70, 130
    flat, X, T, Mk, d = setup(C, B, seed=91)
    rng = np.random.default_rng(92)
    Y = rng.standard_normal((B, C)).astype(np.float32)
    T = T.astype(np.float32)
    Mk = (rng.random((B, C)) < 0.7).astype(np.float32)
    Y[3, 5], T[3, 5], Mk[3, 5] = 0.0, -0.0, 1.0
    if case == "fractions":
        Mk[::3] *= np.float32(0.3)
    if case == "subnormals":
        Y[:], T[:] = 0.0, 0.0
        Y[7, 9], T[7, 8], Mk[7, 8:10] = 1e-42, -1e-42, 1.0
        Y[8, 9], Mk[8, 9] = 1e-15, 1.0
    if case == "infinity":
        Y[64, 69], Mk[64, 69] = np.inf, 1.0
    if case == "masked nan":
        Y[129, 0], Mk[129, 0] = np.nan, 0.0   # 0 * nan is in the sum
    new = lambda *s: torch.zeros(s, dtype=torch.float32, device="cuda")
    grads, work, loss = new(len(flat)), new(B * (C + 128)), new(2)
    alp.alp_mlp_backward(d(flat), C, d(X), B, new(B, 128), d(Y), d(T), d(Mk), grads, work, loss)
    y, t, m = (v.astype(np.float64) for v in (Y, T, Mk))
    want = np.sum(m * (y - t) ** 2) / m.sum()
    got = loss[0].item()
    assert loss[1].item() == np.float32(m.sum())
    if np.isfinite(want):
        assert abs(got - want) <= 2.0 ** -23 * want + 2.0 ** -149
    else:
        assert np.isnan(got) == np.isnan(want) and (np.isnan(got) or got == want)
