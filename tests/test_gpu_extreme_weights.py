"""Softmax with classes masked by weights of fp32's lowest value, of bf16's
edge, or of minus infinity: on positive features their logits are so negative
that the classes have no probability, and the other classes' gradients and the
loss are those of a model without them.

The reference is fp64 numpy over the unmasked classes; tolerances as for the
split kernels (1e-5; 2e-6 for the loss, 2e-2 where the kernels multiply bf16)."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import make_gpu, rel_err

pytestmark = pytest.mark.gpu

BASE = W.WORKLOADS["cr_n128_softmax_k1000"].replace(n=3, s=1, lr=0.1)
LOWEST = float(np.finfo(np.float32).min)
BF16_MAX = 3.3895313892515355e38


def _problem(K, d, m, dtype, masked, value):
    rng = np.random.default_rng([K, d])
    w = BASE.replace(K=K, d=d, m=m, dtype=dtype)
    beta = (rng.standard_normal((K, d)) / np.sqrt(d)).astype(np.float32)
    beta[masked] = value
    keep = np.setdiff1d(np.arange(K), masked)
    Xs, ys = [], []
    for _ in range(w.n):
        X = rng.uniform(0.25, 1.0, (m, d)).astype(np.float32)
        Xs.append(X if dtype == "f32" else W.f32_to_bf16_bits(X))
        ys.append(keep[rng.integers(0, len(keep), m)].astype(np.int32))
    return w, beta, keep, Xs, ys


def _reference(w, beta, keep, Xs, ys):
    grads, loss = [], 0.0
    for X, y in zip(Xs, ys):
        x = W.features_as_float(X, w.dtype).astype(np.float64)
        z = x @ beta[keep].astype(np.float64).T
        z -= z.max(1, keepdims=True)
        at = np.searchsorted(keep, y)
        loss += (np.log(np.exp(z).sum(1)) - z[np.arange(len(y)), at]).sum()
        p = np.exp(z) / np.exp(z).sum(1, keepdims=True)
        p[np.arange(len(y)), at] -= 1.0
        g = np.zeros((w.K, w.d))
        g[keep] = p.T @ x / len(y)
        grads.append(g)
    return grads, loss / sum(len(y) for y in ys)


@pytest.mark.parametrize("value", [LOWEST, -np.inf, -BF16_MAX, -1e38], ids=["lowest", "-inf", "bf16max", "1e38"])
@pytest.mark.parametrize("dtype,K,d,m,tol", [("f32", 10, 100, 90, 1e-5), ("f32", 70, 130, 90, 1e-5), ("bf16", 20, 64, 140, 1e-5),
                                             ("bf16", 300, 96, 130, 2e-2)])
def test_masked_classes(libpgc, cuda, dtype, K, d, m, tol, value):
    """Set at creation time by set_weights, and carried through the update of a
    step (the decode writes the parts anew)."""
    masked = np.arange(128, 256) if K > 256 else np.array([1, K - 1])   # K = 300: a whole block of the loss kernel
    w, beta, keep, Xs, ys = _problem(K, d, m, dtype, masked, value)
    grads, loss = _reference(w, beta, keep, Xs, ys)
    g = make_gpu(libpgc, w, Xs, ys)
    g.set_weights(beta)
    assert g.loss() == pytest.approx(loss, rel=2e-6)
    out = np.zeros(K * d, np.float32)
    mask = np.array([0, 1, 0], np.uint8)
    g.step(mask, out)                                        # warm-up: every store holds its gradient at beta
    for k in range(w.n):
        got = g.store(k, 0)
        assert rel_err(got, grads[k]) < tol
        assert (got[masked] == 0).all()
    after = g.weights()
    assert (after[masked] == np.float32(value)).all() and np.isfinite(after[keep]).all()
    grads, loss = _reference(w, after, keep, Xs, ys)
    assert g.loss() == pytest.approx(loss, rel=2e-6)
    g.step(mask, out)                                        # slot 0: worker k's own partition, at the new beta
    for k in range(w.n):
        assert rel_err(g.store(k, 0), grads[k]) < tol
    g.close()


@pytest.mark.parametrize("dtype,K", [("f32", 10), ("bf16", 20), ("bf16", 300)])
def test_nan_weights_stay_visible(libpgc, cuda, dtype, K):
    """A NaN parameter is not clamped away."""
    w, beta, _, Xs, ys = _problem(K, 64, 40, dtype, np.array([1]), np.nan)
    g = make_gpu(libpgc, w, Xs, ys)
    g.set_weights(beta)
    assert np.isnan(g.loss())
    g.step(np.array([0, 1, 0], np.uint8))
    g.sync()
    assert np.isnan(g.weights()).any()
    g.close()
