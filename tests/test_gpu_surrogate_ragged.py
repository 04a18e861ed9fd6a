"""Gradients of the surrogate on batches of n rows that fill neither a warp's 32 rows of the GELU epilogue (tensor
memory is read by whole warps, rows past the batch included) nor the eight rows of a transposed store: on their
own, and after a larger batch whose leading dimension the work buffers keep. The reference is the same pass on 32 n
rows, whole warps, the other rows with their own predictions as targets (mean 0, deviation 1, so the error
signals there are exactly 0): each error signal is 1/32 of the ragged batch's, and BF16 rounding commutes with a
power of two, so the gradients differ by that factor and the order of FP32 sums of at most 1003 terms. Bound
1e-4 relative Frobenius: a chain of 1003 / 16 accumulations, each off by at most 2^-22 of the partial sum, is off
by 1.5e-5; a lost or doubled row of 1003 changes 3e-2."""
import numpy as np
import pytest

from test_gpu_surrogate import K, NOBS, _handle, _rel, _set_random, _target_fn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


@pytest.mark.parametrize("before", [0, 2048])
@pytest.mark.parametrize("n", [1, 5, 33, 1003])
def test_ragged_batches(n, before):
    h = _handle()
    flat, mu, sd = _set_random(h, 7)
    h.surrogate_set(0, flat, np.concatenate([np.zeros_like(mu), np.ones_like(sd)]))
    theta = np.random.default_rng(n).normal(0, 1, (32 * n, K))
    G, _ = h.surrogate_predict(0, theta)
    G[:n] = _target_fn(theta[:n])
    ref, ref_loss = h.surrogate_grads(0, theta, G)
    h = _handle()
    h.surrogate_set(0, flat, np.concatenate([np.zeros_like(mu), np.ones_like(sd)]))
    if before:
        x = np.random.default_rng(3).normal(0, 1, (before, K))
        h.surrogate_grads(0, x, _target_fn(x))
    g, loss = h.surrogate_grads(0, theta[:n], G[:n])
    assert loss == pytest.approx(32 * ref_loss, rel=1e-12)
    for a, r in zip(sum(h.unflatten(g), []), sum(h.unflatten(ref), [])):
        assert _rel(a, 32 * r) < 1e-4
