"""Standardised targets of the gradient entry point are (G - mu) / sd, rounded to FP64 and then to FP32, as the
training batches' are. With a network of zeros the loss is their mean square, so it shows them to the last bit: the
quotients here are midpoints between two FP32 values, and a product with the rounded reciprocal of sd falls on the
other side of some. FP64 sums of 2 x 49 squares: relative bound 1e-13; one FP32 spacing in one target is above 1e-10."""
import numpy as np
import pytest

from paper_1709_09763_gb300 import native
from test_gpu_surrogate import K, NOBS, _handle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


def test_targets_are_divided():
    h = _handle()
    d = h.surrogate_dims()
    rng = np.random.default_rng(12)
    sd = rng.uniform(0.5, 2.0, NOBS).astype(np.float32)
    q = (2 * rng.integers(2 ** 23, 2 ** 24, (2, NOBS)) + 1) / 2.0 ** 24   # 25 bits, odd: halfway between FP32 values
    G = q * sd.astype(np.float64)                                        # 49 bits: exact
    want = (G / sd).astype(np.float32)
    assert np.sum(want != (G * (1.0 / sd.astype(np.float64))).astype(np.float32)) > 5
    params = np.zeros(sum(d[l + 1] * d[l] + d[l + 1] for l in range(5)), dtype=np.float32)
    mu_sd = np.concatenate([np.zeros(d[5]), sd, np.ones(d[5] - NOBS)]).astype(np.float32)
    h.surrogate_set(0, params, mu_sd)
    _, loss = h.surrogate_grads(0, np.zeros((2, K)), G)
    assert loss == pytest.approx(float(np.mean(want.astype(np.float64) ** 2)), rel=1e-13)
