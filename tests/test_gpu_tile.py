"""The register-tiled solve on 1/32 .. 1/256 (mixed path) where its tiling can go wrong: a single
particle, fewer and more particles than resident blocks or clusters (whose shared memory then holds an
earlier particle's values), observations on the boundary, in corners, in every position of a 4 x 4 patch and
across the borders between the CTAs of a cluster, and the load-vector table. G within 1e-6 of the FP64 oracle (the mixed path's bar: FP32 field with BF16-split
synthesis, whose error dominates), and bit-identical when evaluated again after another launch."""
import numpy as np
import pytest

from oracle import fem as ofem
from oracle import forward as ofwd
from paper_1709_09763_gb300 import native
from paper_1709_09763_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


def _obs(N):
    edge = [(0, 0), (1, 0), (0, 1), (1, 1), (0.5, 0), (0, 0.5), (1, 0.5), (0.5, 1)]
    patch = [((N // 2 + i + 0.3) / N, (N // 2 - j - 0.2) / N) for i in range(4) for j in range(4)]
    last = [((N - 0.5) / N, (N - 0.7) / N), (0.4 / N, 0.6 / N), ((N - 1) / N, 1 / N)]
    rows = [((N - 0.6) / N, (N // 8 * k + d) / N) for k in range(1, 8) for d in (-0.5, 0.5)]
    return np.array(edge + patch + last + rows)


@pytest.mark.parametrize("source", ["one", "nine"])
@pytest.mark.parametrize("N,n", [(32, 1), (32, 3000), (64, 1), (64, 700), (128, 1), (128, 200), (256, 1), (256, 45)])
def test_tile_form_against_oracle(N, n, source):
    K, obs = 12, _obs(N)
    y = np.zeros(len(obs))
    h = native.Handle([N], K, obs, y, 1.0, corr_len=0.2, precision=native.SMC_MIXED, source=source)
    theta = wl.particles(n, K, 17 * N + n)
    G, Phi = h.eval_likelihood(0, theta)
    idx = sorted({0, n // 2, n - 1})
    Gr = ofwd.Level(N, 0.2, 1.0, K, obs, f=ofem.nine_sources if source == "nine" else None).G_batch(theta[idx])
    assert (np.abs(G[idx] - Gr).max(axis=1) / np.abs(Gr).max(axis=1)).max() < 1e-6
    h.eval_likelihood(0, wl.particles(n, K, 5))
    G2, Phi2 = h.eval_likelihood(0, theta)
    assert np.array_equal(G, G2) and np.array_equal(Phi, Phi2)
