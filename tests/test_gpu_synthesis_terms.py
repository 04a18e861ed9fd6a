"""The mixed path's KL synthesis at term counts around its split kernel's tiling: one term, odd counts
(a term per thread) and even ones (two), more terms than a block has threads, and groups of terms with
an odd remainder. G within 1e-6 of the FP64 oracle (the mixed path's bar)."""
import numpy as np
import pytest

from oracle import forward as ofwd
from paper_1709_09763_gb300 import native
from paper_1709_09763_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


@pytest.mark.parametrize("K", [1, 2, 15, 86, 128, 129, 255, 256, 299, 320])
def test_synthesis_term_counts(K):
    N, n, obs = 16, 131, wl.obs_grid(5)
    h = native.Handle([N], K, obs, np.zeros(len(obs)), 1.0, corr_len=0.1, precision=native.SMC_MIXED)
    theta = wl.particles(n, K, K)
    G, _ = h.eval_likelihood(0, theta)
    idx = [0, 64, n - 1]
    Gr = ofwd.Level(N, 0.1, 1.0, K, obs).G_batch(theta[idx])
    assert (np.abs(G[idx] - Gr).max(axis=1) / np.abs(Gr).max(axis=1)).max() < 1e-6
