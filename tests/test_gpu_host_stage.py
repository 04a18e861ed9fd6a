"""Evaluations with host arrays on both sides of the size up to which they run from pinned memory
(256 KiB of particles, observations, potentials and iteration counts): equal, bit for bit, to the
evaluation with device arrays."""
import numpy as np
import pytest
import torch

from paper_1709_09763_gb300 import native
from paper_1709_09763_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


@pytest.mark.parametrize("want_G", [True, False])
@pytest.mark.parametrize("N,precision", [(8, native.SMC_MIXED), (32, native.SMC_MIXED), (8, native.SMC_FP64)])
def test_host_arrays_equal_device_arrays(N, precision, want_G):
    K, obs = 16, wl.obs_grid(5)
    h = native.Handle([N], K, obs, np.zeros(len(obs)), 1.0, corr_len=0.2, precision=precision)
    fit = 256 * 1024 // (8 * (K + 1 + (len(obs) if want_G else 0)) + 4)
    for n in (1, fit, fit + 1, 3):
        theta = wl.particles(n, K, 31 * N + n)
        G, Phi = h.eval_likelihood(0, theta, want_G=want_G)
        t = torch.from_numpy(theta).cuda()
        Gd = torch.empty((n, len(obs)), dtype=torch.float64, device="cuda")
        Pd = torch.empty(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        h.eval_likelihood_device(0, n, t.data_ptr(), Gd.data_ptr(), Pd.data_ptr())
        torch.cuda.synchronize()
        assert np.array_equal(Phi, Pd.cpu().numpy())
        assert G is None if not want_G else np.array_equal(G, Gd.cpu().numpy())
