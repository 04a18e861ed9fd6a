"""The linear forward map from host arrays (read by the kernel from pinned memory when small) at the ends of its
range: equal, bit for bit, to device arrays, and to the FP64 product within the rounding of K terms in two orders
(2 K 2^-53 of the sum of magnitudes). Rows of one term, of less and more than a warp's 32 and of the most admitted."""
import numpy as np
import pytest
import torch

from paper_1709_09763_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


@pytest.mark.parametrize("K,n_obs", [(1, 1), (31, 33), (33, 49), (256, 1024)])
def test_linear_map_host_and_device(K, n_obs):
    rng = np.random.default_rng(K)
    A = rng.normal(size=(1, n_obs, K))
    h = native.Handle([4], K, np.full((n_obs, 2), 0.5), np.zeros(n_obs), 1.0, linear_A=A)
    for n in (1, 9, 300):
        theta = rng.normal(size=(n, K))
        G, Phi = h.eval_likelihood(0, theta)
        t = torch.from_numpy(theta).cuda()
        Gd = torch.empty((n, n_obs), dtype=torch.float64, device="cuda")
        Pd = torch.empty(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        h.eval_likelihood_device(0, n, t.data_ptr(), Gd.data_ptr(), Pd.data_ptr())
        torch.cuda.synchronize()
        assert np.array_equal(G, Gd.cpu().numpy()) and np.array_equal(Phi, Pd.cpu().numpy())
        assert np.all(np.abs(G - theta @ A[0].T) <= 2 * K * 2.0 ** -53 * (np.abs(theta) @ np.abs(A[0]).T))
