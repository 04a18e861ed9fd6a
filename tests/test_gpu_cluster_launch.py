"""The first tickets of the cluster forms (1/128 on two CTAs, 1/256 on eight), which rank 0 hands to CTAs that
have just started: launches of one particle each, queued one behind another and captured in a graph, give the
bits of one launch over all particles (a particle's solve does not depend on the launch it is part of)."""
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


@pytest.mark.parametrize("N,n", [(128, 160), (256, 40)])
def test_single_particle_launches_equal_one_launch(N, n):
    K, obs = 15, wl.obs_grid(5)
    h = native.Handle([N], K, obs, np.zeros(len(obs)), 1.0, corr_len=0.2, precision=native.SMC_MIXED)
    theta = torch.from_numpy(wl.particles(n, K, N)).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def outputs():
        return (torch.zeros((n, len(obs)), dtype=torch.float64, device="cuda"),
                torch.zeros(n, dtype=torch.float64, device="cuda"),
                torch.zeros(n, dtype=torch.int32, device="cuda"))

    def one_by_one(out):
        for i in range(n):
            h.eval_likelihood_device(0, 1, theta[i].data_ptr(), *[x[i:].data_ptr() for x in out],
                                     stream=stream.cuda_stream)

    whole, queued, captured = outputs(), outputs(), outputs()
    torch.cuda.synchronize()
    h.eval_likelihood_device(0, n, theta.data_ptr(), *[x.data_ptr() for x in whole], stream=stream.cuda_stream)
    torch.cuda.synchronize()
    one_by_one(queued)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        one_by_one(captured)
    graph.replay()
    torch.cuda.synchronize()
    assert int(whole[2].min()) > 0
    for got in (queued, captured):
        assert all(torch.equal(a, b) for a, b in zip(whole, got))
