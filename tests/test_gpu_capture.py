"""A device-array evaluation captured by its caller (where the kernels are launched without the programmatic
overlap) and one queued behind other work on the same stream (with it): equal, bit for bit, to an
evaluation on its own, also when the captured graph is replayed on new particles."""
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


@pytest.mark.parametrize("N,precision,n", [(8, native.SMC_MIXED, 100), (32, native.SMC_MIXED, 1300),
                                           (64, native.SMC_MIXED, 310), (128, native.SMC_MIXED, 80),
                                           (16, native.SMC_FP64, 100)])
def test_captured_and_queued_evaluations(N, precision, n):
    K, obs = 15, wl.obs_grid(5)
    h = native.Handle([N], K, obs, np.zeros(len(obs)), 1.0, corr_len=0.2, precision=precision)
    sets = [torch.from_numpy(wl.particles(n, K, N + s)).cuda() for s in range(3)]
    theta = sets[0].clone()
    G = torch.empty((n, len(obs)), dtype=torch.float64, device="cuda")
    Phi = torch.empty(n, dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    args = (0, n, theta.data_ptr(), G.data_ptr(), Phi.data_ptr())
    alone = []
    for x in sets:   # one at a time
        theta.copy_(x)
        torch.cuda.synchronize()
        h.eval_likelihood_device(*args, stream=stream.cuda_stream)
        torch.cuda.synchronize()
        alone.append((G.clone(), Phi.clone()))
    with torch.cuda.stream(stream):   # queued one behind another
        got = []
        for x in sets:
            theta.copy_(x)
            h.eval_likelihood_device(*args, stream=stream.cuda_stream)
            got.append((G.clone(), Phi.clone()))
    torch.cuda.synchronize()
    assert all(torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) for a, b in zip(alone, got))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        h.eval_likelihood_device(*args, stream=stream.cuda_stream)
    for x, a in zip(sets, alone):
        theta.copy_(x)
        G.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(G, a[0]) and torch.equal(Phi, a[1])
