"""A handle whose first evaluation on a level is captured by its caller (relaxed mode, where buffers may be
allocated): nothing that an eager evaluation needs may have gone into the graph alone. Eager evaluations before
the first replay, after it and after the graph is dropped equal those of a handle that never captured."""
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


@pytest.mark.parametrize("N,n", [(32, 1300), (64, 310), (128, 80), (256, 20)])
def test_first_evaluation_captured(N, n):
    K, obs = 15, wl.obs_grid(5)
    theta = torch.from_numpy(wl.particles(n, K, N)).cuda()
    stream = torch.cuda.Stream()

    def handle():
        return native.Handle([N], K, obs, np.zeros(len(obs)), 1.0, corr_len=0.2, precision=native.SMC_MIXED)

    def evaluate(h, out):
        h.eval_likelihood_device(0, n, theta.data_ptr(), *[x.data_ptr() for x in out], stream=stream.cuda_stream)

    def outputs():
        out = (torch.zeros((n, len(obs)), dtype=torch.float64, device="cuda"),
               torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
        torch.cuda.synchronize()
        return out

    want = outputs()
    evaluate(handle(), want)
    torch.cuda.synchronize()
    assert int(want[2].min()) > 0
    dirty = [torch.full((1 << 20,), 0x01010101, dtype=torch.int32, device="cuda") for _ in range(16)]
    del dirty
    torch.cuda.empty_cache()
    h, got, eager = handle(), outputs(), outputs()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        evaluate(h, got)
    for _ in range(2):
        evaluate(h, eager)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, eager))
        for x in eager:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    del graph
    evaluate(h, eager)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, eager))
