"""A CTA's shared memory may be written by the other CTAs of its cluster only once it has started: in every
kernel of the register-tiled solve a cluster barrier comes before the first ticket, which rank 0 stores into
the others' memory. The order is read from the source, since a kernel without the barrier is not to be run."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_09763_gb300", "csrc")


def _kernels(text):
    for m in re.finditer(r"__global__[^{;]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(0), text[m.end():i]


def test_cluster_barrier_before_the_first_store_into_a_peer():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "fem_tile.cu")).read())
    kernels = [body for _, body in _kernels(text) if "st_peer" in body]
    assert len(kernels) == 2   # one problem, many problems
    for body in kernels:
        first_ticket = re.search(r"\btake\(0\)", body).start()
        barrier = re.search(r"sync_all<G::C>\(\)", body)
        assert barrier and barrier.start() < first_ticket
