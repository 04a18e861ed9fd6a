"""The autotuner times each kernel of a level once: on 1/32 and 1/64 of the mixed path, where every block size
names the same one, it keeps the default after four evaluations (one for warm-up, three timed; three kernels each)."""
import numpy as np
import pytest

from paper_1709_09763_gb300 import native
from paper_1709_09763_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1709_09763_gb300 import build
    build.build()


@pytest.mark.parametrize("levels,prec,forms", [([32, 64], native.SMC_MIXED, 2), ([8, 16], native.SMC_MIXED, 4),
                                               ([16, 32], native.SMC_FP64, 4)])
def test_each_kernel_is_timed_once(levels, prec, forms):
    h = native.Handle(levels, 16, wl.obs_grid(5), np.zeros(25), 1.0, corr_len=0.2, precision=prec)
    lib = native.load()
    default = [h.block_size(l) for l in range(2)]
    before = lib.smc_kernel_launches()
    chosen, ms = h.autotune(200)
    launches = lib.smc_kernel_launches() - before
    for l in range(2):
        h.set_block_size(l, 0)
    assert launches == 1 + 4 * forms * (3 if prec == native.SMC_MIXED else 1)   # the draws; split, contraction, solve
    assert all(m > 0 for m in ms)
    if forms == 2:
        assert chosen == default
