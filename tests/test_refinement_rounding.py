"""The refinement's residual update (df_residual of fem_device.h, compiled here for the host): bit for bit the
double-float sum of a node's four edge fluxes that is renormalised after every edge and then subtracted, the
arithmetic of the one-node form, and at least 1.25 times as accurate as one that gathers the low parts."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_09763_gb300", "csrc")
SOURCE = r"""
#include "fem_device.h"
extern "C" void residuals(int n, float* rh, float* rl, const float* f) {
    for (int i = 0; i < n; ++i, f += 8)
        mls2mc::df_residual(rh[i], rl[i], f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7]);
}
"""
f32 = np.float32


def two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def df_add(ah, al, bh, bl):
    s, e = two_sum(ah, bh)
    e = e + (al + bl)
    h = s + e
    return h, e - (h - s)


def renormalised(rh, rl, f):
    ah, al = np.zeros_like(rh), np.zeros_like(rh)
    for t in range(4):
        ah, al = df_add(ah, al, f[:, 2 * t], f[:, 2 * t + 1])
    return df_add(rh, rl, -ah, -al)


def gathered(rh, rl, f):
    h, l = rh, rl
    for t in range(4):
        h, e = two_sum(h, -f[:, 2 * t])
        l = l + (e - f[:, 2 * t + 1])
    return h + l, l - ((h + l) - h)


def test_residual_update(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    (tmp_path / "r.cu").write_text(SOURCE)
    so = tmp_path / "r.so"
    subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, str(tmp_path / "r.cu"), "-o", str(so)], check=True)
    rng = np.random.default_rng(3)
    n = 200000
    exact = rng.normal(size=(n, 4))
    exact[:, 1] = -exact[:, 0] * (1 + 0.01 * rng.normal(size=n))   # east against west, north against south
    exact[:, 3] = -exact[:, 2] * (1 + 0.01 * rng.normal(size=n))
    f = np.empty((n, 8), dtype=f32)
    f[:, ::2] = exact
    f[:, 1::2] = exact - f[:, ::2]
    r = f.astype(np.float64).sum(axis=1) * (1 + 1e-4 * rng.normal(size=n))
    rh = r.astype(f32)
    rl = (r - rh).astype(f32)
    # every partial sum of these pairs spans under 60 bits: a long double (64 bits or more) holds it exactly enough
    want = rh.astype(np.longdouble) + rl - f.astype(np.longdouble).sum(axis=1)
    got_h, got_l = rh.copy(), rl.copy()
    lib = ctypes.CDLL(str(so))
    lib.residuals(n, *[ctypes.c_void_p(x.ctypes.data) for x in (got_h, got_l, f)])
    ref_h, ref_l = renormalised(rh, rl, f)
    assert np.array_equal(got_h, ref_h) and np.array_equal(got_l, ref_l)

    def rms(h, l):
        return float(np.sqrt(np.mean((h.astype(np.longdouble) + l - want) ** 2)))
    assert 1.25 * rms(got_h, got_l) < rms(*gathered(rh, rl, f))
