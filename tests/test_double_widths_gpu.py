"""Sums of doubles at every vector width the autotuner may build the streaming
kernels with: a chunk of equal exponents and significands near 2 fills the
integer sum as far as it goes."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1412_1127_gb300 import autotune, build

pytestmark = pytest.mark.gpu

WIDTHS = sorted({v for _, _, cands in autotune.WIDTHS.values() for c in cands for v in (c[:2] if len(c) == 3 else c)} | {1})

SOURCE = r"""
#include "fold.cuh"
using namespace accr;
// one thread a block folds NV vectors of two doubles
template <int NV>
__global__ void chunks(const double *x, double *out) {
    uint4 v[NV];
    for (int i = 0; i < NV; ++i) v[i] = reinterpret_cast<const uint4 *>(x + 2 * NV * blockIdx.x)[i];
    Acc A;
    A.a = d2u(-0.0);
    A.c = 0.f;
    fold_vec<double, NV>(W_ADDF, A, v);
    out[blockIdx.x] = u2d(A.a);
}
extern "C" __attribute__((visibility("default"))) int run(int nv, const double *x, double *out, int n) {
    switch (nv) {
%s
    default: return -1;
    }
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("widths")
    cases = "\n".join("    case %d: chunks<%d><<<n, 1>>>(x, out); break;" % (w, w) for w in WIDTHS)
    src, lib = os.path.join(d, "probe.cu"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(SOURCE % cases)
    r = subprocess.run([build.nvcc()] + build.NVCC_FLAGS + ["-shared", src, "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(lib)
    L.run.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    return L


@pytest.mark.parametrize("width", WIDTHS)
@pytest.mark.parametrize("kind", ["ones", "near_two", "minus_near_two", "mixed"])
def test_full_chunks(probe, width, kind):
    n = 64
    g = np.random.default_rng(width)
    x = {"ones": np.ones((n, 2 * width)), "near_two": np.full((n, 2 * width), 2 - 2.0 ** -52),
         "minus_near_two": np.full((n, 2 * width), -(2 - 2.0 ** -52)),
         "mixed": 1 + g.random((n, 2 * width))}[kind]
    xt = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert probe.run(width, xt.data_ptr(), out.data_ptr(), n) == 0
    want = x.sum(1)
    # per value 2^-6 ulp of the largest is cut off, and every sum rounds once
    bound = 2 * width * 2.0 ** -53 * np.abs(x).sum(1)
    assert np.all(np.abs(out.cpu().numpy() - want) <= bound)
