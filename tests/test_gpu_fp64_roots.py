"""The division-free reciprocal and reciprocal square roots of csrc/fp64.cuh and csrc/boys.cuh
against 1 / sqrt(a) and 1 / a: within 2 units in the last place, over the exponents that take them,
at the ends of a binade and at random mantissas; arguments outside rsqrt_fast's range go to the
library's own functions."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
dfscf = pytest.importorskip("paper_2506_06661_gb300")

SOURCE = """
#include <cstdint>
#include "common.cuh"
#include "boys.cuh"
#include "fp64.cuh"
__global__ void roots(const double* a, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = dfscf::rsqrt_ordinary(a[i]);
  out[n + i] = dfscf::rcp_ordinary(a[i]);
  out[2 * n + i] = rsqrt_fast(a[i]);
  out[3 * n + i] = dfscf::ordinary(a[i]) ? 1.0 : 0.0;
}
extern "C" int run(const double* a, int n, double* out) {
  roots<<<(n + 127) / 128, 128>>>(a, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    b = dfscf._build
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cu").write_text(SOURCE)
    subprocess.run([b.nvcc(), "-shared", "-o", str(d / "roots.so"), str(d / "roots.cu")] + b.NVCC_FLAGS, check=True)
    lib = ctypes.CDLL(str(d / "roots.so"))

    def call(a):
        dev = torch.as_tensor(a, dtype=torch.float64, device="cuda")
        out = torch.empty(4, len(a), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(ctypes.c_void_p(dev.data_ptr()), len(a), ctypes.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy()

    return call


def ulps(x, ref):
    return np.abs(x - ref) / np.spacing(np.abs(ref))


def test_ordinary_arguments(run):
    rng = np.random.default_rng(0)
    edges = np.concatenate([np.ldexp(m, np.arange(-821, 823)) for m in (1.0, 1.0 + 2.0 ** -52, 1.5, 2.0 - 2.0 ** -52)])
    a = np.concatenate([edges, np.ldexp(rng.uniform(1.0, 2.0, 200000), rng.integers(-821, 823, 200000))])
    rsqrt, rcp, fast, ok = run(a)
    assert np.all(ok == 1.0)
    assert np.max(ulps(rsqrt, 1.0 / np.sqrt(a))) <= 2.0
    assert np.max(ulps(fast, 1.0 / np.sqrt(a))) <= 2.0
    assert np.max(ulps(rcp, 1.0 / a)) <= 2.0


def test_range_of_rsqrt_fast(run):
    a = np.array([5e-324, 1e-310, 2.3e-308, 1e-300, 1e300, 8.9e307, 1.7e308, np.inf, 0.0])
    out = run(a)
    with np.errstate(divide="ignore"):
        ref = 1.0 / np.sqrt(a)
    assert np.max(ulps(out[2][:-2], ref[:-2])) <= 2.0 and np.array_equal(out[2][-2:], ref[-2:])
    assert not out[3][[0, 1, 2, 6, 7, 8]].any()
    assert np.isnan(run(np.array([np.nan, -1.0]))[2]).all()
