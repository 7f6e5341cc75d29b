"""Fixed-point forms of the FP64 kernels at the ends of their range: values that
are not finite, fields near the identity, nearly dependent rows, long lines."""

import ctypes
import subprocess

import numpy as np
import pytest

from paper_1206_0675_gb300 import build, fields, lgf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    lgf.load_library()


# Device functions that no entry point reaches by themselves, as a small library of their own.
PROBE = r"""
#include "lgf_gauge.cuh"
using namespace lgf;
// G of one site after g with the given FP64 rows (stored as a lane stores them)
__global__ void accumulate(const double2* rows, double2* gf, double2* G) {
  fxg_store(gf, 1, 0, rows, rows + 3, rows + 6);
  accumulate_gauge_fx(1, 0, reinterpret_cast<const int4*>(gf), 1, G);
}
extern "C" int probe_accumulate(const double* rows, double* G) {
  double2* d;
  cudaMalloc(&d, 27 * sizeof(double2));
  cudaMemcpy(d, rows, 9 * sizeof(double2), cudaMemcpyHostToDevice);
  cudaMemcpy(d + 18, G, 9 * sizeof(double2), cudaMemcpyHostToDevice);
  accumulate<<<1, 1>>>(d, d + 9, d + 18);
  const cudaError_t e = cudaMemcpy(G, d + 18, 9 * sizeof(double2), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    subprocess.run([build.nvcc(), "-shared", *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-o",
                    str(d / "libprobe.so"), str(d / "probe.cu")], check=True)
    return ctypes.CDLL(str(d / "libprobe.so"))


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


# ---------------------------------------------------------------------------
# a g that is not finite
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_transform_of_a_nonfinite_g(probe, bad):
    """G <- g G with an entry of g that is not finite is not finite, also where every sum that the entry's mark would
    enter as a number (-2) stays in range."""
    g = np.eye(3, dtype=np.complex128)
    g[1, 2] = bad
    G = np.full((3, 3), 0.3 + 0.2j)
    assert probe.probe_accumulate(ptr(g), ptr(G)) == 0
    assert not np.isfinite(G).any()


def test_transform_of_a_finite_g(probe):
    g = fields.random_links((2, 2, 2, 2), 0.9, seed=3).reshape(-1, 3, 3)[0]
    G = fields.random_links((2, 2, 2, 2), 0.9, seed=4).reshape(-1, 3, 3)[1].copy()
    want = g @ G
    assert probe.probe_accumulate(ptr(np.ascontiguousarray(g)), ptr(G)) == 0
    assert np.max(np.abs(G - want)) < 2e-15
