"""Device functions whose rounding no entry point shows by itself, in a small library built for the test: the FP64 root of an
integer."""

import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_1512_07295_gb300 import build

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "common.cuh"
__global__ void k_probe_sqrt(double* out, int n) {
  for (int64_t i = pk::gtid(); i < n; i += pk::gstride()) out[i] = pk::sqrt_int(int(i) + 1);
}
extern "C" int probe_sqrt(double* out, int n) {
  k_probe_sqrt<<<256, 256>>>(out, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "probe.so"), str(d / "probe.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(d / "probe.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_sqrt_int_rounds_to_nearest_for_every_argument(probe):
    n = 2**20 - 1
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    assert probe.probe_sqrt(_p(out), n) == 0
    assert np.array_equal(out.cpu().numpy(), np.sqrt(np.arange(1, n + 1, dtype=np.float64)))
