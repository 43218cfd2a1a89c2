"""Device functions and kernels whose rounding no entry point shows by itself, in a small library built for the test:
the FP64 root of an integer, and the FP32 mode kernel of the gradient on transforms that leave only its
window, phase and normalisation."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1512_07295_gb300 import build

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "adjoint.cu"
__global__ void k_probe_sqrt(double* out, int n) {
  for (int64_t i = pk::gtid(); i < n; i += pk::gstride()) out[i] = pk::sqrt_int(int(i) + 1);
}
extern "C" int probe_sqrt(double* out, int n) {
  k_probe_sqrt<<<256, 256>>>(out, n);
  return cudaDeviceSynchronize();
}
// counts: nbins entries; tab: 3 ng
extern "C" int probe_modes(void* g1, void* g2, int ng, int order, int nbins, double box, double* tab, const double* wsums,
                           const double* dl, const unsigned long long* counts) {
  using namespace pk;
  k_adjoint_tables<<<1, 128>>>(tab, ng, order);
  k_adjoint_modes<float><<<16, 256, (size_t(nbins) + 3 * size_t(ng / 2 + 1)) * 8>>>(
      static_cast<CC<float>*>(g1), static_cast<CC<float>*>(g2), ng, 1, 1, 2, nbins, box, tab, wsums, dl, counts);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    lib = os.path.dirname(build.lib_path())
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(d / "probe.so"), str(d / "probe.cu"),
                        "-L", lib, "-l:libpk.so", "-Xlinker", "-rpath," + lib, "-lcufft"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(d / "probe.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_sqrt_int_rounds_to_nearest_for_every_argument(probe):
    n = 2**20 - 1
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    assert probe.probe_sqrt(_p(out), n) == 0
    assert np.array_equal(out.cpu().numpy(), np.sqrt(np.arange(1, n + 1, dtype=np.float64)))


@pytest.mark.parametrize("ng,order", [(64, 4), (46, 3)])
def test_gradient_modes_round_window_and_phase_once(probe, ng, order):
    # G_1 = 0, G_2 = 1: X_1 = 2 kappa c^2 phi and X_2 = 2 kappa c^2 off the Nyquist slots. X_1's components are products of
    # phi, c twice and 2 kappa, each rounded once to FP32, by three rounded multiplications: 7 half-ulps, taken
    # as 8; also where the cosine or the sine is small (next to zero: what FP64 leaves of it)
    half, lz, box = ng // 2, ng // 2 + 1, 100.0
    g1 = torch.zeros((ng, ng, lz), dtype=torch.complex64, device="cuda")
    g2 = torch.ones_like(g1)
    rng = np.random.default_rng(ng)
    dl = rng.uniform(0.5, 2.0, half) / box**3
    counts = rng.integers(1, 1000, half)
    wsum = 12345.0
    dev = lambda a, t: torch.from_numpy(np.asarray(a, dtype=t)).cuda()
    tab = torch.empty(3 * ng, dtype=torch.float64, device="cuda")
    args = [dev([wsum, wsum, wsum], np.float64), dev(dl, np.float64), dev(counts, np.int64)]
    assert probe.probe_modes(_p(g1), _p(g2), ng, order, half, ctypes.c_double(box), _p(tab), *map(_p, args)) == 0
    n = np.fft.fftfreq(ng, 1.0 / ng)
    nz = np.arange(lz)
    nx, ny, nz = n[:, None, None], n[None, :, None], nz[None, None, :]
    n2 = nx**2 + ny**2 + nz**2
    b = np.floor(np.sqrt(n2) - 0.5).astype(int)  # edges b + 1/2; 4 |n|^2 is even, no edge is hit
    live = (n2 > 0) & (b < half) & (abs(nx) < half) & (abs(ny) < half) & (nz < half)
    win = np.sinc(nx / ng) * np.sinc(ny / ng) * np.sinc(nz / ng)
    kap = 2.0 * dl * box**3 / counts
    amp = kap[np.clip(b, 0, half - 1)] * (0.5 / (wsum * win**order)) ** 2
    ph = np.pi * (nx + ny + nz) / ng
    x1, x2 = g1.cpu().numpy().astype(np.complex128), g2.cpu().numpy().astype(np.complex128)
    for got, ref in ((x1.real, amp * np.cos(ph)), (x1.imag, amp * np.sin(ph))):
        assert np.all((np.abs(got - ref) <= 8 * 2.0**-24 * np.abs(ref) + 1e-14 * amp)[live])
    # X_2 = X_1 conj phi: two more roundings and phi's again, of terms of at most the size of the sum
    assert np.all((np.abs(x2 - amp) <= 16 * 2.0**-24 * amp)[live])
