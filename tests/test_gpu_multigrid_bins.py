"""Shell sums of the multi-grid estimate: rows that no warp divides, both bin tests, |n| sums by row symmetry."""

import numpy as np
import pytest
import torch

import oracle
from paper_1512_07295_gb300 import api, catalogs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# Bins with squared edges below and above 2^31 (the 32-bit and the 64-bit bin test), each with every mode in its first bin.
@pytest.mark.parametrize("ng", [8, 26, 40])
@pytest.mark.parametrize("ngrids", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_every_mode_once(ng, ngrids, prec):
    box = 100.0
    host = catalogs.poisson(4000, box, seed=ng)
    shifts = oracle.fourier.multigrid_shifts(ngrids)
    u = oracle.assign.grid_units(host, box, ng)
    delta = oracle.fourier.density_modes_multi([oracle.assign.assign_units(u, ng, 3, None, shift=d) for d in shifts], shifts, 3)
    power = box**3 * ((np.abs(delta) ** 2).sum() - abs(delta[0, 0, 0]) ** 2) / (ng**3 - 1)
    pos = torch.from_numpy(host).to(DEV)
    kw = dict(ng=ng, box=box, order=3, prec=prec, bin_lo2=1)
    a = [t.cpu().numpy() for t in api.power_multigrid(pos, api.Config(bin_w2=200, nbins=1, **kw), ngrids)]
    b = [t.cpu().numpy() for t in api.power_multigrid(pos, api.Config(bin_w2=20000, nbins=3, **kw), ngrids)]
    assert a[2][0] == b[2][0] == ng**3 - 1 and not b[2][1:].any()
    n = np.fft.fftfreq(ng, 1.0 / ng)
    mean = np.sqrt(n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2).sum() / (ng**3 - 1) * 2 * np.pi / box
    for r in (a, b):
        assert abs(r[1][0] / mean - 1) <= 1e-12
        # the tolerances of P(k) per bin; two FP32 calls differ among themselves by the order of the assignment's additions
        assert abs(r[0][0] / power - 1) <= (1e-5 if prec == "fp32" else 1e-10)
