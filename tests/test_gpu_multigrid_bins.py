"""Shell sums of the multi-grid estimate: rows that no warp divides, both bin tests, |n| sums by row symmetry."""

import numpy as np
import pytest
import torch

from paper_1512_07295_gb300 import api, catalogs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# Bins with squared edges below and above 2^31 (the 32-bit and the 64-bit bin test), each with every mode in its first bin.
@pytest.mark.parametrize("ng", [8, 26, 40])
@pytest.mark.parametrize("ngrids", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_every_mode_once(ng, ngrids, prec):
    box = 100.0
    pos = torch.from_numpy(catalogs.poisson(4000, box, seed=ng)).to(DEV)
    kw = dict(ng=ng, box=box, order=3, prec=prec, bin_lo2=1)
    a = [t.cpu().numpy() for t in api.power_multigrid(pos, api.Config(bin_w2=200, nbins=1, **kw), ngrids)]
    b = [t.cpu().numpy() for t in api.power_multigrid(pos, api.Config(bin_w2=20000, nbins=3, **kw), ngrids)]
    assert a[2][0] == b[2][0] == ng**3 - 1 and not b[2][1:].any()
    n = np.fft.fftfreq(ng, 1.0 / ng)
    mean = np.sqrt(n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2).sum() / (ng**3 - 1) * 2 * np.pi / box
    for r in (a, b):
        assert abs(r[1][0] / mean - 1) <= 1e-12
    # the same values in another order of FP64 additions (FP32 runs of at most 32 lanes are the same runs)
    assert abs(a[0][0] / b[0][0] - 1) <= 1e-12
