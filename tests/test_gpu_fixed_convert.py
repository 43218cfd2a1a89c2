"""PK_FIXED64's conversion of both integer grids to doubles in one launch."""

import math

import numpy as np
import pytest
import torch

from paper_1512_07295_gb300 import api, catalogs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# Node counts below, at and past what the grid's blocks take in a round, odd parts of the four loads in flight.
@pytest.mark.parametrize("ng", [8, 18, 64, 98])
@pytest.mark.parametrize("interlace", [False, True])
@pytest.mark.parametrize("signed", [False, True])
def test_grids_are_multiples_of_the_scale(ng, interlace, signed):
    box, n = 100.0, 20000
    pos = torch.from_numpy(catalogs.poisson(n, box, seed=ng)).to(DEV)
    w = np.random.default_rng(ng).uniform(-1.0 if signed else 0.25, 1.0, n).astype(np.float32)
    tw = torch.from_numpy(w).to(DEV)
    kw = dict(ng=ng, box=box, order=3, interlace=interlace)
    got = api.assign(pos, api.Config(prec="fixed64", **kw), tw)
    ref = api.assign(pos, api.Config(prec="fp64", **kw), tw)
    scale = 2.0 ** (62 - math.ceil(math.log2(np.abs(w.astype(np.float64)).sum())))
    assert (got[1] is None) == (not interlace)
    for g, r in zip(got, ref):
        if g is None:
            continue
        q = (g * scale).cpu().numpy()  # exact: a power of two
        assert np.array_equal(q, np.rint(q))  # an integer, rounded to 53 bits
        # the mode's grids: 32-bit products of weights near 1, at most a few hundred per node
        assert float((g - r).abs().max()) <= 1e-5 * float(r.abs().max())
