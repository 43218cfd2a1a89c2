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
    # The mode's products: FP32 (three weights and w, within 4 ulp of at most 1), rounded at a scale 2^e that keeps a tile's
    # 32-bit sums from overflowing: 2^e count node_share max|w| < 2^30 and 2^e node_share max|w| < 2^19, node_share = (3/4)^3.
    u = pos.cpu().numpy() * (ng / box)
    t = np.minimum(u.astype(int), ng - 1) // 8
    share, wmax = 0.75**3, float(np.abs(w).max())
    count = np.bincount((t[:, 0] * 64 + t[:, 1]) * 64 + t[:, 2]).max()
    e = min(30 - math.frexp(max(count * wmax * share, 1.0))[1], 19 - math.frexp(wmax * share)[1])
    for k, (g, r) in enumerate(zip(got, ref)):
        if g is None:
            continue
        q = (g * scale).cpu().numpy()  # exact: a power of two
        assert np.array_equal(q, np.rint(q))  # an integer, rounded to 53 bits
        near = np.zeros((ng,) * 3)  # products per node: particles whose nearest node is at most one away on each axis
        np.add.at(near, tuple((np.rint(u + 0.5 * k).astype(int) % ng).T), 1)
        for axis in range(3):
            near = near + np.roll(near, 1, axis) + np.roll(near, -1, axis)
        bound = near * (2.0 ** -(e + 1) + 4 * 2.0**-24) + 1e-14 * float(r.abs().max())
        assert np.all(np.abs((g - r).cpu().numpy()) <= bound)
